// isosurface.cu -- iso-surfaces of a cell field (the paper's Fig. 3 shows
// iso-surfaces of the Q criterion) and their orthographic depth image, in
// CUDA, with no graphics API.
//
// Extraction: marching tetrahedra.  The cube whose corners are cells
// (i + dx, j + dy, k + dz) (values with periodic wrap, coordinates unwrapped,
// corner b = dx + 2 dy + 4 dz at ((i + dx + 1/2) h, ...)) is split into the six
// tetrahedra of the Freudenthal triangulation (paths 0 -> e_a -> e_a + e_b -> 7),
// the same split in every cube, so the surface is closed.  A corner is inside
// when f > iso; a tetrahedron with one corner apart gives one triangle, two
// and two give two (the fixed vertex orders below).  Edge points are the
// linear zero of f - iso from the edge's lower corner.  Triangles are written
// cube by cube in flat cube order: a count pass, a scan of the block totals, and
// an emit pass that scans its block in shared memory.
//
// Rasterisation in single precision: view along +z, W x W pixel centres
// ((p + 1/2) L / W, in double), coordinates relative to each triangle's first
// corner rounded to FP32, edge functions and barycentric depth in FP32, a
// pixel covered when its three edge functions share a sign, z-buffer min
// through a 32-bit atomicMin on the bits of z >= 0.
//
// Every floating-point step is a single rounded IEEE operation in a fixed
// order (no contraction into FMAs): double precision for the extraction (for
// either field type), single precision for the image, so the results are those
// of the same arithmetic done step by step.  Both kernels spread uneven work
// (triangles per cube, pixels per triangle) over full warps through lists in
// shared memory, because one FP64 instruction costs a warp 16 clocks here.
#include <cmath>

#include "fe_internal.cuh"
#include "widen.cuh"

namespace fe {

constexpr int ISO_THREADS = 256;
constexpr int ISO_CH = 128;        // cubes (and threads) per block of the count and emit passes
constexpr int ISO_MAXE = 13;       // cut edges of a cube, at most (over the 256 sign patterns)
constexpr int ISO_MAXT = 12;       // triangles of a cube, at most

__device__ __forceinline__ double mul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double add(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double sub(double a, double b) { return __dsub_rn(a, b); }

__device__ __forceinline__ double tri_area(const double (&p)[9]) {
  const double e1[3] = {p[3] - p[0], p[4] - p[1], p[5] - p[2]};
  const double e2[3] = {p[6] - p[0], p[7] - p[1], p[8] - p[2]};
  const double c0 = e1[1] * e2[2] - e1[2] * e2[1];
  const double c1 = e1[2] * e2[0] - e1[0] * e2[2];
  const double c2 = e1[0] * e2[1] - e1[1] * e2[0];
  return 0.5 * sqrt(c0 * c0 + c1 * c1 + c2 * c2);
}

// The 19 edges of the split: corner pairs (a, b) with a's bits among b's, in order of a, then b.
__constant__ unsigned char kIsoEdge[19] = {0x10, 0x20, 0x30, 0x40, 0x50, 0x60, 0x70, 0x31, 0x51, 0x71,
                                           0x32, 0x62, 0x72, 0x73, 0x54, 0x64, 0x74, 0x75, 0x76};  // b << 4 | a

// Corner q (0..3) of tetrahedron n: the paths 0 -> e_a -> e_a + e_b -> 7.
__host__ __device__ constexpr int iso_tet(int n, int q) {
  return q == 0 ? 0 : q == 3 ? 7 : q == 1 ? (n < 2 ? 1 : n < 4 ? 2 : 4)
                                          : (n == 0 || n == 2 ? 3 : n == 1 || n == 4 ? 5 : 6);
}
__host__ __device__ constexpr int iso_edge_id(int a, int b) {  // a, b in either order
  const int lo = a < b ? a : b, hi = a < b ? b : a;
  int id = 0;
  for (int x = 0; x < 8; ++x)
    for (int y = x + 1; y < 8; ++y)
      if ((x & y) == x) {
        if (x == lo && y == hi) return id;
        ++id;
      }
  return -1;
}

// Triangle table: entry (n * 16 + pattern) * 2 + sub = the edge ids of its three points, 5 bits each.
// One corner apart (a; b, c, d the others in order): P(a,b) P(a,c) P(a,d); two in (a, b), two out
// (c, d): P(a,c) P(a,d) P(b,d), then P(a,c) P(b,d) P(b,c).
struct IsoTable {
  unsigned short e[6 * 16 * 2];
};
constexpr IsoTable iso_table() {
  IsoTable t{};
  for (int n = 0; n < 6; ++n)
    for (int p = 1; p < 15; ++p) {
      int in[4] = {}, out[4] = {}, ni = 0, no = 0;
      for (int q = 0; q < 4; ++q) {
        if ((p >> q) & 1) in[ni++] = iso_tet(n, q);
        else out[no++] = iso_tet(n, q);
      }
      auto pack = [](int x, int y, int z) { return (unsigned short)(x | (y << 5) | (z << 10)); };
      unsigned short* d = &t.e[(n * 16 + p) * 2];
      if (ni == 2) {
        const int ac = iso_edge_id(in[0], out[0]), ad = iso_edge_id(in[0], out[1]);
        const int bc = iso_edge_id(in[1], out[0]), bd = iso_edge_id(in[1], out[1]);
        d[0] = pack(ac, ad, bd);
        d[1] = pack(ac, bd, bc);
      } else {
        const int lone = ni == 1 ? in[0] : out[0];
        const int* r = ni == 1 ? out : in;
        d[0] = pack(iso_edge_id(lone, r[0]), iso_edge_id(lone, r[1]), iso_edge_id(lone, r[2]));
      }
    }
  return t;
}
__constant__ IsoTable kIsoTable = iso_table();

// pattern of tetrahedron N's corners from the cube's corner bits
template <int N>
__device__ __forceinline__ int tet_bits(int mask) {
  return ((mask >> iso_tet(N, 0)) & 1) | (((mask >> iso_tet(N, 1)) & 1) << 1) | (((mask >> iso_tet(N, 2)) & 1) << 2) |
         (((mask >> iso_tet(N, 3)) & 1) << 3);
}
__device__ __forceinline__ int tet_count(int bits) {
  const int n = __popc(bits);
  return (n & 1) ? 1 : (n == 2 ? 2 : 0);
}
__device__ __forceinline__ int cube_count(int mask) {
  return tet_count(tet_bits<0>(mask)) + tet_count(tet_bits<1>(mask)) + tet_count(tet_bits<2>(mask)) +
         tet_count(tet_bits<3>(mask)) + tet_count(tet_bits<4>(mask)) + tet_count(tet_bits<5>(mask));
}

// v > iso for a value of the field type.  FP32: against iso rounded down, the same verdict for every v.
__device__ __forceinline__ double iso_level(double iso, double) { return iso; }
__device__ __forceinline__ float iso_level(double iso, float) { return __double2float_rd(iso); }

// the eight corner values of cube c (periodic)
template <typename T>
__device__ __forceinline__ void cube_values(const T* __restrict__ f, int N, long c, T (&v)[8]) {
  const int i = (int)(c % N), j = (int)((c / N) % N), k = (int)(c / ((long)N * N));
  const int i1 = i + 1 < N ? i + 1 : 0, j1 = j + 1 < N ? j + 1 : 0, k1 = k + 1 < N ? k + 1 : 0;
#pragma unroll
  for (int b = 0; b < 8; ++b)
    v[b] = f[(b & 1 ? i1 : i) + (long)N * ((b & 2 ? j1 : j) + (long)N * (b & 4 ? k1 : k))];
}
template <typename T>
__device__ __forceinline__ int cube_mask(const T (&v)[8], T level) {
  int m = 0;
#pragma unroll
  for (int b = 0; b < 8; ++b) m |= (v[b] > level ? 1 : 0) << b;
  return m;
}

// inclusive scan of one value per thread over the block's ISO_CH threads
__device__ __forceinline__ int iso_scan(int v, int* warp_sum) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += t;
  }
  if (lane == 31) warp_sum[w] = v;
  __syncthreads();
  for (int q = 0; q < w; ++q) v += warp_sum[q];
  __syncthreads();
  return v;
}

// triangles of the cubes of each block
template <typename T>
__global__ void __launch_bounds__(ISO_CH) k_iso_count(const T* __restrict__ f, int N, double iso,
                                                      int* __restrict__ bsum) {
  __shared__ int ws[ISO_CH / 32];
  const long c = (long)blockIdx.x * ISO_CH + threadIdx.x;
  int n = 0;
  if (c < (long)N * N * N) {
    T v[8];
    cube_values<T>(f, N, c, v);
    n = cube_count(cube_mask<T>(v, iso_level(iso, T())));
  }
  n = __reduce_add_sync(0xffffffffu, n);
  if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = n;
  __syncthreads();
  if (threadIdx.x == 0) {
    n = 0;
    for (int w = 0; w < ISO_CH / 32; ++w) n += ws[w];
    bsum[blockIdx.x] = n;
  }
}

// boff[b] = triangles before block b, boff[nb] = all (one block; each thread a run of blocks)
constexpr int ISO_SCAN = 1024;
__global__ void __launch_bounds__(ISO_SCAN) k_iso_scan(const int* __restrict__ bsum, long nb,
                                                       long long* __restrict__ boff) {
  __shared__ long long sh[ISO_SCAN];
  const long per = (nb + ISO_SCAN - 1) / ISO_SCAN, b0 = min(per * threadIdx.x, nb), b1 = min(b0 + per, nb);
  long long s = 0;
  for (long b = b0; b < b1; ++b) s += bsum[b];
  sh[threadIdx.x] = s;
  __syncthreads();
  for (int o = 1; o < ISO_SCAN; o <<= 1) {
    const long long t = threadIdx.x >= o ? sh[threadIdx.x - o] : 0;
    __syncthreads();
    sh[threadIdx.x] += t;
    __syncthreads();
  }
  long long run = sh[threadIdx.x] - s;
  for (long b = b0; b < b1; ++b) {
    boff[b] = run;
    run += bsum[b];
  }
  if (threadIdx.x == ISO_SCAN - 1) boff[nb] = sh[ISO_SCAN - 1];
}

// cell-centre coordinates c_i = (i + 1/2) h, i = 0 .. N (one rounding each), c_{i+1} - c_i after them
__global__ void k_iso_centres(double* __restrict__ c, int N, double h) {
  for (int i = threadIdx.x; i <= N; i += blockDim.x) {
    const double a = mul((double)i + 0.5, h);
    c[i] = a;
    if (i < N) c[N + 1 + i] = sub(mul((double)(i + 1) + 0.5, h), a);
  }
}

// Emit: a block lists the cut edges and the triangles of its cubes, forms the edge parameters
// t = (iso - f_a) / (f_b - f_a) once per edge, then the triangles, each list over full warps, and
// writes the triangles through shared memory as one contiguous run.  About 25 FP64 operations per
// edge and 60 per triangle (area included) bound it.  One cube per thread, its tetrahedra in
// divergent branches and every point evaluated for each of its triangles, took 4.66 ms on the Q surface of a
// 192^3 turbulent flow against 0.89 ms.
template <typename T>
__global__ void __launch_bounds__(ISO_CH) k_iso_emit(const T* __restrict__ f, int N, double iso,
                                                     const double* __restrict__ cen,
                                                     const long long* __restrict__ boff, double* __restrict__ tri,
                                                     long long max_tri, double* __restrict__ apart) {
  __shared__ double ts[ISO_CH * ISO_MAXE];
  __shared__ double stage[ISO_CH * 9];
  __shared__ T val[8][ISO_CH];
  __shared__ unsigned short el[ISO_CH * ISO_MAXE], tl[ISO_CH * ISO_MAXT];
  __shared__ unsigned short eoff[ISO_CH];
  __shared__ unsigned char masks[ISO_CH];
  __shared__ unsigned emask[ISO_CH];
  __shared__ unsigned short table[6 * 16 * 2];
  __shared__ int ws[ISO_CH / 32];
  __shared__ double red[ISO_CH / 32];
  const int tid = threadIdx.x;
  const long long t0 = boff[blockIdx.x];
  const int nt = (int)(boff[blockIdx.x + 1] - t0);
  if (nt == 0) {
    if (tid == 0) apart[blockIdx.x] = 0.0;
    return;
  }
  const long base = (long)blockIdx.x * ISO_CH, c = base + tid, n = (long)N * N * N;
  for (int q = tid; q < 6 * 16 * 2; q += ISO_CH) table[q] = kIsoTable.e[q];
  int mask = 0;
  if (c < n) {
    T v[8];
    cube_values<T>(f, N, c, v);
    mask = cube_mask<T>(v, iso_level(iso, T()));
#pragma unroll
    for (int b = 0; b < 8; ++b) val[b][tid] = v[b];
  }
  unsigned cut = 0;
#pragma unroll
  for (int e = 0; e < 19; ++e) {
    const int a = kIsoEdge[e] & 15, b = kIsoEdge[e] >> 4;
    cut |= (unsigned)(((mask >> a) ^ (mask >> b)) & 1) << e;
  }
  masks[tid] = (unsigned char)mask;
  emask[tid] = cut;
  const int mine = cube_count(mask), ne = __popc(cut);
  int to = iso_scan(mine, ws) - mine, eo = iso_scan(ne, ws);
  __shared__ int etotal;
  if (tid == ISO_CH - 1) etotal = eo;
  eo -= ne;
  eoff[tid] = (unsigned short)eo;
  for (unsigned m = cut; m; m &= m - 1) el[eo++] = (unsigned short)((tid << 5) | (__ffs(m) - 1));
  auto list = [&](int nth, int bits) {
    const int k = tet_count(bits);
    for (int q = 0; q < k; ++q) tl[to++] = (unsigned short)((tid << 4) | (nth << 1) | q);
  };
  if (mine) {
    list(0, tet_bits<0>(mask));
    list(1, tet_bits<1>(mask));
    list(2, tet_bits<2>(mask));
    list(3, tet_bits<3>(mask));
    list(4, tet_bits<4>(mask));
    list(5, tet_bits<5>(mask));
  }
  __syncthreads();
  for (int q = tid; q < etotal; q += ISO_CH) {
    const int w = el[q], e = kIsoEdge[w & 31], cube = w >> 5;
    const double fa = widen(val[e & 15][cube]), fb = widen(val[e >> 4][cube]);
    ts[q] = (iso - fa) / sub(fb, fa);
  }
  __syncthreads();
  double area = 0.0;
  for (int q0 = 0; q0 < nt; q0 += ISO_CH) {
    const int q = q0 + tid;
    if (q < nt) {
      const int w = tl[q], cube = w >> 4, nth = (w >> 1) & 7;
      const int m = masks[cube];
      const unsigned cm = emask[cube];
      int bits = 0;
#pragma unroll
      for (int x = 0; x < 4; ++x) bits |= ((m >> iso_tet(nth, x)) & 1) << x;
      const int pts = table[(nth * 16 + bits) * 2 + (w & 1)];
      const long g = base + cube;
      const int ci[3] = {(int)(g % N), (int)((g / N) % N), (int)(g / ((long)N * N))};
      double c0[3], c1[3], dc[3], p[9];
#pragma unroll
      for (int x = 0; x < 3; ++x) {
        c0[x] = cen[ci[x]];
        c1[x] = cen[ci[x] + 1];
        dc[x] = cen[N + 1 + ci[x]];
      }
#pragma unroll
      for (int v = 0; v < 3; ++v) {
        const int id = (pts >> (5 * v)) & 31, e = kIsoEdge[id];
        const double t = ts[eoff[cube] + __popc(cm & ((1u << id) - 1u))];
#pragma unroll
        for (int x = 0; x < 3; ++x) {
          const int a = (e >> x) & 1, b = (e >> (4 + x)) & 1;
          p[3 * v + x] = add(a ? c1[x] : c0[x], mul(t, a != b ? dc[x] : 0.0));
        }
      }
      area += tri_area(p);
#pragma unroll
      for (int x = 0; x < 9; ++x) stage[tid * 9 + x] = p[x];
    }
    __syncthreads();
    const long long room = max_tri - (t0 + q0);
    const int now = (int)min((long long)min(ISO_CH, nt - q0), room > 0 ? room : 0LL);
    if (tri)
      for (int x = tid; x < now * 9; x += ISO_CH) tri[(t0 + q0) * 9 + x] = stage[x];
    __syncthreads();
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) area += __shfl_down_sync(0xffffffffu, area, o);
  if ((tid & 31) == 0) red[tid >> 5] = area;
  __syncthreads();
  if (tid == 0) {
    for (int w = 1; w < ISO_CH / 32; ++w) area += red[w];
    apart[blockIdx.x] = area;
  }
}

// total area: the block sums in a fixed order (one block)
__global__ void __launch_bounds__(ISO_SCAN) k_iso_area(const double* __restrict__ apart, long nb,
                                                       double* __restrict__ area) {
  __shared__ double sh[ISO_SCAN];
  double s = 0.0;
  for (long b = threadIdx.x; b < nb; b += ISO_SCAN) s += apart[b];
  sh[threadIdx.x] = s;
  __syncthreads();
  for (int o = ISO_SCAN / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) *area = sh[0];
}

__device__ __forceinline__ float fmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float fsub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float fadd(float a, float b) { return __fadd_rn(a, b); }

__device__ __forceinline__ float edge_fn(float xa, float ya, float xb, float yb, float px, float py) {
  return fsub(fmul(fsub(xb, xa), fsub(py, ya)), fmul(fsub(yb, ya), fsub(px, xa)));
}

__global__ void k_fill_u32(unsigned* a, long n, unsigned v) {
  for (long q = blockIdx.x * (long)blockDim.x + threadIdx.x; q < n; q += (long)gridDim.x * blockDim.x) a[q] = v;
}

// one thread per triangle; the bits of a float z >= 0 are ordered like z
__global__ void __launch_bounds__(ISO_THREADS) k_raster(const double* __restrict__ tri, long long ntri, int W,
                                                        double step, unsigned* __restrict__ depth) {
  for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < ntri;
       q += (long long)gridDim.x * blockDim.x) {
    const double* p = tri + q * 9;
    const double x0 = p[0], y0 = p[1];
    const float X1 = (float)(p[3] - x0), Y1 = (float)(p[4] - y0), X2 = (float)(p[6] - x0), Y2 = (float)(p[7] - y0);
    const float Z0 = (float)p[2], Z1 = (float)p[5], Z2 = (float)p[8];
    if (fsub(fmul(X1, Y2), fmul(Y1, X2)) == 0.f) continue;
    const int lo_x = max((int)floor(fmin(x0, fmin(p[3], p[6])) / step - 0.5) - 1, 0);
    const int hi_x = min((int)ceil(fmax(x0, fmax(p[3], p[6])) / step - 0.5) + 1, W - 1);
    const int lo_y = max((int)floor(fmin(y0, fmin(p[4], p[7])) / step - 0.5) - 1, 0);
    const int hi_y = min((int)ceil(fmax(y0, fmax(p[4], p[7])) / step - 0.5) + 1, W - 1);
    for (int py = lo_y; py <= hi_y; ++py) {
      const float CY = (float)__dsub_rn(__dmul_rn((double)py + 0.5, step), y0);
      for (int px = lo_x; px <= hi_x; ++px) {
        const float CX = (float)__dsub_rn(__dmul_rn((double)px + 0.5, step), x0);
        const float e12 = edge_fn(X1, Y1, X2, Y2, CX, CY);
        const float e20 = edge_fn(X2, Y2, 0.f, 0.f, CX, CY);
        const float e01 = edge_fn(0.f, 0.f, X1, Y1, CX, CY);
        if ((e12 >= 0.f && e20 >= 0.f && e01 >= 0.f) || (e12 <= 0.f && e20 <= 0.f && e01 <= 0.f)) {
          const float num = fadd(fadd(fmul(e12, Z0), fmul(e20, Z1)), fmul(e01, Z2));
          const float z = __fdiv_rn(num, fadd(fadd(e12, e20), e01));
          // the depth only decreases, so a read that is already <= z (even an older value) means the
          // atomic would change nothing: most covered pixels of a many-layered surface skip it
          unsigned* d = &depth[(long)py * W + px];
          const unsigned zb = __float_as_uint(z);
          if (z >= 0.f && zb < *d) atomicMin(d, zb);
        }
      }
    }
  }
}

static int iso_grid(long n, int nsm) {
  const long g = (n + ISO_THREADS - 1) / ISO_THREADS;
  const long cap = (long)nsm * 8;
  return (int)(g < cap ? g : cap);
}

static long iso_blocks(long n) { return (n + ISO_CH - 1) / ISO_CH; }

// work: boff (nb + 1 long longs), area and apart (1 + nb doubles), centres (2 N + 2 doubles), bsum (nb ints)
size_t iso_work_bytes(int N) {
  const size_t nb = (size_t)iso_blocks((long)N * N * N);
  return (nb + 1) * sizeof(long long) + (nb + 1 + 2 * (size_t)N + 2) * sizeof(double) + nb * sizeof(int);
}

template <typename T>
int isosurface(const T* f, int N, double iso, double* tri, long long max_tri, void* work, long long* ntri,
               double* area, cudaStream_t st) {
  const long nb = iso_blocks((long)N * N * N);
  long long* boff = (long long*)work;
  double* total = (double*)(boff + nb + 1);  // after boff[nb]: one copy brings the count and the area
  double* apart = total + 1;
  double* cen = apart + nb;
  int* bsum = (int*)(cen + 2 * (size_t)N + 2);
  k_iso_centres<<<1, ISO_THREADS, 0, st>>>(cen, N, 2.0 * M_PI / N);
  k_iso_count<T><<<(unsigned)nb, ISO_CH, 0, st>>>(f, N, iso, bsum);
  k_iso_scan<<<1, ISO_SCAN, 0, st>>>(bsum, nb, boff);
  k_iso_emit<T><<<(unsigned)nb, ISO_CH, 0, st>>>(f, N, iso, cen, boff, tri, max_tri, apart);
  k_iso_area<<<1, ISO_SCAN, 0, st>>>(apart, nb, total);
  struct {
    long long n;
    double a;
  } res;
  if (cudaMemcpyAsync(&res, boff + nb, sizeof(res), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
      cudaStreamSynchronize(st) != cudaSuccess || cudaGetLastError() != cudaSuccess)
    return FE_ERR_CUDA;
  *ntri = res.n;
  *area = res.a;
  return FE_OK;
}

int raster_depth(const double* tri, long long ntri, int W, double extent, float* depth, int nsm, cudaStream_t st) {
  const long npx = (long)W * W;
  k_fill_u32<<<iso_grid(npx, nsm), ISO_THREADS, 0, st>>>((unsigned*)depth, npx, 0x7F800000u);
  if (ntri > 0)
    k_raster<<<iso_grid((long)ntri, nsm), ISO_THREADS, 0, st>>>(tri, ntri, W, extent / W, (unsigned*)depth);
  return cudaGetLastError() == cudaSuccess ? FE_OK : FE_ERR_CUDA;
}

template int isosurface<double>(const double*, int, double, double*, long long, void*, long long*, double*,
                                cudaStream_t);
template int isosurface<float>(const float*, int, double, double*, long long, void*, long long*, double*,
                               cudaStream_t);

}  // namespace fe
