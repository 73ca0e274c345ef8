// les.cu -- a-priori analysis of the sub-grid stress for large-eddy simulation
// (the paper's Sec. 1 names LES of the plume as the goal of its DNS, Sec. 2
// the a-priori use of the DNS database; neither names a filter or a model).
//
// Filter: top-hat of width Delta = 2 m h per axis by the trapezoidal rule
// (end points at half weight), applied as a tensor product.  Favre filtering:
// rho_bar = bar(rho), u~_i = bar(rho u_i) / rho_bar; sub-grid stress
// tau_ij = bar(rho u_i u_j) - bar(rho u_i) bar(rho u_j) / rho_bar.  Resolved
// strain from the Gauss cell gradient of u~ (the method's own Gc, in the
// compact form (f_{i-2} - 10 f_{i-1} + 10 f_{i+1} - f_{i+2}) / 16h), model
// slot: Smagorinsky B_ij = -2 rho_bar Delta^2 |S| S^d_ij.  Statistics: means
// of tau_kk / 2, -tau^d:S, tau^d:B, B:B, tau^d:tau^d and B:S.
//
// FP32 fields with m <= 4: one pass reads rho and u (4 words per cell), filters along all three
// axes and writes rho_bar, u~ and tau (10); the statistics pass reads them back (10).  FP64 fields
// (bound by the FP64 pipe, for which the halo rows of that pass are extra work) and wider filters:
// an x pass (4 + 10), y and z passes (20 each) and the closing pass (20) first.
#include <cmath>

#include "gradtile.cuh"

namespace fe {

constexpr int LES_NF = 10;       // rho, rho u (3), rho u u (6: 00 01 02 11 12 22)
constexpr int LES_THREADS = 256;

template <typename T>
struct LesPtrs {
  T* f[LES_NF];
};

__device__ __forceinline__ long les_wrap(long i, long N) { return i < 0 ? i + N : (i >= N ? i - N : i); }

// trapezoidal top-hat weight of offset o in -m..m
template <typename T>
__device__ __forceinline__ T les_w(int o, int m) {
  const T w = T(1) / T(2 * m);
  return (o == -m || o == m) ? T(0.5) * w : w;
}

// x pass: products formed on the fly, filtered along x
template <typename T>
__global__ void __launch_bounds__(LES_THREADS) k_les_x(const T* __restrict__ rho, const T* __restrict__ u0,
                                                       const T* __restrict__ u1, const T* __restrict__ u2, int N,
                                                       int m, LesPtrs<T> out) {
  const long n = (long)N * N * N;
  for (long c = blockIdx.x * (long)blockDim.x + threadIdx.x; c < n; c += (long)gridDim.x * blockDim.x) {
    const long i = c % N, row = c - i;
    T acc[LES_NF];
#pragma unroll
    for (int q = 0; q < LES_NF; ++q) acc[q] = T(0);
    for (int o = -m; o <= m; ++o) {
      const long s = row + les_wrap(i + o, N);
      const T w = les_w<T>(o, m);
      const T r = rho[s], a = u0[s], b = u1[s], d = u2[s];
      const T ra = r * a, rb = r * b, rd = r * d;
      acc[0] += w * r;
      acc[1] += w * ra;
      acc[2] += w * rb;
      acc[3] += w * rd;
      acc[4] += w * (ra * a);
      acc[5] += w * (ra * b);
      acc[6] += w * (ra * d);
      acc[7] += w * (rb * b);
      acc[8] += w * (rb * d);
      acc[9] += w * (rd * d);
    }
#pragma unroll
    for (int q = 0; q < LES_NF; ++q) out.f[q][c] = acc[q];
  }
}

// y (axis 1) or z (axis 2) pass over the ten fields
template <typename T>
__global__ void __launch_bounds__(LES_THREADS) k_les_line(LesPtrs<T> in, LesPtrs<T> out, int N, int m, int axis) {
  const long n = (long)N * N * N;
  const long stride = axis == 1 ? N : (long)N * N;
  for (long c = blockIdx.x * (long)blockDim.x + threadIdx.x; c < n; c += (long)gridDim.x * blockDim.x) {
    const long pos = (c / stride) % N;
    const long base = c - pos * stride;
    T acc[LES_NF];
#pragma unroll
    for (int q = 0; q < LES_NF; ++q) acc[q] = T(0);
    for (int o = -m; o <= m; ++o) {
      const long s = base + les_wrap(pos + o, N) * stride;
      const T w = les_w<T>(o, m);
#pragma unroll
      for (int q = 0; q < LES_NF; ++q) acc[q] += w * in.f[q][s];
    }
#pragma unroll
    for (int q = 0; q < LES_NF; ++q) out.f[q][c] = acc[q];
  }
}

// y (axis 1) or z (axis 2) pass with a register window: each thread makes LES_OUTS consecutive outputs
// along the axis from LES_OUTS + 2M loads per field (N a multiple of LES_OUTS); the weighted sum of
// each output runs over the offsets -M..M in order, as in k_les_line.
constexpr int LES_OUTS = 8;
template <typename T, int M>
__global__ void __launch_bounds__(LES_THREADS) k_les_win(LesPtrs<T> in, LesPtrs<T> out, int N, int axis) {
  const long nb = (long)N * N * (N / LES_OUTS);
  const long stride = axis == 1 ? N : (long)N * N;
  const T w = T(1) / T(2 * M), we = T(0.5) * w;
  for (long q = blockIdx.x * (long)blockDim.x + threadIdx.x; q < nb; q += (long)gridDim.x * blockDim.x) {
    // q = i + N (a + N b) with a in [0, N), b in [0, N / LES_OUTS): axis 1: (i, k = a, block of j = b);
    // axis 2: (i, j = a, block of k = b); the outputs are p0 .. p0 + LES_OUTS - 1 < N along the axis
    const long i = q % N, a = (q / N) % N, b = q / ((long)N * N);
    const long base = axis == 1 ? i + (long)N * (long)N * a : i + (long)N * a;
    const long p0 = b * LES_OUTS;
#pragma unroll
    for (int f = 0; f < LES_NF; ++f) {  // unrolled: the field pointers stay in registers
      const T* src = in.f[f];
      T win[LES_OUTS + 2 * M];
#pragma unroll
      for (int t = 0; t < LES_OUTS + 2 * M; ++t) win[t] = src[base + les_wrap(p0 - M + t, N) * stride];
      T* dst = out.f[f];
#pragma unroll
      for (int o = 0; o < LES_OUTS; ++o) {
        T acc = T(0);
#pragma unroll
        for (int t = 0; t <= 2 * M; ++t) acc += ((t == 0 || t == 2 * M) ? we : w) * win[o + t];
        dst[base + (p0 + o) * stride] = acc;
      }
    }
  }
}

// rho_bar, u~ and tau from the ten filtered quantities of a cell
template <typename T>
__device__ __forceinline__ void les_close(const T (&v)[LES_NF], T (&o)[LES_NF]) {
  const T ir = T(1) / v[0];
  o[0] = v[0];
#pragma unroll
  for (int q = 1; q < 4; ++q) o[q] = v[q] * ir;
  o[4] = v[4] - v[1] * v[1] * ir;
  o[5] = v[5] - v[1] * v[2] * ir;
  o[6] = v[6] - v[1] * v[3] * ir;
  o[7] = v[7] - v[2] * v[2] * ir;
  o[8] = v[8] - v[2] * v[3] * ir;
  o[9] = v[9] - v[3] * v[3] * ir;
}

template <typename T>
__global__ void __launch_bounds__(LES_THREADS) k_les_close(LesPtrs<T> F, T* __restrict__ out, long n) {
  for (long c = blockIdx.x * (long)blockDim.x + threadIdx.x; c < n; c += (long)gridDim.x * blockDim.x) {
    T v[LES_NF], o[LES_NF];
#pragma unroll
    for (int q = 0; q < LES_NF; ++q) v[q] = F.f[q][c];
    les_close<T>(v, o);
#pragma unroll
    for (int q = 0; q < LES_NF; ++q) out[q * n + c] = o[q];
  }
}

// All three filter passes and the closing in one (FP32 fields): a block walks kLesTz planes of a
// 32 x 8 tile.  rho and u of a plane with a halo of M cells are staged, the ten quantities filtered
// along x go to shared memory (tile rows and their y halo), a thread filters its column's along y
// and keeps the last 2 M + 1 planes of them in registers for z.  24 words of traffic per cell with
// the statistics pass instead of 74, at the price of (8 + 2 M) / 8 times the x work; products and
// taps are summed in the order of the separate passes.  The next plane's loads are in flight while
// a plane is filtered.
constexpr int kLesTz = 32;
template <int M>
__global__ void __launch_bounds__(NTHR) k_les_fused(const float* __restrict__ rho, const float* __restrict__ u0,
                                                    const float* __restrict__ u1, const float* __restrict__ u2, int N,
                                                    float* __restrict__ out) {
  constexpr int W = TX + 2 * M, R = TY + 2 * M, CELLS = W * R, PER = (CELLS + NTHR - 1) / NTHR;
  __shared__ float in[4][CELLS];
  __shared__ float xf[LES_NF][R][TX];
  const int tid = threadIdx.x + TX * threadIdx.y;
  const int i = blockIdx.x * TX + threadIdx.x, j = blockIdx.y * TY + threadIdx.y;
  const int k0 = blockIdx.z * kLesTz, kend = min(k0 + kLesTz, N);
  const size_t NN = (size_t)N * N;
  const long n = (long)N * NN;
  const float* f[4] = {rho, u0, u1, u2};
  const float w = 1.f / (2 * M), we = 0.5f * w;
  int off[PER];
#pragma unroll
  for (int q = 0; q < PER; ++q) {
    const int t = min(tid + q * NTHR, CELLS - 1);
    const int x = (int)(blockIdx.x * TX) - M + t % W, y = (int)(blockIdx.y * TY) - M + t / W;
    off[q] = (x + N) % N + N * ((y + N) % N);
  }
  float ld[4][PER], win[LES_NF][2 * M + 1];
  auto fetch = [&](int k) {
    const size_t p = (size_t)((k + N) % N) * NN;
#pragma unroll
    for (int l = 0; l < 4; ++l)
#pragma unroll
      for (int q = 0; q < PER; ++q) ld[l][q] = f[l][p + off[q]];
  };
  fetch(k0 - M);
  for (int k = k0 - M; k < kend + M; ++k) {
#pragma unroll
    for (int l = 0; l < 4; ++l)
#pragma unroll
      for (int q = 0; q < PER; ++q)
        if (tid + q * NTHR < CELLS) in[l][tid + q * NTHR] = ld[l][q];
    __syncthreads();
    if (k + 1 < kend + M) fetch(k + 1);
    for (int y = threadIdx.y; y < R; y += TY) {
      float acc[LES_NF];
#pragma unroll
      for (int q = 0; q < LES_NF; ++q) acc[q] = 0.f;
#pragma unroll
      for (int o = 0; o <= 2 * M; ++o) {
        const int s = y * W + threadIdx.x + o;
        const float t = (o == 0 || o == 2 * M) ? we : w;
        const float r = in[0][s], a = in[1][s], b = in[2][s], d = in[3][s];
        const float ra = r * a, rb = r * b, rd = r * d;
        acc[0] += t * r;
        acc[1] += t * ra;
        acc[2] += t * rb;
        acc[3] += t * rd;
        acc[4] += t * (ra * a);
        acc[5] += t * (ra * b);
        acc[6] += t * (ra * d);
        acc[7] += t * (rb * b);
        acc[8] += t * (rb * d);
        acc[9] += t * (rd * d);
      }
#pragma unroll
      for (int q = 0; q < LES_NF; ++q) xf[q][y][threadIdx.x] = acc[q];
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < LES_NF; ++q) {
      float acc = 0.f;
#pragma unroll
      for (int o = 0; o <= 2 * M; ++o)
        acc += ((o == 0 || o == 2 * M) ? we : w) * xf[q][threadIdx.y + o][threadIdx.x];
#pragma unroll
      for (int o = 0; o < 2 * M; ++o) win[q][o] = win[q][o + 1];
      win[q][2 * M] = acc;
    }
    if (k - M >= k0 && i < N && j < N) {
      float v[LES_NF], o[LES_NF];
#pragma unroll
      for (int q = 0; q < LES_NF; ++q) {
        float acc = 0.f;
#pragma unroll
        for (int t = 0; t <= 2 * M; ++t) acc += ((t == 0 || t == 2 * M) ? we : w) * win[q][t];
        v[q] = acc;
      }
      les_close<float>(v, o);
      const size_t c = (size_t)(k - M) * NN + (size_t)j * N + i;
#pragma unroll
      for (int q = 0; q < LES_NF; ++q) out[q * n + c] = o[q];
    }
  }
}

// symmetric tensors in the order 00 01 02 11 12 22
template <typename T>
__device__ __forceinline__ T les_contract(const T (&a)[6], const T (&b)[6]) {
  return a[0] * b[0] + a[3] * b[3] + a[5] * b[5] + T(2) * (a[1] * b[1] + a[2] * b[2] + a[4] * b[4]);
}

template <typename T>
__device__ __forceinline__ void les_dev(T (&a)[6]) {
  const T tr = (a[0] + a[3] + a[5]) * T(1.0 / 3.0);
  a[0] -= tr;
  a[3] -= tr;
  a[5] -= tr;
}

constexpr int LES_NS = 6;  // sums: tr tau, tau^d:S, tau^d:B, B:B, tau^d:tau^d, B:S

// Statistics of the ten fields f (rho_bar, u~ (3), tau (6)): block sums part[block][LES_NS].
template <typename T>
__global__ void __launch_bounds__(NTHR) k_les_stats(const T* __restrict__ f, int N, double ih, double delta,
                                                    double* __restrict__ part) {
  __shared__ T sh[3][kGradH][kGradW];
  const long n = (long)N * N * N;
  const T ihT = (T)ih, d2 = (T)(delta * delta);
  GradTile<T, T> t(f + n, f + 2 * n, f + 3 * n, N, sh);
  const int k0 = blockIdx.z * kGradTz, kend = min(k0 + kGradTz, N);
  T acc[LES_NS];
#pragma unroll
  for (int q = 0; q < LES_NS; ++q) acc[q] = T(0);
  t.start(k0);
  for (int k = k0; k < kend; ++k) {
    t.next(k);
    if (t.i >= N || t.j >= N) continue;
    const size_t c = t.plane(k) + t.own;
    const T rb = f[c];
    T tau[6];
#pragma unroll
    for (int q = 0; q < 6; ++q) tau[q] = f[(4 + q) * n + c];
    T g[3][3];  // g[a][b] = Gc_b u~_a
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        T v[4];
        t.line(a, b, v);
        g[a][b] = ((v[0] - v[3]) + T(10) * (v[2] - v[1])) * T(0.0625) * ihT;
      }
    T S[6] = {g[0][0], T(0.5) * (g[0][1] + g[1][0]), T(0.5) * (g[0][2] + g[2][0]), g[1][1],
              T(0.5) * (g[1][2] + g[2][1]), g[2][2]};
    const T mag = sqrt(T(2) * les_contract<T>(S, S));
    T Sd[6] = {S[0], S[1], S[2], S[3], S[4], S[5]};
    les_dev<T>(Sd);
    T B[6];
#pragma unroll
    for (int q = 0; q < 6; ++q) B[q] = T(-2) * rb * d2 * mag * Sd[q];
    T td[6] = {tau[0], tau[1], tau[2], tau[3], tau[4], tau[5]};
    les_dev<T>(td);
    acc[0] += tau[0] + tau[3] + tau[5];
    acc[1] += les_contract<T>(td, S);
    acc[2] += les_contract<T>(td, B);
    acc[3] += les_contract<T>(B, B);
    acc[4] += les_contract<T>(td, td);
    acc[5] += les_contract<T>(B, S);
  }
  __shared__ double red[NTHR / 32][LES_NS];
#pragma unroll
  for (int q = 0; q < LES_NS; ++q) {
    double v = (double)acc[q];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if ((t.tid & 31) == 0) red[t.tid >> 5][q] = v;
  }
  __syncthreads();
  if (t.tid < LES_NS) {
    double s = 0.0;
    for (int w = 0; w < NTHR / 32; ++w) s += red[w][t.tid];
    part[(size_t)(blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z)) * LES_NS + t.tid] = s;
  }
}

static int les_grid(long n, int nsm) {
  const long g = (n + LES_THREADS - 1) / LES_THREADS;
  const long cap = (long)nsm * 8;
  return (int)(g < cap ? g : cap);
}

template <typename T>
static bool les_fused(int m) {
  return sizeof(T) == 4 && m <= 4;
}

// Work memory: the ten fields of a caller that does not take them, or the two sets of the separate
// passes; then the block sums of the statistics and the sums.
size_t les_work_bytes(int N, int m, int word) {
  const dim3 g = grad_grid(N);
  const size_t n = (size_t)N * N * N, sets = word == 4 && les_fused<float>(m) ? 1 : 2;
  return (sets * LES_NF * n * word + 255) / 256 * 256 + ((size_t)g.x * g.y * g.z + 1) * LES_NS * sizeof(double);
}

// Statistics in stats[0..5]: delta, k_sgs, pi_sgs, cs2_opt, corr, pi_model (fixed-order sums); out: the
// ten fields rho_bar, u~ (3), tau (6), or null.
template <typename T>
int les_apriori(const T* rho, const T* u0, const T* u1, const T* u2, int N, int m, double cs, void* work, int nsm,
                T* out, double* stats, cudaStream_t st) {
  const long n = (long)N * N * N;
  const bool fused = les_fused<T>(m);
  T* A0 = static_cast<T*>(work);
  double* part = reinterpret_cast<double*>(static_cast<char*>(work) +
                                           ((size_t)(fused ? 1 : 2) * LES_NF * n * sizeof(T) + 255) / 256 * 256);
  T* f = out ? out : A0;
  if constexpr (sizeof(T) == 4) {
    if (fused) {
      const dim3 g((N + TX - 1) / TX, (N + TY - 1) / TY, (N + kLesTz - 1) / kLesTz), b(TX, TY);
      switch (m) {
        case 1: k_les_fused<1><<<g, b, 0, st>>>(rho, u0, u1, u2, N, f); break;
        case 2: k_les_fused<2><<<g, b, 0, st>>>(rho, u0, u1, u2, N, f); break;
        case 3: k_les_fused<3><<<g, b, 0, st>>>(rho, u0, u1, u2, N, f); break;
        default: k_les_fused<4><<<g, b, 0, st>>>(rho, u0, u1, u2, N, f); break;
      }
    }
  }
  if (!fused) {
    LesPtrs<T> A, Bp;
    for (int q = 0; q < LES_NF; ++q) {
      A.f[q] = A0 + q * n;
      Bp.f[q] = A0 + (LES_NF + q) * n;
    }
    const int grid = les_grid(n, nsm);
    k_les_x<T><<<grid, LES_THREADS, 0, st>>>(rho, u0, u1, u2, N, m, A);
    if (N % LES_OUTS == 0 && m <= 4) {
      const int gw = les_grid(n / LES_OUTS, nsm);
      for (int axis = 1; axis <= 2; ++axis) {
        const LesPtrs<T>& src = axis == 1 ? A : Bp;
        const LesPtrs<T>& dst = axis == 1 ? Bp : A;
        switch (m) {
          case 1: k_les_win<T, 1><<<gw, LES_THREADS, 0, st>>>(src, dst, N, axis); break;
          case 2: k_les_win<T, 2><<<gw, LES_THREADS, 0, st>>>(src, dst, N, axis); break;
          case 3: k_les_win<T, 3><<<gw, LES_THREADS, 0, st>>>(src, dst, N, axis); break;
          default: k_les_win<T, 4><<<gw, LES_THREADS, 0, st>>>(src, dst, N, axis); break;
        }
      }
    } else {
      k_les_line<T><<<grid, LES_THREADS, 0, st>>>(A, Bp, N, m, 1);
      k_les_line<T><<<grid, LES_THREADS, 0, st>>>(Bp, A, N, m, 2);
    }
    if (!out) f = Bp.f[0];  // the closing pass reads A
    k_les_close<T><<<grid, LES_THREADS, 0, st>>>(A, f, n);
  }
  const double h = 2.0 * M_PI / N, delta = 2.0 * m * h;
  const dim3 g = grad_grid(N);
  const int blocks = (int)(g.x * g.y * g.z);
  double* sums = part + (size_t)blocks * LES_NS;
  double s[LES_NS];
  k_les_stats<T><<<g, dim3(TX, TY), 0, st>>>(f, N, 1.0 / h, delta, part);
  k_sum_parts<<<LES_NS, NTHR, 0, st>>>(part, blocks, LES_NS, sums);
  if (cudaMemcpyAsync(s, sums, sizeof(s), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
      cudaStreamSynchronize(st) != cudaSuccess || cudaGetLastError() != cudaSuccess)
    return FE_ERR_CUDA;
  for (int q = 0; q < LES_NS; ++q) s[q] /= (double)n;
  stats[0] = delta;
  stats[1] = 0.5 * s[0];
  stats[2] = -s[1];
  stats[3] = s[3] > 0.0 ? s[2] / s[3] : 0.0;
  stats[4] = (s[3] > 0.0 && s[4] > 0.0) ? s[2] / std::sqrt(s[3] * s[4]) : 0.0;
  stats[5] = -cs * cs * s[5];
  return FE_OK;
}

template int les_apriori<double>(const double*, const double*, const double*, const double*, int, int, double, void*,
                                 int, double*, double*, cudaStream_t);
template int les_apriori<float>(const float*, const float*, const float*, const float*, int, int, double, void*, int,
                                float*, double*, cudaStream_t);

}  // namespace fe
