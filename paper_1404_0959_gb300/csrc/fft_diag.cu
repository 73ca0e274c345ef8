// fft_diag.cu -- spectral initial condition, turbulence diagnostics, Q field.
//
// Sec. 1 of arXiv:1404.0959: freely decaying homogeneous isotropic turbulence
// at r.m.s. Mach 0.2 / 0.5.  Sec. 2 par. 1: energy spectrum, enstrophy, kinetic
// energy and Taylor microscale; Fig. 1: density r.m.s.; Fig. 3: Q iso-surfaces.
//
// The 3D DFT is done as 1D transforms of the grid lines, several per block, with a
// mixed-radix Stockham autosort FFT in shared memory (FP64).  N = 2^a 3^b,
// N <= 512.  None of this is on the per-step hot path.
#include <vector>

#include "fe_internal.cuh"
#include "gradtile.cuh"

namespace fe {

template <typename T>
__device__ __forceinline__ T* F(const BoxDev& B, int slot) {
  return reinterpret_cast<T*>(B.f[slot]);
}

// ---- FFT -------------------------------------------------------------------------------
// A block transforms kFftLines lines at a time in shared memory, element x of line w at [x][w]:
// the eight lanes of a quarter-warp then read and write 128 contiguous bytes whatever the radix
// and the stage, and the lines of the y and z passes are loaded as contiguous runs.  The stages
// are Stockham butterflies of radix 16, 8, 4, 2 and 3 held in registers, twiddles from a table of
// the N-th roots of unity.  FP64 throughput (2 lanes per clock and SM) is the bound, so what counts
// is the number of FP64 instructions: 160 per radix-16 butterfly and 4 per twiddle, 6.3 thousand
// per 256-point line.  Evaluating the roots in the butterflies (sincospi per factor) took 29.5 ms
// per 256^3 pass where these take 0.9 ms (complex) and the real input halves the lines again.
constexpr int kFftThreads = 128;
constexpr int kFftLines = 8;
constexpr int kFftMaxN = 512;
constexpr int kFftGrid = 456;  // blocks of the binning pass: three per SM at N = 256 (64 KB each)

struct Radices {
  int n, r[12];
};

__device__ __forceinline__ double2 cadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 csub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
  return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ double2 cmul_mi(double2 a) { return make_double2(a.y, -a.x); }  // -i a

__device__ __forceinline__ void dft4(double2& a, double2& b, double2& c, double2& d) {
  const double2 p = cadd(a, c), q = csub(a, c), r = cadd(b, d), t = cmul_mi(csub(b, d));
  a = cadd(p, r);
  b = cadd(q, t);
  c = csub(p, r);
  d = csub(q, t);
}

// forward DFT of R values in registers, natural order
template <int R>
__device__ __forceinline__ void dft(double2 (&a)[R]);
template <>
__device__ __forceinline__ void dft<2>(double2 (&a)[2]) {
  const double2 t = csub(a[0], a[1]);
  a[0] = cadd(a[0], a[1]);
  a[1] = t;
}
template <>
__device__ __forceinline__ void dft<3>(double2 (&a)[3]) {
  const double c = 0.86602540378443864676;  // sqrt(3) / 2
  const double2 s = cadd(a[1], a[2]), d = cmul_mi(csub(a[1], a[2]));
  const double2 m = make_double2(a[0].x - 0.5 * s.x, a[0].y - 0.5 * s.y);
  a[0] = cadd(a[0], s);
  a[1] = make_double2(m.x + c * d.x, m.y + c * d.y);
  a[2] = make_double2(m.x - c * d.x, m.y - c * d.y);
}
template <>
__device__ __forceinline__ void dft<4>(double2 (&a)[4]) {
  dft4(a[0], a[1], a[2], a[3]);
}
template <>
__device__ __forceinline__ void dft<8>(double2 (&a)[8]) {
  const double c = 0.70710678118654752440;  // sqrt(1/2)
  double2 e[4], o[4];
#pragma unroll
  for (int t = 0; t < 4; ++t) {
    e[t] = cadd(a[t], a[t + 4]);
    o[t] = csub(a[t], a[t + 4]);
  }
  o[1] = make_double2(c * (o[1].x + o[1].y), c * (o[1].y - o[1].x));
  o[2] = cmul_mi(o[2]);
  o[3] = make_double2(c * (o[3].y - o[3].x), -c * (o[3].x + o[3].y));
  dft4(e[0], e[1], e[2], e[3]);
  dft4(o[0], o[1], o[2], o[3]);
#pragma unroll
  for (int t = 0; t < 4; ++t) {
    a[2 * t] = e[t];
    a[2 * t + 1] = o[t];
  }
}
template <>
__device__ __forceinline__ void dft<16>(double2 (&a)[16]) {
  const double c = 0.70710678118654752440;                                     // sqrt(1/2)
  const double c1 = 0.92387953251128675613, s1 = 0.38268343236508977173;       // cos, sin of pi/8
#pragma unroll
  for (int j = 0; j < 4; ++j) dft4(a[j], a[j + 4], a[j + 8], a[j + 12]);
  // a[j + 4 i] *= w^(i j), w = exp(-2 pi i / 16)
  const double2 w1 = make_double2(c1, -s1), w3 = make_double2(s1, -c1);
  a[5] = cmul(a[5], w1);
  a[6] = make_double2(c * (a[6].x + a[6].y), c * (a[6].y - a[6].x));
  a[7] = cmul(a[7], w3);
  a[9] = make_double2(c * (a[9].x + a[9].y), c * (a[9].y - a[9].x));
  a[10] = cmul_mi(a[10]);
  a[11] = make_double2(c * (a[11].y - a[11].x), -c * (a[11].x + a[11].y));
  a[13] = cmul(a[13], w3);
  a[14] = make_double2(c * (a[14].y - a[14].x), -c * (a[14].x + a[14].y));
  a[15] = cmul(a[15], make_double2(-c1, s1));
#pragma unroll
  for (int i = 0; i < 4; ++i) dft4(a[4 * i], a[4 * i + 1], a[4 * i + 2], a[4 * i + 3]);
  // value k = i + 4 t sits at a[4 i + t]: transpose
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int t = i + 1; t < 4; ++t) {
      const double2 x = a[4 * i + t];
      a[4 * i + t] = a[4 * t + i];
      a[4 * t + i] = x;
    }
}

// One Stockham stage of radix R on the block's lines: n = remaining length, s = N / n.
template <int R>
__device__ __forceinline__ void fft_stage(const double2* X, double2* Y, int n, int s, const double2* __restrict__ tw) {
  const int m = n / R;
  for (int idx = threadIdx.x; idx < m * s * kFftLines; idx += kFftThreads) {
    const int w = idx % kFftLines, b = idx / kFftLines;
    const int p = b / s, q = b - p * s;
    double2 a[R];
#pragma unroll
    for (int t = 0; t < R; ++t) a[t] = X[(q + s * (p + t * m)) * kFftLines + w];
    dft<R>(a);
    if (m > 1) {
#pragma unroll
      for (int t = 1; t < R; ++t) a[t] = cmul(a[t], __ldg(&tw[p * t * s]));
    }
#pragma unroll
    for (int t = 0; t < R; ++t) Y[(q + s * (R * p + t)) * kFftLines + w] = a[t];
  }
}

// All stages; returns the buffer (buf or buf + N * kFftLines) that holds the result.
__device__ __forceinline__ double2* fft_block(double2* buf, int N, const Radices& rad, const double2* tw) {
  double2 *X = buf, *Y = buf + (size_t)N * kFftLines;
  int n = N, s = 1;
  for (int st = 0; st < rad.n; ++st) {
    __syncthreads();
    const int r = rad.r[st];
    if (r == 16) fft_stage<16>(X, Y, n, s, tw);
    else if (r == 8) fft_stage<8>(X, Y, n, s, tw);
    else if (r == 4) fft_stage<4>(X, Y, n, s, tw);
    else if (r == 3) fft_stage<3>(X, Y, n, s, tw);
    else fft_stage<2>(X, Y, n, s, tw);
    double2* z = X;
    X = Y;
    Y = z;
    n /= r;
    s *= r;
  }
  __syncthreads();
  return X;
}

__global__ void k_roots(double2* tw, int N) {
  for (int q = threadIdx.x; q < N; q += blockDim.x) {
    double sn, cs;
    sincospi(-2.0 * (double)q / (double)N, &sn, &cs);
    tw[q] = make_double2(cs, sn);
  }
}

// x pass of a real field: two rows at a time as one complex line (a + i b), the half spectra
// k = 0 .. H - 1 (H = N / 2 + 1) of both separated after it.  They are stored without the factor
// 1/2 of the separation (the binning takes 1/4 off the squares, exactly).
template <typename T, int VL>
__global__ void __launch_bounds__(kFftThreads) k_fft_rows(const T* __restrict__ f, double2* __restrict__ out, int N,
                                                          Radices rad, const double2* __restrict__ tw) {
  extern __shared__ double2 fft_buf[];
  const int H = N / 2 + 1, rows = N * N;
  const int l0 = blockIdx.x * 2 * kFftLines;
  for (int idx = threadIdx.x; idx < (N / VL) * kFftLines; idx += kFftThreads) {
    const int w = idx % kFftLines, x = idx / kFftLines * VL;
    const int ra = l0 + 2 * w;
    T a[VL], b[VL];
#pragma unroll
    for (int e = 0; e < VL; ++e) a[e] = b[e] = T(0);
    if constexpr (VL == 1) {
      if (ra < rows) a[0] = f[(size_t)ra * N + x];
      if (ra + 1 < rows) b[0] = f[(size_t)(ra + 1) * N + x];
    } else {  // 16-byte loads: N is a multiple of VL and the field 16-byte aligned
      struct alignas(16) Vec { T v[VL]; };
      if (ra < rows) {
        const Vec t = *reinterpret_cast<const Vec*>(f + (size_t)ra * N + x);
#pragma unroll
        for (int e = 0; e < VL; ++e) a[e] = t.v[e];
      }
      if (ra + 1 < rows) {
        const Vec t = *reinterpret_cast<const Vec*>(f + (size_t)(ra + 1) * N + x);
#pragma unroll
        for (int e = 0; e < VL; ++e) b[e] = t.v[e];
      }
    }
#pragma unroll
    for (int e = 0; e < VL; ++e) fft_buf[(x + e) * kFftLines + w] = make_double2((double)a[e], (double)b[e]);
  }
  const double2* Z = fft_block(fft_buf, N, rad, tw);
  for (int idx = threadIdx.x; idx < H * kFftLines; idx += kFftThreads) {
    const int w = idx % kFftLines, k = idx / kFftLines;
    const int ra = l0 + 2 * w;
    const double2 u = Z[k * kFftLines + w], v = Z[(k ? N - k : 0) * kFftLines + w];
    if (ra < rows) out[(size_t)ra * H + k] = make_double2(u.x + v.x, u.y - v.y);
    if (ra + 1 < rows) out[(size_t)(ra + 1) * H + k] = make_double2(u.y + v.y, v.x - u.x);
  }
}

// In-place pass along one axis of complex data: line l starts at (l / inner) * outer + l % inner,
// its elements are `stride` apart.  inverse: the unnormalised inverse transform, by swapping real
// and imaginary parts on the way in and out.
__global__ void __launch_bounds__(kFftThreads) k_fft_axis(double2* __restrict__ data, int N, int lines, int inner,
                                                          long outer, long stride, int inverse, Radices rad,
                                                          const double2* __restrict__ tw) {
  extern __shared__ double2 fft_buf[];
  const int w = threadIdx.x % kFftLines;
  const int l = blockIdx.x * kFftLines + w;
  const bool on = l < lines;
  double2* line = data + (on ? (long)(l / inner) * outer + l % inner : 0);
  for (int x = threadIdx.x / kFftLines; x < N; x += kFftThreads / kFftLines) {
    double2 v = on ? line[x * stride] : make_double2(0.0, 0.0);
    fft_buf[x * kFftLines + w] = inverse ? make_double2(v.y, v.x) : v;
  }
  const double2* Z = fft_block(fft_buf, N, rad, tw);
  if (!on) return;
  for (int x = threadIdx.x / kFftLines; x < N; x += kFftThreads / kFftLines) {
    const double2 v = Z[x * kFftLines + w];
    line[x * stride] = inverse ? make_double2(v.y, v.x) : v;
  }
}

__device__ __forceinline__ int isqrt(int v) {  // floor(sqrt(v)), v >= 0
  int r = (int)sqrtf((float)v);
  while (r * r > v) --r;
  while ((r + 1) * (r + 1) <= v) ++r;
  return r;
}

// z pass of the half spectra and the shell sums in one: the transformed lines are not written, the
// squares of a line go from shared memory into the shells.  Shell b holds the modes with
// round(|k|) = b, b^2 - b < |k|^2 <= b^2 + b in whole numbers, on one line a contiguous range of
// |kz|.  Each thread owns the shells b = threadIdx.x, + kFftThreads, ..., so no sums collide (one
// FP64 atomic per mode into a few hundred addresses took 2.0 ms per component); a block keeps its
// sums over all its lines and writes them once (part[block][nb], added to when `more`).
__global__ void __launch_bounds__(kFftThreads) k_fft_shells(const double2* __restrict__ data, int N, int nb, int more,
                                                            Radices rad, const double2* __restrict__ tw,
                                                            double* __restrict__ part) {
  extern __shared__ double2 fft_buf[];
  const int H = N / 2 + 1, lines = N * H;
  const long stride = (long)N * H;
  constexpr int kOwn = (kFftMaxN + kFftThreads - 1) / kFftThreads;  // shells per thread: up to sqrt(3) N / 2 < kFftMaxN
  double sum[kOwn];
#pragma unroll
  for (int q = 0; q < kOwn; ++q) sum[q] = 0.0;
  const int kmax = N / 2;
  for (int l0 = blockIdx.x * kFftLines; l0 < lines; l0 += gridDim.x * kFftLines) {
    const int w = threadIdx.x % kFftLines;
    const int l = l0 + w;
    for (int z = threadIdx.x / kFftLines; z < N; z += kFftThreads / kFftLines)
      fft_buf[z * kFftLines + w] = l < lines ? data[l + z * stride] : make_double2(0.0, 0.0);
    double2* Z = fft_block(fft_buf, N, rad, tw);
    double* E = reinterpret_cast<double*>(Z == fft_buf ? fft_buf + (size_t)N * kFftLines : fft_buf);
    // energy of the modes +-kz of the line and, but for kx = 0 and the Nyquist plane, of its mirror
    const int kx = l % H;
    const double wt = (kx == 0 || 2 * kx == N) ? 1.0 : 2.0;
    for (int z = threadIdx.x / kFftLines; z <= kmax; z += kFftThreads / kFftLines) {
      const double2 a = Z[z * kFftLines + w];
      double e = a.x * a.x + a.y * a.y;
      if (z > 0 && 2 * z != N) {
        const double2 b = Z[(N - z) * kFftLines + w];
        e += b.x * b.x + b.y * b.y;
      }
      E[z * kFftLines + w] = wt * e;
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < kOwn; ++q) {
      const int b = threadIdx.x + q * kFftThreads;
      if (b < nb) {
        for (int v = 0; v < kFftLines && l0 + v < lines; ++v) {
          const int x = (l0 + v) % H, j = (l0 + v) / H, y = j <= N - j ? j : N - j;
          const int kp = x * x + y * y;
          const int top = b * b + b - kp, low = b > 0 ? b * b - b + 1 - kp : 0;
          if (top < 0 || low > kmax * kmax) continue;
          const int z1 = min(isqrt(top), kmax);
          for (int z = low > 0 ? isqrt(low - 1) + 1 : 0; z <= z1; ++z) sum[q] += E[z * kFftLines + v];
        }
      }
    }
    __syncthreads();
  }
#pragma unroll
  for (int q = 0; q < kOwn; ++q) {
    const int b = threadIdx.x + q * kFftThreads;
    if (b < nb) {
      double* d = &part[(size_t)blockIdx.x * nb + b];
      *d = more ? *d + sum[q] : sum[q];
    }
  }
}

// bins[b] = norm * sum over blocks of part[block][b], in a fixed order
__global__ void __launch_bounds__(kFftThreads) k_fft_bins(const double* __restrict__ part, int blocks, int nb,
                                                          double norm, double* __restrict__ bins) {
  __shared__ double red[kFftThreads];
  double s = 0.0;
  for (int q = threadIdx.x; q < blocks; q += kFftThreads) s += part[(size_t)q * nb + blockIdx.x];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int o = kFftThreads / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) bins[blockIdx.x] = norm * red[0];
}

// Radices of N = 2^a 3^b: the powers of two as 16 s, closed by what keeps the butterflies large
// (512 as 8 8 8: fewer operations than 16 16 2).
static Radices radices_of(int N) {
  Radices R;
  R.n = 0;
  int a = 0, v = N;
  while (v % 2 == 0) { v /= 2; ++a; }
  while (a >= 4 && a != 5 && a != 6 && a != 9) { R.r[R.n++] = 16; a -= 4; }
  while (a >= 3 && a != 4) { R.r[R.n++] = 8; a -= 3; }
  if (a == 2) R.r[R.n++] = 4;
  if (a == 1) R.r[R.n++] = 2;
  while (v % 3 == 0) { R.r[R.n++] = 3; v /= 3; }
  if (v != 1) R.n = -1;
  return R;
}

bool fft_supported(int N) { return N >= 2 && N <= kFftMaxN && radices_of(N).n >= 0; }

static int fft_smem(int N) { return 2 * N * kFftLines * (int)sizeof(double2); }

// the limit is one value per kernel and device, whoever launches it: always that of the longest line
template <typename K>
static cudaError_t fft_allow(K* kernel) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, fft_smem(kFftMaxN));
}

// complex 3D transform in place (tw: the N-th roots)
static int fft3d(double2* data, int N, int inverse, const double2* tw, cudaStream_t st) {
  const Radices R = radices_of(N);
  const int lines = N * N, sm = fft_smem(N), grid = (lines + kFftLines - 1) / kFftLines;
  const long NN = (long)N * N;
  if (fft_allow(k_fft_axis) != cudaSuccess) return FE_ERR_CUDA;
  k_fft_axis<<<grid, kFftThreads, sm, st>>>(data, N, lines, 1, N, 1, inverse, R, tw);
  k_fft_axis<<<grid, kFftThreads, sm, st>>>(data, N, lines, N, NN, N, inverse, R, tw);
  k_fft_axis<<<grid, kFftThreads, sm, st>>>(data, N, lines, lines, 0, NN, inverse, R, tw);
  return FE_OK;
}

// ---- spectral initial condition ---------------------------------------------------------
// SplitMix64 (Steele, Lea, Flood 2014): output m of the stream seeded with s is
// mix(s + (m+1) * 0x9E3779B97F4A7C15).
__device__ __forceinline__ uint64_t splitmix64_at(uint64_t seed, uint64_t m) {
  uint64_t z = seed + (m + 1ull) * 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}
__device__ __forceinline__ double u01(uint64_t z) { return (double)((z >> 11) + 1ull) * 0x1.0p-53; }

__global__ void k_ic_modes(double2* uh0, double2* uh1, double2* uh2, int N, uint64_t seed, double k0) {
  const long NNN = (long)N * N * N;
  for (long f = blockIdx.x * (long)blockDim.x + threadIdx.x; f < NNN; f += (long)gridDim.x * blockDim.x) {
    int i = (int)(f % N), j = (int)((f / N) % N), k = (int)(f / ((long)N * N));
    double kv[3] = {(double)(i < (N + 1) / 2 ? i : i - N), (double)(j < (N + 1) / 2 ? j : j - N),
                    (double)(k < (N + 1) / 2 ? k : k - N)};
    double2 g[3];
    for (int c = 0; c < 3; ++c) {
      uint64_t m0 = 2ull * (3ull * (uint64_t)f + (uint64_t)c);
      double a = u01(splitmix64_at(seed, m0)), b = u01(splitmix64_at(seed, m0 + 1ull));
      double r = sqrt(-2.0 * log(a));
      double sn, cs;
      sincospi(2.0 * b, &sn, &cs);
      g[c] = make_double2(r * cs * M_SQRT1_2, r * sn * M_SQRT1_2);
    }
    double k2 = kv[0] * kv[0] + kv[1] * kv[1] + kv[2] * kv[2];
    bool keep = k2 > 0.0;
    if (N % 2 == 0) {
      double nyq = -(double)(N / 2);
      keep = keep && kv[0] != nyq && kv[1] != nyq && kv[2] != nyq;
    }
    double2* out[3] = {uh0, uh1, uh2};
    if (!keep) {
      for (int c = 0; c < 3; ++c) out[c][f] = make_double2(0.0, 0.0);
      continue;
    }
    double kd_re = kv[0] * g[0].x + kv[1] * g[1].x + kv[2] * g[2].x;
    double kd_im = kv[0] * g[0].y + kv[1] * g[1].y + kv[2] * g[2].y;
    double km = sqrt(k2);
    double E = k2 * k2 * exp(-2.0 * (km / k0) * (km / k0));
    double amp = sqrt(E / (4.0 * M_PI * k2));
    for (int c = 0; c < 3; ++c) {
      double re = (g[c].x - kv[c] * kd_re / k2) * amp;
      double im = (g[c].y - kv[c] * kd_im / k2) * amp;
      out[c][f] = make_double2(re, im);
    }
  }
}

// partial sums of |Re u|^2 per block (fixed order), for the Mach rescaling
__global__ void k_sumsq_real(const double2* a, const double2* b, const double2* c, long n, double* part) {
  __shared__ double red[256];
  double s = 0.0;
  for (long q = blockIdx.x * (long)blockDim.x + threadIdx.x; q < n; q += (long)gridDim.x * blockDim.x)
    s += a[q].x * a[q].x + b[q].x * b[q].x + c[q].x * c[q].x;
  red[threadIdx.x] = s;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.x] = red[0];
}

template <typename T>
__global__ void k_ic_store(const double2* uh, T* u, long n, double scale) {
  for (long q = blockIdx.x * (long)blockDim.x + threadIdx.x; q < n; q += (long)gridDim.x * blockDim.x)
    u[q] = (T)(uh[q].x * scale);
}

template <typename T>
__global__ void k_fill(T* a, long n, double v) {
  for (long q = blockIdx.x * (long)blockDim.x + threadIdx.x; q < n; q += (long)gridDim.x * blockDim.x) a[q] = (T)v;
}

// ---- cell diagnostics --------------------------------------------------------------------
// Block sums of the cell diagnostics (part[block][NDIAG]): rho |u|^2, |u|^2, |w|^2, sum_d (Gc_d u_d)^2
// (both times (16 h)^2), rho, rho T (Fourier), rho Y_j ...  About 45 FP64 operations per cell, which
// bound it.
constexpr int NDIAG = 6 + MAXD;

template <typename T>
__global__ void __launch_bounds__(NTHR) k_diag(const BoxDev* boxes, int box, int s, double* part) {
  __shared__ double sh[3][kGradH][kGradW];
  const BoxDev& B = boxes[box];
  const int N = B.N, nd = B.nd;
  const bool fourier = B.closure == FE_FOURIER;
  const T* rho = F<T>(B, S(s, F_RHO));
  const T* Tf = F<T>(B, S(s, F_T));
  GradTile<T, double> t(F<T>(B, S(s, F_U0)), F<T>(B, S(s, F_U1)), F<T>(B, S(s, F_U2)), N, sh);
  const int k0 = blockIdx.z * kGradTz, kend = min(k0 + kGradTz, N);
  const bool active = t.i < N && t.j < N;
  double acc[NDIAG];
#pragma unroll
  for (int q = 0; q < NDIAG; ++q) acc[q] = 0.0;
  t.start(k0);
  for (int k = k0; k < kend; ++k) {
    t.next(k);
    if (!active) continue;
    double g[3][3];  // g[m][l] = 16 h Gc_m u_l
#pragma unroll
    for (int m = 0; m < 3; ++m)
#pragma unroll
      for (int l = 0; l < 3; ++l) {
        double v[4];
        t.line(l, m, v);
        g[m][l] = 10.0 * (v[2] - v[1]) - (v[3] - v[0]);
      }
    const double w0 = g[1][2] - g[2][1], w1 = g[2][0] - g[0][2], w2 = g[0][1] - g[1][0];
    const size_t c = t.plane(k) + t.own;
    const double r = widen(rho[c]);
    const double uu = t.z[0][2] * t.z[0][2] + t.z[1][2] * t.z[1][2] + t.z[2][2] * t.z[2][2];
    acc[0] += r * uu;
    acc[1] += uu;
    acc[2] += w0 * w0 + w1 * w1 + w2 * w2;
    acc[3] += g[0][0] * g[0][0] + g[1][1] * g[1][1] + g[2][2] * g[2][2];
    acc[4] += r;
    if (fourier) acc[5] += r * widen(Tf[c]);
#pragma unroll
    for (int q = 0; q < MAXD; ++q)
      if (q < nd) acc[6 + q] += r * widen(F<T>(B, S(s, F_Y0 + q))[c]);
  }
  __shared__ double red[NDIAG][NTHR / 32];
  const int lane = t.tid & 31, warp = t.tid >> 5;
#pragma unroll
  for (int q = 0; q < NDIAG; ++q) {
    if (q >= 6 + nd) break;
    double v = acc[q];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (lane == 0) red[q][warp] = v;
  }
  __syncthreads();
  if (t.tid < NDIAG) {
    double v = 0.0;
    if (t.tid < 6 + nd)
      for (int w = 0; w < NTHR / 32; ++w) v += red[t.tid][w];
    part[(size_t)(blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z)) * NDIAG + t.tid] = v;
  }
}

// Block sums of (rho - mean)^2, the mean from the sum of the first pass.
template <typename T>
__global__ void __launch_bounds__(NTHR) k_rho_var(const T* __restrict__ rho, long n, const double* __restrict__ sums,
                                                  double* __restrict__ part) {
  __shared__ double red[NTHR / 32];
  const double mean = sums[4] / (double)n;
  double v = 0.0;
  for (long q = blockIdx.x * (long)NTHR + threadIdx.x; q < n; q += (long)gridDim.x * NTHR) {
    const double d = (double)rho[q] - mean;
    v += d * d;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    v = 0.0;
    for (int w = 0; w < NTHR / 32; ++w) v += red[w];
    part[blockIdx.x] = v;
  }
}

// Q = (|Omega|^2 - |S|^2) / 2 = -(sum_i A_ii^2 / 2 + A_01 A_10 + A_02 A_20 + A_12 A_21), A the Gauss
// velocity gradient; in FP64 for either field type, rounded to it once: strain and rotation may cancel.  About 36
// FP64 operations per cell bound it, the planes staged as FP64 like k_diag's: 1.48 ms at 256^3 from FP32 fields
// (with every neighbour read and converted per use 4.0; in float pairs 0.30, with 70 times the error in the terms).
template <typename T>
__global__ void __launch_bounds__(NTHR) k_qcrit(const BoxDev* boxes, int box, int s, T* __restrict__ q) {
  __shared__ double sh[3][kGradH][kGradW];
  const BoxDev& B = boxes[box];
  const int N = B.N;
  GradTile<T, double> t(F<T>(B, S(s, F_U0)), F<T>(B, S(s, F_U1)), F<T>(B, S(s, F_U2)), N, sh);
  const double scale = B.ih * B.ih * (1.0 / 256.0);
  const int k0 = blockIdx.z * kGradTz, kend = min(k0 + kGradTz, N);
  t.start(k0);
  for (int k = k0; k < kend; ++k) {
    t.next(k);
    if (t.i >= N || t.j >= N) continue;
    double g[3][3];  // g[m][l] = 16 h Gc_m u_l
#pragma unroll
    for (int m = 0; m < 3; ++m)
#pragma unroll
      for (int l = 0; l < 3; ++l) {
        double v[4];
        t.line(l, m, v);
        g[m][l] = 10.0 * (v[2] - v[1]) - (v[3] - v[0]);
      }
    const double qv = -scale * (0.5 * (g[0][0] * g[0][0] + g[1][1] * g[1][1] + g[2][2] * g[2][2]) + g[0][1] * g[1][0] +
                                g[0][2] * g[2][0] + g[1][2] * g[2][1]);
    if constexpr (sizeof(T) == 4) q[t.plane(k) + t.own] = narrow(qv);
    else q[t.plane(k) + t.own] = qv;
  }
}

// ---- host-side drivers (called from fe_api.cu) -------------------------------------------
static int ew_grid(long n) {
  long g = (n + 255) / 256;
  return (int)(g < 152L * 16 ? g : 152L * 16);
}

template <typename T>
int ic_spectral(T* u0, T* u1, T* u2, int N, uint64_t seed, double k0, double mach, cudaStream_t st) {
  const long n = (long)N * N * N;
  const int nb = ew_grid(n);
  double2* buf = nullptr;  // three complex fields, the roots of unity, the block sums
  if (cudaMalloc(&buf, (3 * n + N) * sizeof(double2) + nb * sizeof(double)) != cudaSuccess) {
    cudaGetLastError();
    return FE_ERR_OOM;
  }
  double2* tw = buf + 3 * n;
  double* part = reinterpret_cast<double*>(tw + N);
  k_roots<<<1, 256, 0, st>>>(tw, N);
  k_ic_modes<<<ew_grid(n), 256, 0, st>>>(buf, buf + n, buf + 2 * n, N, seed, k0);
  int rc = FE_OK;
  for (int c = 0; c < 3 && rc == FE_OK; ++c) rc = fft3d(buf + c * n, N, 1, tw, st);
  k_sumsq_real<<<nb, 256, 0, st>>>(buf, buf + n, buf + 2 * n, n, part);
  std::vector<double> hp(nb);
  cudaMemcpyAsync(hp.data(), part, nb * sizeof(double), cudaMemcpyDeviceToHost, st);
  cudaStreamSynchronize(st);
  double ss = 0.0;
  for (int b = 0; b < nb; ++b) ss += hp[b];
  double ms = ss / (double)n;
  double scale = ms > 0.0 ? mach / sqrt(ms) : 0.0;
  T* out[3] = {u0, u1, u2};
  for (int c = 0; c < 3; ++c) k_ic_store<T><<<ew_grid(n), 256, 0, st>>>(buf + c * n, out[c], n, scale);
  cudaStreamSynchronize(st);
  cudaFree(buf);
  if (rc != FE_OK) return rc;
  return cudaGetLastError() == cudaSuccess ? FE_OK : FE_ERR_CUDA;
}

template <typename T>
void fill(T* a, long n, double v, cudaStream_t st) {
  k_fill<T><<<ew_grid(n), 256, 0, st>>>(a, n, v);
}

// Shells that a spectrum of an N^3 box can fill.
static int shells_of(int N) { return (int)floor(sqrt(3.0) * (N / 2) + 0.5) + 1; }

// Work memory of spectrum() (the context keeps it): a half spectrum, the roots of unity, the
// binning pass's block sums and the bins.
size_t spectrum_work_bytes(int N) {
  const size_t H = N / 2 + 1;
  return ((size_t)N * N * H + N) * sizeof(double2) + (size_t)(kFftGrid + 1) * shells_of(N) * sizeof(double);
}

// E(k) of the shells 0 .. nbins - 1 into host_bins (complete on return).
template <typename T>
int spectrum(const T* u0, const T* u1, const T* u2, int N, double* host_bins, int nbins, void* work, cudaStream_t st) {
  const Radices R = radices_of(N);
  const int H = N / 2 + 1, lines = N * H, sm = fft_smem(N);
  const int nb = nbins < shells_of(N) ? nbins : shells_of(N);
  double2* buf = static_cast<double2*>(work);
  double2* tw = buf + (size_t)N * lines;
  double* part = reinterpret_cast<double*>(tw + N);
  double* bins = part + (size_t)kFftGrid * nb;
  constexpr int VL = 16 / sizeof(T);
  const bool vec = N % VL == 0;
  if (fft_allow(k_fft_rows<T, VL>) != cudaSuccess || fft_allow(k_fft_rows<T, 1>) != cudaSuccess ||
      fft_allow(k_fft_axis) != cudaSuccess || fft_allow(k_fft_shells) != cudaSuccess)
    return FE_ERR_CUDA;
  const int pairs = (N * N + 1) / 2, gx = (pairs + kFftLines - 1) / kFftLines, gl = (lines + kFftLines - 1) / kFftLines;
  const int gs = gl < kFftGrid ? gl : kFftGrid;
  k_roots<<<1, 256, 0, st>>>(tw, N);
  const T* u[3] = {u0, u1, u2};
  for (int c = 0; c < 3; ++c) {
    if (vec) k_fft_rows<T, VL><<<gx, kFftThreads, sm, st>>>(u[c], buf, N, R, tw);
    else k_fft_rows<T, 1><<<gx, kFftThreads, sm, st>>>(u[c], buf, N, R, tw);
    k_fft_axis<<<gl, kFftThreads, sm, st>>>(buf, N, lines, H, (long)N * H, H, 0, R, tw);
    k_fft_shells<<<gs, kFftThreads, sm, st>>>(buf, N, nb, c > 0, R, tw, part);
  }
  // 1 / (2 N^6), and the 1/4 left out by the separation of the rows
  const double n3 = (double)N * N * N;
  k_fft_bins<<<nb, kFftThreads, 0, st>>>(part, gs, nb, 1.0 / (8.0 * n3 * n3), bins);
  for (int b = nb; b < nbins; ++b) host_bins[b] = 0.0;
  if (cudaMemcpyAsync(host_bins, bins, nb * sizeof(double), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
      cudaStreamSynchronize(st) != cudaSuccess)
    return FE_ERR_CUDA;
  return cudaGetLastError() == cudaSuccess ? FE_OK : FE_ERR_CUDA;
}

constexpr int kVarBlocks = 1024;

// Work memory of diag_sums(): the block sums of both passes and the totals.
size_t diag_work_bytes(int N) {
  const dim3 g = grad_grid(N);
  return ((size_t)g.x * g.y * g.z * NDIAG + kVarBlocks + NDIAG + 1) * sizeof(double);
}

// Sums of the cell diagnostics of one box (complete on return): rho |u|^2, |u|^2, |w|^2,
// sum_d (Gc_d u_d)^2, rho, (rho - mean)^2, energy density, rho Y_j ...
template <typename T>
int diag_sums(const Launch& L, const BoxDev& hb, int box, int s, double* out, void* work) {
  const dim3 g = grad_grid(hb.N);
  const int blocks = (int)(g.x * g.y * g.z);
  const long n = (long)hb.N * hb.N * hb.N;
  double* part = static_cast<double*>(work);
  double* vpart = part + (size_t)blocks * NDIAG;
  double* sums = vpart + kVarBlocks;
  double h[NDIAG + 1];
  k_diag<T><<<g, dim3(TX, TY), 0, L.st>>>(L.boxes, box, s, part);
  k_sum_parts<<<NDIAG, NTHR, 0, L.st>>>(part, blocks, NDIAG, sums);
  k_rho_var<T><<<kVarBlocks, NTHR, 0, L.st>>>((const T*)hb.f[S(s, F_RHO)], n, sums, vpart);
  k_sum_parts<<<1, NTHR, 0, L.st>>>(vpart, kVarBlocks, 1, sums + NDIAG);
  if (cudaMemcpyAsync(h, sums, sizeof(h), cudaMemcpyDeviceToHost, L.st) != cudaSuccess ||
      cudaStreamSynchronize(L.st) != cudaSuccess)
    return FE_ERR_CUDA;
  const double g2 = hb.ih * hb.ih / 256.0;
  out[0] = h[0];
  out[1] = h[1];
  out[2] = h[2] * g2;
  out[3] = h[3] * g2;
  out[4] = h[4];
  out[5] = h[NDIAG];
  out[6] = 0.5 * h[0] + (hb.closure == FE_FOURIER ? hb.cv * h[5] : 0.0);
  for (int j = 0; j < MAXD; ++j) out[7 + j] = h[6 + j];
  return cudaGetLastError() == cudaSuccess ? FE_OK : FE_ERR_CUDA;
}

template <typename T>
void qcrit(const Launch& L, const BoxDev& hb, int box, int s, T* q) {
  k_qcrit<T><<<grad_grid(hb.N), dim3(TX, TY), 0, L.st>>>(L.boxes, box, s, q);
}

#define INST(T)                                                                                   \
  template int ic_spectral<T>(T*, T*, T*, int, uint64_t, double, double, cudaStream_t);           \
  template void fill<T>(T*, long, double, cudaStream_t);                                          \
  template int spectrum<T>(const T*, const T*, const T*, int, double*, int, void*, cudaStream_t); \
  template int diag_sums<T>(const Launch&, const BoxDev&, int, int, double*, void*);              \
  template void qcrit<T>(const Launch&, const BoxDev&, int, int, T*);
INST(double)
INST(float)

}  // namespace fe
