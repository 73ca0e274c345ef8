// gradtile.cuh -- staged planes for the velocity-gradient kernels (diagnostics, Q, a-priori LES) and
// the fixed-order sum of their block partials.
#pragma once
#include "fe_internal.cuh"
#include "widen.cuh"

namespace fe {

template <typename S_, typename T>
__device__ __forceinline__ S_ stage_as(T v) {
  if constexpr (sizeof(S_) > sizeof(T)) return widen(v);
  else return v;
}

// The velocity gradient by columns: a block walks kGradTz planes of a 32 x 8 tile.  Each plane of
// the three components lies in shared memory with its halo of two cells in x and y (converted to S
// once per cell, not once per use), the z-neighbours of a cell stay in registers.  Reading all
// twelve neighbours of every component from global memory and converting each to FP64 took 3.6 ms
// (sums) and 4.0 ms (Q) at 256^3.
constexpr int kGradTz = 16;
constexpr int kGradW = TX + 4, kGradH = TY + 4;

template <typename T, typename S_>
struct GradTile {
  const T* u[3];
  S_ (*sh)[kGradH][kGradW];
  int N, i, j, own;      // own: flat x, y offset of the thread's column
  int off[2];            // flat x, y offsets of the staged cells threadIdx, + NTHR
  int tid;
  S_ z[3][5];            // z[l][2 + s]: component l at plane k + s
  __device__ __forceinline__ GradTile(const T* a, const T* b, const T* c, int N_, S_ (*sh_)[kGradH][kGradW])
      : sh(sh_), N(N_) {
    u[0] = a;
    u[1] = b;
    u[2] = c;
    tid = threadIdx.x + TX * threadIdx.y;
    i = blockIdx.x * TX + threadIdx.x;
    j = blockIdx.y * TY + threadIdx.y;
    own = i % N + N * (j % N);
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int t = min(tid + q * NTHR, kGradW * kGradH - 1);
      const int x = (int)(blockIdx.x * TX) - 2 + t % kGradW, y = (int)(blockIdx.y * TY) - 2 + t / kGradW;
      off[q] = (x + N) % N + N * ((y + N) % N);
    }
  }
  __device__ __forceinline__ size_t plane(int k) const { return (size_t)((k + 2 * N) % N) * N * N; }
  __device__ __forceinline__ void start(int k0) {
#pragma unroll
    for (int l = 0; l < 3; ++l)
#pragma unroll
      for (int s = 0; s < 4; ++s) z[l][s + 1] = stage_as<S_>(u[l][plane(k0 - 2 + s) + own]);
  }
  // plane k into shared memory, the queue one plane on
  __device__ __forceinline__ void next(int k) {
    const size_t p = plane(k), p2 = plane(k + 2);
    __syncthreads();
#pragma unroll
    for (int l = 0; l < 3; ++l) {
#pragma unroll
      for (int s = 0; s < 4; ++s) z[l][s] = z[l][s + 1];
      z[l][4] = stage_as<S_>(u[l][p2 + own]);
      S_* d = &sh[l][0][0];
      d[tid] = stage_as<S_>(u[l][p + off[0]]);
      if (tid + NTHR < kGradW * kGradH) d[tid + NTHR] = stage_as<S_>(u[l][p + off[1]]);
    }
    __syncthreads();
  }
  // the four neighbours of component l along m at distance -2, -1, 1, 2
  __device__ __forceinline__ void line(int l, int m, S_ (&v)[4]) const {
    const int x = threadIdx.x + 2, y = threadIdx.y + 2;
    if (m == 0) {
      v[0] = sh[l][y][x - 2], v[1] = sh[l][y][x - 1], v[2] = sh[l][y][x + 1], v[3] = sh[l][y][x + 2];
    } else if (m == 1) {
      v[0] = sh[l][y - 2][x], v[1] = sh[l][y - 1][x], v[2] = sh[l][y + 1][x], v[3] = sh[l][y + 2][x];
    } else {
      v[0] = z[l][0], v[1] = z[l][1], v[2] = z[l][3], v[3] = z[l][4];
    }
  }
};

inline dim3 grad_grid(int N) {
  return dim3((N + TX - 1) / TX, (N + TY - 1) / TY, (N + kGradTz - 1) / kGradTz);
}

// out[q] = sum over blocks of part[block * stride + q] in a fixed order, q = blockIdx.x
static __global__ void __launch_bounds__(NTHR) k_sum_parts(const double* __restrict__ part, int blocks, int stride,
                                                    double* __restrict__ out) {
  __shared__ double red[NTHR];
  double s = 0.0;
  for (int b = threadIdx.x; b < blocks; b += NTHR) s += part[(size_t)b * stride + blockIdx.x];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int o = NTHR / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) out[blockIdx.x] = red[0];
}

}  // namespace fe
