// unet.cu -- learned preconditioner for the pressure-correction solve.
//
// The paper (arXiv:1404.0959, Sec. 2 par. 1) solves a pressure-correction
// equation in every PISO corrector; this file adds a 3-level 3D-conv U-Net
// whose output serves as a search direction of flexible CG (the Jacobi
// direction remains the fallback).  Layers (3x3x3 kernels, periodic, ReLU
// after all but the last):
//   e1a 16->16, e1b 16->16 (N), d1 16->32 stride 2, e2 32->32 (N/2),
//   d2 32->64 stride 2, e3 64->64 (N/4), u2 [up2(e3), e2] 96->32 (N/2),
//   u1 [up2(u2), e1b] 48->16 (N), out 16->16 (N; channel 0 is the output).
// The first layer's input has 16 channels of which 2 carry data (the
// normalised residual and psi - 1), the last layer's 16 outputs of which 1 is
// used; the padding channels have zero inputs / zero loss and stay inert
// (16-wide channel groups keep every K step of the tensor-core GEMM full).
//
// Activations are channels-last BF16 (voxel-major, channels contiguous).
// Convolutions are implicit GEMMs on the tensor cores (BF16 x BF16 -> FP32):
// rows = voxels per tap, K = input channels, columns = output channels.
// Stride-1 layers on grids of a multiple of 128 run on tcgen05.mma
// (unet_tc.cu); other layers and the data gradients of stride 1 (transposed
// weights, negated taps) on k_conv_st, operands staged in shared memory
// (mma.sync m16n8k16); the data gradients of stride 2 and the deepest
// stride-2 layer on k_conv, which gathers its operands and serves any layer
// the others refuse.  The weight gradient (k_wgrad) is a GEMM over voxels
// from staged rows, one FP32 atomic per weight and chunk of voxels.
#include <cuda_bf16.h>

#include <cstring>
#include <vector>

#include "fe_internal.cuh"
#include "widen.cuh"

namespace fe {

typedef __nv_bfloat16 bf16;

// ---- gather modes -------------------------------------------------------------------
enum Gather {
  G_SAME = 0,    // input on the output grid, position p + t
  G_DOWN = 1,    // input on the grid twice as fine (stride-2 conv), position 2p + t
  G_UP = 2,      // input on the grid half as fine, read at (p + t) / 2 (nearest upsampling)
  G_SAME_T = 3,  // data gradient of a stride-1 conv: position p - t
  G_DOWN_T = 4,  // data gradient of a stride-2 conv: output grid fine, input coarse, (p - t)/2 if even
};

struct Src {
  const bf16* ptr;
  int C;      // channels of this source (multiple of 16)
  int mode;   // Gather
  int n;      // cells per side of the source grid
};

struct ConvArgs {
  Src s0, s1;          // channels [0, s0.C) then [s0.C, s0.C + s1.C)
  int Cin;             // s0.C + s1.C
  int Cout;            // multiple of 8
  int No;              // cells per side of the output grid
  const bf16* W;       // [27][Cout][Cin] (k = ci contiguous)
  const float* bias;   // [Cout] or null
  bf16* out;           // [No^3][Cout] or null
  float* out32;        // [No^3][Cout] or null (fp32 copy)
  int out32_ch;        // channels written to out32 (1: channel 0 only, else Cout)
  int relu;
  int accumulate;      // out32 += result
};

__device__ __forceinline__ int wrapn(int v, int n) {
  v %= n;
  return v < 0 ? v + n : v;
}

// Source voxel index of output position (x, y, z) for tap t, or -1 (zero).
__device__ __forceinline__ int gather_index(const Src& s, int x, int y, int z, int dx, int dy, int dz, int No) {
  int px, py, pz;
  switch (s.mode) {
    case G_SAME:
      px = wrapn(x + dx, s.n); py = wrapn(y + dy, s.n); pz = wrapn(z + dz, s.n);
      break;
    case G_DOWN:
      px = wrapn(2 * x + dx, s.n); py = wrapn(2 * y + dy, s.n); pz = wrapn(2 * z + dz, s.n);
      break;
    case G_UP:
      px = wrapn(x + dx, No) >> 1; py = wrapn(y + dy, No) >> 1; pz = wrapn(z + dz, No) >> 1;
      break;
    case G_SAME_T:
      px = wrapn(x - dx, s.n); py = wrapn(y - dy, s.n); pz = wrapn(z - dz, s.n);
      break;
    default: {  // G_DOWN_T: fine output grid No = 2 n
      int qx = wrapn(x - dx, No), qy = wrapn(y - dy, No), qz = wrapn(z - dz, No);
      if ((qx | qy | qz) & 1) return -1;
      px = qx >> 1; py = qy >> 1; pz = qz >> 1;
    }
  }
  return px + s.n * (py + s.n * pz);
}

__device__ __forceinline__ uint32_t ld_pair(const bf16* p) { return *reinterpret_cast<const uint32_t*>(p); }

__device__ __forceinline__ void mma_bf16(float (&c)[4], const uint32_t (&a)[4], const uint32_t (&b)[2]) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};\n"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

constexpr int CONV_WARPS = 4;
constexpr int CONV_MT = 2;  // 16-voxel m-tiles per warp

// Gather convolution: each warp computes 32 output voxels x all Cout (NT
// n-tiles of 8).  A fragments come straight from the channels-last source
// (two adjacent channels per 32-bit load), B fragments from the weights.
// Data gradients of stride 2 (G_DOWN_T) take the fine voxels one parity class after the other: a tap reaches only
// the voxels whose parity it matches, 27 of the 8 x 27 (class, tap) pairs, so a warp of one class skips the taps
// that contribute nothing (64^3 x 16 channels from 32^3 x 32: 138 us in voxel order, 109; 32^3 x 32 from 16^3 x 64: 100, 40).
template <int NT, bool DT>
__global__ void __launch_bounds__(CONV_WARPS * 32) k_conv(ConvArgs a) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int g = lane >> 2, tig = lane & 3;
  const long nvox = (long)a.No * a.No * a.No;
  const long vbase = ((long)blockIdx.x * CONV_WARPS + warp) * (16 * CONV_MT);
  if (vbase >= nvox) return;
  constexpr bool down_t = DT;  // No is even
  // the two rows (voxels) of each m-tile this thread feeds
  int rx[CONV_MT][2], ry[CONV_MT][2], rz[CONV_MT][2];
  bool rv[CONV_MT][2];
#pragma unroll
  for (int m = 0; m < CONV_MT; ++m)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      long v = vbase + 16 * m + g + 8 * h;
      rv[m][h] = v < nvox;
      if (!rv[m][h]) v = 0;
      const int n = down_t ? a.No / 2 : a.No;
      const long per = (long)n * n * n;
      const int cls = down_t ? (int)(v / per) : 0;
      v -= cls * per;
      rx[m][h] = (int)(v % n);
      ry[m][h] = (int)((v / n) % n);
      rz[m][h] = (int)(v / ((long)n * n));
      if (down_t) {
        rx[m][h] = 2 * rx[m][h] + (cls & 1);
        ry[m][h] = 2 * ry[m][h] + ((cls >> 1) & 1);
        rz[m][h] = 2 * rz[m][h] + (cls >> 2);
      }
    }
  float acc[CONV_MT][NT][4];
#pragma unroll
  for (int m = 0; m < CONV_MT; ++m)
#pragma unroll
    for (int n = 0; n < NT; ++n)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[m][n][e] = 0.f;

  for (int t = 0; t < 27; ++t) {
    const int dz = t / 9 - 1, dy = (t / 3) % 3 - 1, dx = t % 3 - 1;
#pragma unroll
    for (int sidx = 0; sidx < 2; ++sidx) {
      const Src& s = sidx == 0 ? a.s0 : a.s1;
      if (s.C == 0) continue;
      const int cofs = sidx == 0 ? 0 : a.s0.C;
      int idx[CONV_MT][2];
#pragma unroll
      for (int m = 0; m < CONV_MT; ++m)
#pragma unroll
        for (int h = 0; h < 2; ++h)
          idx[m][h] = rv[m][h] ? gather_index(s, rx[m][h], ry[m][h], rz[m][h], dx, dy, dz, a.No) : -1;
      if (down_t) {
        bool any = false;
#pragma unroll
        for (int m = 0; m < CONV_MT; ++m) any = any || idx[m][0] >= 0 || idx[m][1] >= 0;
        if (!__any_sync(0xffffffffu, any)) continue;
      }
      for (int c0 = 0; c0 < s.C; c0 += 16) {
        uint32_t af[CONV_MT][4];
#pragma unroll
        for (int m = 0; m < CONV_MT; ++m) {
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int id = idx[m][h];
            const bf16* p = s.ptr + (long)(id < 0 ? 0 : id) * s.C + c0 + 2 * tig;
            uint32_t lo = id < 0 ? 0u : ld_pair(p), hi = id < 0 ? 0u : ld_pair(p + 8);
            af[m][h] = lo;      // a0 (row g) / a1 (row g+8)
            af[m][2 + h] = hi;  // a2 / a3: columns + 8
          }
        }
        const bf16* wt = a.W + ((long)t * a.Cout) * a.Cin + cofs + c0 + 2 * tig;
#pragma unroll
        for (int n = 0; n < NT; ++n) {
          const bf16* wp = wt + (long)(8 * n + g) * a.Cin;
          uint32_t bfr[2] = {ld_pair(wp), ld_pair(wp + 8)};
#pragma unroll
          for (int m = 0; m < CONV_MT; ++m) mma_bf16(acc[m][n], af[m], bfr);
        }
      }
    }
  }
  // epilogue: bias, ReLU, store
#pragma unroll
  for (int m = 0; m < CONV_MT; ++m)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      if (!rv[m][h]) continue;
      const long v = rx[m][h] + (long)a.No * (ry[m][h] + (long)a.No * rz[m][h]);
#pragma unroll
      for (int n = 0; n < NT; ++n) {
        const int co = 8 * n + 2 * tig;
        float v0 = acc[m][n][2 * h], v1 = acc[m][n][2 * h + 1];
        if (a.bias) {
          v0 += a.bias[co];
          v1 += a.bias[co + 1];
        }
        if (a.relu) {
          v0 = fmaxf(v0, 0.f);
          v1 = fmaxf(v1, 0.f);
        }
        if (a.out) {
          __nv_bfloat162 pr = __floats2bfloat162_rn(v0, v1);
          *reinterpret_cast<__nv_bfloat162*>(a.out + v * a.Cout + co) = pr;
        }
        if (a.out32) {
          if (a.out32_ch == 1) {
            if (co == 0) a.out32[v] = a.accumulate ? a.out32[v] + v0 : v0;
          } else {
            float* o = a.out32 + v * a.Cout + co;
            if (a.accumulate) {
              o[0] += v0;
              o[1] += v1;
            } else {
              o[0] = v0;
              o[1] = v1;
            }
          }
        }
      }
    }
}

// ---- staged gather convolution ---------------------------------------------------------------
// k_conv with its operands staged: a CTA of 8 warps computes a tile of 16 x 4 x 4 (MT = 2), 16 x 8 x 4
// (4) or 32 x 8 x 4 (8) output voxels, MT 16-voxel m-tiles per warp.  The input voxels that the tile
// touches are copied into shared memory once, all channels, [channel octet][voxel][8 channels] (an
// upsampled source at its own resolution), the weights, [tap][channel octet][output channel][8 channels],
// all at once where they fit, else in groups of taps one group ahead (tap by tap their latency set the
// pace: 218 us for a 16-channel layer of 128^3 voxels, 174 us with all taps staged); both fragments come
// by ldmatrix, eight voxels or channels being 128 contiguous bytes.  k_conv gathers every fragment from
// global memory, the input 27 times and the weights once per 32 voxels (the half-grid layers of a 128^3
// network: 311 us each, 70 TFLOP/s, against 68 to 147 us).  The order of the matrix instructions of an
// output (tap, source, channel slice) is k_conv's, so the results are its bits.
// Modes: same grid, nearest upsampling, stride 2, and the data gradient of stride 1 (negated taps).
constexpr int kStThreads = 256;

__device__ __forceinline__ unsigned st_smem(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], unsigned addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr)
               : "memory");
}
__device__ __forceinline__ void st_cp16(unsigned dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}

// Staged box of one source: voxels per axis for an output tile of w voxels along the axis.
__host__ __device__ constexpr int st_extent(int mode, int w) {
  return mode == G_UP ? w / 2 + 2 : (mode == G_DOWN ? 2 * w + 1 : w + 2);
}
constexpr int st_tx(int mt) { return mt == 8 ? 32 : 16; }
constexpr int st_ty(int mt) { return mt == 2 ? 4 : 8; }
constexpr int kStTz = 4;

static int st_src_bytes(const Src& s, int mt) {
  return s.C * 2 * st_extent(s.mode, st_tx(mt)) * st_extent(s.mode, st_ty(mt)) * st_extent(s.mode, kStTz);
}
// with the weights in groups of `taps` (27: one buffer, else two)
static int st_bytes(const ConvArgs& a, int mt, int taps) {
  return st_src_bytes(a.s0, mt) + (a.s1.C ? st_src_bytes(a.s1, mt) : 0) +
         (taps == 27 ? 27 : 2 * taps) * a.Cin * a.Cout * 2;
}

template <int NT, int MT>
__global__ void __launch_bounds__(kStThreads, NT * MT <= 16 ? 2 : 1) k_conv_st(ConvArgs a, int taps) {
  constexpr int TXO = MT == 8 ? 32 : 16, TYO = MT == 2 ? 4 : 8, COUT = 8 * NT;
  extern __shared__ __align__(128) unsigned char st_sm[];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int g = lane >> 2, tig = lane & 3;
  const int ntx = (a.No + TXO - 1) / TXO, nty = (a.No + TYO - 1) / TYO;
  const int x0 = TXO * (blockIdx.x % ntx), y0 = TYO * ((blockIdx.x / ntx) % nty), z0 = kStTz * (blockIdx.x / (ntx * nty));
  // staged boxes: extents, voxels, shared base
  int ex[2], ey[2], nv[2];
  unsigned sb[2];
  unsigned base = st_smem(st_sm);
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const Src& s = q == 0 ? a.s0 : a.s1;
    ex[q] = st_extent(s.mode, TXO);
    ey[q] = st_extent(s.mode, TYO);
    nv[q] = s.C ? ex[q] * ey[q] * st_extent(s.mode, kStTz) : 0;
    sb[q] = base;
    base += nv[q] * s.C * 2;
  }
  const unsigned wbuf = base, wtap = (unsigned)(a.Cin * COUT * 2);
  auto stage_weights = [&](int group) {  // taps group * taps .. + taps - 1
    const int octs = a.Cin / 8, per = COUT * octs;
    const bf16* w = a.W + (long)group * taps * COUT * a.Cin;
    const unsigned dst = wbuf + (group & 1) * taps * wtap;
    for (int q = tid; q < taps * per; q += kStThreads) {
      const int c8 = q % octs, r = q / octs, co = r % COUT, t = r / COUT;
      st_cp16(dst + t * wtap + (unsigned)(c8 * COUT + co) * 16, w + (long)r * a.Cin + 8 * c8);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  auto wrapv = [](int v, int n) {
    v += v < 0 ? n : 0;
    while (v >= n) v -= n;
    return v;
  };
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const Src& s = q == 0 ? a.s0 : a.s1;
    if (s.C == 0) continue;
    const int lo = __ffs(s.C / 8) - 1;  // log2 of the channel octets (16, 32 or 64 channels)
    // first voxel of the box on the source's grid; a warp copies rows of voxels
    const int ox = s.mode == G_UP ? x0 / 2 - 1 : (s.mode == G_DOWN ? 2 * x0 - 1 : x0 - 1);
    const int oy = s.mode == G_UP ? y0 / 2 - 1 : (s.mode == G_DOWN ? 2 * y0 - 1 : y0 - 1);
    const int oz = s.mode == G_UP ? z0 / 2 - 1 : (s.mode == G_DOWN ? 2 * z0 - 1 : z0 - 1);
    const int rows = nv[q] / ex[q];
    for (int r = warp; r < rows; r += kStThreads / 32) {
      const int lz = r / ey[q], ly = r - lz * ey[q];
      const bf16* src = s.ptr + (long)s.n * (wrapv(oy + ly, s.n) + (long)s.n * wrapv(oz + lz, s.n)) * s.C;
      for (int c = lane; c < ex[q] << lo; c += 32) {
        const int c8 = c & ((1 << lo) - 1), lx = c >> lo;
        st_cp16(sb[q] + (unsigned)(c8 * nv[q] + r * ex[q] + lx) * 16, src + wrapv(ox + lx, s.n) * s.C + 8 * c8);
      }
    }
  }
  stage_weights(0);  // one group with the input
  float acc[MT][NT][4];
#pragma unroll
  for (int m = 0; m < MT; ++m)
#pragma unroll
    for (int n = 0; n < NT; ++n)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[m][n][e] = 0.f;
  // this lane's row of an m-tile and channel half for ldmatrix; the warp's m-tiles: one z, MT (x, y) rows
  const int row = (lane & 7) + (lane & 8), half = lane >> 4;
  const int zt = warp >> 1, yt = (warp & 1) * (TYO / 2);
  const int sgn = a.s0.mode == G_SAME_T ? -1 : 1;
  const int brow = (lane & 7) + ((lane >> 4) << 3), bhalf = (lane >> 3) & 1;
  for (int t = 0; t < 27; ++t) {
    const int group = t / taps;
    if (t == group * taps) {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
      __syncthreads();
      if (t + taps < 27) stage_weights(group + 1);
    }
    const int dz = sgn * (t / 9 - 1), dy = sgn * ((t / 3) % 3 - 1), dx = sgn * (t % 3 - 1);
    const unsigned wb = wbuf + ((group & 1) * taps + t - group * taps) * wtap + (unsigned)(bhalf * COUT + brow) * 16;
    int oct = 0;  // channel octet among both sources
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const Src& s = q == 0 ? a.s0 : a.s1;
      if (s.C == 0) continue;
      unsigned va[MT];  // shared address of this lane's voxel, per m-tile
#pragma unroll
      for (int m = 0; m < MT; ++m) {
        const int xb = (MT == 8 ? 16 * (m & 1) : 0) + row, yb = yt + (MT == 8 ? m >> 1 : m);
        int lx, ly, lz;
        if (s.mode == G_UP) {
          lx = (xb + 2 + dx) >> 1;
          ly = (yb + 2 + dy) >> 1;
          lz = (zt + 2 + dz) >> 1;
        } else if (s.mode == G_DOWN) {
          lx = 2 * xb + 1 + dx;
          ly = 2 * yb + 1 + dy;
          lz = 2 * zt + 1 + dz;
        } else {
          lx = xb + 1 + dx;
          ly = yb + 1 + dy;
          lz = zt + 1 + dz;
        }
        va[m] = sb[q] + (unsigned)(half * nv[q] + (lz * ey[q] + ly) * ex[q] + lx) * 16;
      }
      for (int c = 0; c < s.C / 16; ++c, oct += 2) {
        uint32_t af[MT][4];
#pragma unroll
        for (int m = 0; m < MT; ++m) ldsm4(af[m], va[m] + (unsigned)(2 * c * nv[q]) * 16);
#pragma unroll
        for (int n = 0; n < NT; n += 2) {
          uint32_t bf[4];
          ldsm4(bf, wb + (unsigned)(oct * COUT + 8 * n) * 16);
          const uint32_t b0[2] = {bf[0], bf[1]}, b1[2] = {bf[2], bf[3]};
#pragma unroll
          for (int m = 0; m < MT; ++m) {
            mma_bf16(acc[m][n], af[m], b0);
            mma_bf16(acc[m][n + 1], af[m], b1);
          }
        }
      }
    }
  }
#pragma unroll
  for (int m = 0; m < MT; ++m) {
    const int yo = y0 + yt + (MT == 8 ? m >> 1 : m), zo = z0 + zt;
    if (yo >= a.No || zo >= a.No) continue;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int xo = x0 + (MT == 8 ? 16 * (m & 1) : 0) + g + 8 * h;
      if (xo >= a.No) continue;
      const long v = xo + (long)a.No * (yo + (long)a.No * zo);
#pragma unroll
      for (int n = 0; n < NT; ++n) {
        const int co = 8 * n + 2 * tig;
        float v0 = acc[m][n][2 * h], v1 = acc[m][n][2 * h + 1];
        if (a.bias) {
          v0 += a.bias[co];
          v1 += a.bias[co + 1];
        }
        if (a.relu) {
          v0 = fmaxf(v0, 0.f);
          v1 = fmaxf(v1, 0.f);
        }
        if (a.out) *reinterpret_cast<__nv_bfloat162*>(a.out + v * COUT + co) = __floats2bfloat162_rn(v0, v1);
        if (a.out32) {
          if (a.out32_ch == 1) {
            if (co == 0) a.out32[v] = v0;
          } else {
            *reinterpret_cast<float2*>(a.out32 + v * COUT + co) = make_float2(v0, v1);
          }
        }
      }
    }
  }
}

// dpre = bf16(d * (act > 0))  (act null: no mask), optional second addend
__global__ void k_mask(const float* d, const float* d2, const bf16* act, long n, bf16* out) {
  for (long q = blockIdx.x * (long)blockDim.x + threadIdx.x; q < n; q += (long)gridDim.x * blockDim.x) {
    float v = d[q] + (d2 ? d2[q] : 0.f);
    if (act && !(__bfloat162float(act[q]) > 0.f)) v = 0.f;
    out[q] = __float2bfloat16(v);
  }
}

// sum over the 8 fine children of channels [0, Cc) of a fine [n^3][Cf] fp32 tensor -> coarse [(n/2)^3][Cc]
__global__ void k_up2_back(const float* fine, int nf, int Cf, int Cc, float* coarse) {
  const int nc = nf / 2;
  const long total = (long)nc * nc * nc * Cc;
  for (long q = blockIdx.x * (long)blockDim.x + threadIdx.x; q < total; q += (long)gridDim.x * blockDim.x) {
    const int c = (int)(q % Cc);
    const long u = q / Cc;
    const int x = (int)(u % nc), y = (int)((u / nc) % nc), z = (int)(u / ((long)nc * nc));
    float s = 0.f;
    for (int oz = 0; oz < 2; ++oz)
      for (int oy = 0; oy < 2; ++oy)
        for (int ox = 0; ox < 2; ++ox) {
          const long v = (2 * x + ox) + (long)nf * ((2 * y + oy) + (long)nf * (2 * z + oz));
          s += fine[v * Cf + c];
        }
    coarse[q] = s;
  }
}

// copy channels [c0, c0 + C) of a [n][Cf] fp32 tensor into a dense [n][C]
__global__ void k_slice(const float* src, long n, int Cf, int c0, int C, float* dst) {
  for (long q = blockIdx.x * (long)blockDim.x + threadIdx.x; q < n * C; q += (long)gridDim.x * blockDim.x)
    dst[q] = src[(q / C) * Cf + c0 + q % C];
}

// Network input of the residual-form preconditioner, for a residual r of the
// operator M = diag(psi/dt) - dt/2 D(G2 .) with Jacobi inverse dinv = 1/d,
// d = psi/dt + 3 dt/h^2: channel 0 = (r dinv) / (rms(r) d0) with d0 the
// Jacobi inverse at psi = 1, channel 1 = (3 dt/h^2) dinv (the Laplacian's
// share of the diagonal, which carries dt and psi), channels 2..15 = 0.  The
// direction is z = r dinv + rms(r) d0 y for the network output y.
// 16-channel input voxel: (c0, c1, 0, ..., 0) in two 16-byte stores
__device__ __forceinline__ void pack_voxel(bf16* o, float c0, float c1) {
  __nv_bfloat162 p = __floats2bfloat162_rn(c0, c1);
  uint4 a;
  a.x = *reinterpret_cast<uint32_t*>(&p);
  a.y = a.z = a.w = 0u;
  reinterpret_cast<uint4*>(o)[0] = a;
  reinterpret_cast<uint4*>(o)[1] = make_uint4(0u, 0u, 0u, 0u);
}

// a = 1 / (rms(r) d0), w = 3 dt / h^2
template <typename T>
__global__ void k_pack_input(const T* r, const T* dinv, long n, double a, double w, bf16* in16) {
  for (long q = blockIdx.x * (long)blockDim.x + threadIdx.x; q < n; q += (long)gridDim.x * blockDim.x) {
    const double dq = widen(dinv[q]);
    pack_voxel(in16 + q * 16, narrow(widen(r[q]) * dq * a), narrow(dq * w));
  }
}

// z = r dinv + scale y (the residual-form direction, FP32)
template <typename T>
__global__ void k_direction(const T* r, const T* dinv, const float* y, double scale, long n, float* z) {
  for (long q = blockIdx.x * (long)blockDim.x + threadIdx.x; q < n; q += (long)gridDim.x * blockDim.x)
    z[q] = narrow(widen(r[q]) * widen(dinv[q]) + scale * widen(y[q]));
}

// training target t = (e - r dinv) * inv_scale into tgt; block partial sums of t^2
template <typename T>
__global__ void k_target(const T* r, const T* e, const T* dinv, long n, double inv_scale, float* tgt, double* part) {
  __shared__ double red[256];
  double s = 0.0;
  for (long q = blockIdx.x * (long)blockDim.x + threadIdx.x; q < n; q += (long)gridDim.x * blockDim.x) {
    const float t = (float)(((double)e[q] - (double)r[q] * (double)dinv[q]) * inv_scale);
    tgt[q] = t;
    s += (double)t * (double)t;
  }
  red[threadIdx.x] = s;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.x] = red[0];
}

// Adam (Kingma and Ba 2015) on the FP32 master weights; refreshes the BF16
// forward copy [27][Cout][Cin] and the transposed copy [27][Cin][Cout].
__global__ void k_adam(float* w, const float* g, float* m, float* v, long n, float lr, float b1, float b2, float eps,
                       float c1, float c2, int taps, int Cout, int Cin, bf16* wf, bf16* wt, int mask_ci, int mask_co) {
  for (long q = blockIdx.x * (long)blockDim.x + threadIdx.x; q < n; q += (long)gridDim.x * blockDim.x) {
    float gq = g[q];
    float mq = b1 * m[q] + (1.f - b1) * gq;
    float vq = b2 * v[q] + (1.f - b2) * gq * gq;
    m[q] = mq;
    v[q] = vq;
    float wq = w[q] - lr * (mq / c1) / (sqrtf(vq / c2) + eps);
    if (taps > 0) {
      const int ci = (int)(q % Cin);
      const int co = (int)((q / Cin) % Cout);
      const int t = (int)(q / ((long)Cin * Cout));
      if (ci >= mask_ci || co >= mask_co) wq = 0.f;  // padding channels stay inert
      wf[q] = __float2bfloat16(wq);
      wt[((long)t * Cin + ci) * Cout + co] = __float2bfloat16(wq);
    }
    w[q] = wq;
  }
}

__global__ void k_cast_weights(const float* w, long n, int Cout, int Cin, bf16* wf, bf16* wt) {
  for (long q = blockIdx.x * (long)blockDim.x + threadIdx.x; q < n; q += (long)gridDim.x * blockDim.x) {
    const int ci = (int)(q % Cin);
    const int co = (int)((q / Cin) % Cout);
    const int t = (int)(q / ((long)Cin * Cout));
    wf[q] = __float2bfloat16(w[q]);
    wt[((long)t * Cin + ci) * Cout + co] = __float2bfloat16(w[q]);
  }
}

// loss = ||y - t||^2 / ||t||^2 partial sums (y: channel 0 of out32) and dy in the 16-channel layout
__global__ void k_loss_grad(const float* y, const float* tgt, long n, double inv_tt, float* dy8, double* part) {
  __shared__ double red[256];
  double s = 0.0;
  for (long q = blockIdx.x * (long)blockDim.x + threadIdx.x; q < n; q += (long)gridDim.x * blockDim.x) {
    const double d = (double)y[q] - (double)tgt[q];
    s += d * d;
    float* o = dy8 + q * 16;
    o[0] = (float)(2.0 * d * inv_tt);
    for (int c = 1; c < 16; ++c) o[c] = 0.f;
  }
  red[threadIdx.x] = s;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.x] = red[0];
}

// ---- host side ----------------------------------------------------------------------------
struct Layer {
  const char* name;
  int cin, cout, cin_real, cout_real, level_out, stride;
  float* w;  // fp32 master [27][cout][cin]
  float* b;
  float* gw;
  float* gb;
  float* mw;
  float* vw;
  float* mb;
  float* vb;
  bf16* wf;
  bf16* wt;
};

static const int kNL = 9;
// name, cin, cout, cin_real, cout_real, level of the output, stride
static const int kDims[kNL][6] = {{16, 16, 2, 16, 0, 1},  {16, 16, 16, 16, 0, 1}, {16, 32, 16, 32, 1, 2},
                                  {32, 32, 32, 32, 1, 1}, {32, 64, 32, 64, 2, 2}, {64, 64, 64, 64, 2, 1},
                                  {96, 32, 96, 32, 1, 1}, {48, 16, 48, 16, 0, 1}, {16, 16, 16, 1, 0, 1}};
static const char* kNames[kNL] = {"e1a", "e1b", "d1", "e2", "d2", "e3", "u2", "u1", "out"};

long unet_param_count() {
  long n = 0;
  for (int l = 0; l < kNL; ++l) n += 27L * kDims[l][2] * kDims[l][3] + kDims[l][3];
  return n;
}

struct UNet {
  int N = 0;  // finest grid
  Layer L[kNL];
  void* wslab = nullptr;
  // activations (bf16 channels-last)
  bf16 *in16 = nullptr, *e1a = nullptr, *e1b = nullptr, *d1 = nullptr, *e2 = nullptr, *d2 = nullptr,
       *e3 = nullptr, *u2 = nullptr, *u1 = nullptr;
  float* out32 = nullptr;  // [N^3] channel 0
  float* xfer = nullptr;   // parameters or gradients in the host's order, on their way out
  // training buffers
  float *g0 = nullptr, *g1 = nullptr, *g2 = nullptr, *gsk0 = nullptr, *gsk1 = nullptr, *dy8 = nullptr;
  bf16* dpre = nullptr;
  double* part = nullptr;  // block sums of a reduction, then `err`: one copy brings both
  int adam_step = 0;
  std::vector<void*> allocs;
  bool trained = false;
  int use_tc = 1;      // stride-1 layers on the fifth-generation tensor cores where they fit
  int* err = nullptr;  // device flag: a tensor-core convolution gave up a bounded wait
  int* herr = nullptr;  // pinned copy of it
  int nsm = 152;
};

struct TcConvArgs {
  const bf16* s0;
  const bf16* s1;
  int c0, c1, m0, m1;
  int No;
  const bf16* W;
  const float* bias;
  bf16* out;
  float* out32;
  int relu;
  int* err;
};
int conv_tc(const TcConvArgs& a, int Cout, int nsm, cudaStream_t st);

static long cube(long n) { return n * n * n; }

static int ew(long n) {
  long g = (n + 255) / 256;
  return (int)(g < 152L * 8 ? g : 152L * 8);
}

static int unet_alloc(UNet& U, int N, bool training) {
  U.N = N;
  const long n0 = cube(N), n1 = cube(N / 2), n2 = cube(N / 4);
  auto A = [&](size_t bytes) -> void* {
    void* p = nullptr;
    if (cudaMalloc(&p, bytes) != cudaSuccess) return nullptr;
    U.allocs.push_back(p);
    return p;
  };
  U.in16 = (bf16*)A(n0 * 16 * 2);
  U.e1a = (bf16*)A(n0 * 16 * 2);
  U.e1b = (bf16*)A(n0 * 16 * 2);
  U.d1 = (bf16*)A(n1 * 32 * 2);
  U.e2 = (bf16*)A(n1 * 32 * 2);
  U.d2 = (bf16*)A(n2 * 64 * 2);
  U.e3 = (bf16*)A(n2 * 64 * 2);
  U.u2 = (bf16*)A(n1 * 32 * 2);
  U.u1 = (bf16*)A(n0 * 16 * 2);
  U.out32 = (float*)A(n0 * 4);
  U.part = (double*)A((ew(n0) + 1) * sizeof(double));
  if (U.part) {
    cudaMemset(U.part, 0, (ew(n0) + 1) * sizeof(double));
    U.err = (int*)(U.part + ew(n0));
  }
  {
    int dev = 0, nsm = 0;
    if (cudaGetDevice(&dev) == cudaSuccess &&
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && nsm > 0)
      U.nsm = nsm;
  }
  U.xfer = (float*)A(unet_param_count() * 4);
  if (cudaMallocHost(&U.herr, sizeof(int)) != cudaSuccess) return FE_ERR_OOM;
  if (!U.xfer || !U.in16 || !U.e1a || !U.e1b || !U.d1 || !U.e2 || !U.d2 || !U.e3 || !U.u2 || !U.u1 || !U.out32 || !U.err)
    return FE_ERR_OOM;
  size_t wtotal = 0;
  for (int l = 0; l < kNL; ++l) {
    const long nw = 27L * kDims[l][0] * kDims[l][1];
    wtotal += (nw * 4 * 4 + kDims[l][1] * 4 * 4 + nw * 2 * 2 + 10 * 256);  // 10 slices, each 256-aligned
  }
  char* ws = (char*)A(wtotal);
  if (!ws) return FE_ERR_OOM;
  cudaMemset(ws, 0, wtotal);
  for (int l = 0; l < kNL; ++l) {
    Layer& y = U.L[l];
    y.name = kNames[l];
    y.cin = kDims[l][0];
    y.cout = kDims[l][1];
    y.cin_real = kDims[l][2];
    y.cout_real = kDims[l][3];
    y.level_out = kDims[l][4];
    y.stride = kDims[l][5];
    const long nw = 27L * y.cin * y.cout;
    auto take = [&](size_t bytes) {
      void* p = ws;
      ws += (bytes + 255) & ~(size_t)255;
      return p;
    };
    y.w = (float*)take(nw * 4);
    y.gw = (float*)take(nw * 4);
    y.mw = (float*)take(nw * 4);
    y.vw = (float*)take(nw * 4);
    y.b = (float*)take(y.cout * 4);
    y.gb = (float*)take(y.cout * 4);
    y.mb = (float*)take(y.cout * 4);
    y.vb = (float*)take(y.cout * 4);
    y.wf = (bf16*)take(nw * 2);
    y.wt = (bf16*)take(nw * 2);
  }
  if (training) {
    U.g0 = (float*)A(n0 * 48 * 4);
    U.g1 = (float*)A(n1 * 96 * 4);
    U.g2 = (float*)A(n2 * 64 * 4);
    U.gsk0 = (float*)A(n0 * 16 * 4);
    U.gsk1 = (float*)A(n1 * 32 * 4);
    U.dy8 = (float*)A(n0 * 16 * 4);
    U.dpre = (bf16*)A(n0 * 64 * 2 > n1 * 96 * 2 ? n0 * 64 * 2 : n1 * 96 * 2);
    if (!U.g0 || !U.g1 || !U.g2 || !U.gsk0 || !U.gsk1 || !U.dy8 || !U.dpre) return FE_ERR_OOM;
  }
  return FE_OK;
}

static void unet_free(UNet& U) {
  for (void* p : U.allocs) cudaFree(p);
  U.allocs.clear();
  if (U.herr) cudaFreeHost(U.herr);
  U.herr = nullptr;
}

// ---- weight and bias gradients ---------------------------------------------------------------
// dW[t][co][ci] += sum_v dpre(v)[co] in(v, t)[ci].
// A CTA has a chunk of consecutive voxels (64 per layer), the three taps of one (dz, dy), one slice of 16 input
// channels and up to 32 output channels.  It walks over the chunk in batches of 256 voxels (128 at stride 2): the
// input row of every row that a batch touches and the batch's dpre are copied into shared memory, [channel octet]
// [voxel][8 channels], the next batch's behind the current one's products, and both fragments come by ldmatrix
// with transposition, sixteen consecutive voxels being one K step; each lane finds its voxel's row, so a step may
// straddle rows and planes.  A warp holds 3 taps x 16 x 16 sums in registers and reads its dpre fragment once for
// the three (nine taps of one dz per warp: a third of the dpre copies, but 192 CTAs of four warps for a 16-channel
// layer leave the chip idle: 637 us a 64^3 step; the same with the three dy in twelve warps: 629).  The order of
// the sums is fixed: four chains of K steps per chunk (step j to chain j mod 4), added in order, then one atomic
// per weight and chunk -- a gradient near zero decides the sign of a first Adam step, so sums must not move by more
// than the order of the 64 atomics moves them.
// With one tap per CTA and every fragment element gathered from global memory (2 bytes a load) the input was
// read 27 times: 4.1 ms of the 6.3 ms of a 64^3 training step, 0.50 ms now.
struct WgradArgs {
  Src s0, s1;
  int Cin, Cout, No;
  const bf16* dpre;  // [No^3][Cout]
  float* dW;         // [27][Cout][Cin]
  long chunk;        // voxels per chunk, a multiple of 16
};

__device__ __forceinline__ void ldsm4t(uint32_t (&r)[4], unsigned addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr)
               : "memory");
}
// batch length, staged row length and most rows of a batch on an output grid of side N
__host__ __device__ constexpr int wg_run(int mode) { return mode == G_DOWN ? 128 : 256; }
__host__ __device__ constexpr int wg_pitch(int mode, int N) {
  const int w = N < wg_run(mode) ? N : wg_run(mode);
  return mode == G_UP ? w / 2 + 2 : (mode == G_DOWN ? 2 * w + 1 : w + 2);
}
__host__ __device__ constexpr int wg_rows(int mode, int N) { return (N + wg_run(mode) - 2) / N + 1; }
// one buffer: two channel octets of the input rows, the batch's dpre
static int wg_stage_bytes(int mode, int N, int cout) {
  return wg_rows(mode, N) * wg_pitch(mode, N) * 32 + wg_run(mode) * cout * 2;
}

__global__ void __launch_bounds__(256) k_wgrad(WgradArgs a) {
  extern __shared__ __align__(128) unsigned char st_sm[];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarp = blockDim.x >> 5;
  const int g = lane >> 2, tig = lane & 3;
  const int slices = a.Cin / 16, slice = blockIdx.z % slices, co0 = 32 * (blockIdx.z / slices);
  const bool first = 16 * slice < a.s0.C;
  const Src s = first ? a.s0 : a.s1;
  const bf16* in = s.ptr + 16 * slice - (first ? 0 : a.s0.C);
  const int mode = s.mode, No = a.No, dz = (int)blockIdx.y / 3 - 1, dy = (int)blockIdx.y % 3 - 1;
  const int V = wg_run(mode), P = wg_pitch(mode, No), np = wg_rows(mode, No) * P;
  const int ncb = nwarp / 4, lco = ncb;  // blocks of 16 output channels; log2 of their octets (1 -> 2, 2 -> 4)
  const unsigned base = st_smem(st_sm), stage = (unsigned)(np * 32 + V * ncb * 32);
  const long nvox = (long)No * No * No, vc = (long)blockIdx.x * a.chunk;
  const long v1 = vc + a.chunk < nvox ? vc + a.chunk : nvox;
  const int chain = warp & 3, cob = warp >> 2;
  auto wrapv = [](int v, int n) {
    v += v < 0 ? n : 0;
    while (v >= n) v -= n;
    return v;
  };
  // first source voxel of a staged row, relative to the row: of the batch's first row (which begins at x0) or a later one
  auto row_origin = [&](bool head, int x0) {
    return !head ? -1 : (mode == G_UP ? (x0 - 1) >> 1 : (mode == G_DOWN ? 2 * x0 - 1 : x0 - 1));
  };
  auto along = [&](int v, int d) {  // source coordinate, not wrapped
    return mode == G_UP ? (v + d) >> 1 : (mode == G_DOWN ? 2 * v + d : v + d);
  };
  auto across = [&](int v, int d) {
    return mode == G_UP ? wrapn(v + d, No) >> 1 : wrapn(mode == G_DOWN ? 2 * v + d : v + d, s.n);
  };
  auto copy = [&](long v0, unsigned dst) {
    const long vend = v0 + V < v1 ? v0 + V : v1;
    const int R0 = (int)(v0 / No), x0 = (int)(v0 - (long)R0 * No), nr = (int)((vend - 1) / No) - R0 + 1;
    for (int lr = warp; lr < nr; lr += nwarp) {
      const int R = R0 + lr, z = R / No, y = R - z * No;
      const bf16* src = in + (long)s.n * (across(y, dy) + (long)s.n * across(z, dz)) * s.C;
      const int xo = row_origin(lr == 0, x0);
      for (int c = lane; c < 2 * P; c += 32) {
        const int c8 = c & 1, lx = c >> 1;
        st_cp16(dst + (unsigned)(c8 * np + lr * P + lx) * 16, src + wrapv(xo + lx, s.n) * s.C + 8 * c8);
      }
    }
    const unsigned dd = dst + np * 32;
    for (int q = tid; q < V << lco; q += blockDim.x) {
      const int c8 = q & ((1 << lco) - 1), v = q >> lco;
      const unsigned d = dd + (unsigned)(c8 * V + v) * 16;
      if (v0 + v < v1)
        st_cp16(d, a.dpre + (v0 + v) * a.Cout + co0 + 8 * c8);
      else
        asm volatile("st.shared.v4.u32 [%0], {%1, %1, %1, %1};" ::"r"(d), "r"(0) : "memory");
    }
  };
  float acc[3][2][4];
#pragma unroll
  for (int t = 0; t < 3; ++t)
#pragma unroll
    for (int n = 0; n < 2; ++n)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[t][n][e] = 0.f;
  // ldmatrix rows of this lane: voxel and octet of the dpre fragment and of the input fragment
  const int ak = (lane & 7) + ((lane >> 4) << 3), aoct = 2 * cob + ((lane >> 3) & 1);
  const int bk = lane & 15, boct = lane >> 4;
  int cur = 0;
  copy(vc, base);
  asm volatile("cp.async.commit_group;" ::: "memory");
  for (long v0 = vc; v0 < v1; v0 += V, cur ^= 1) {
    if (v0 + V < v1) copy(v0 + V, base + (cur ^ 1) * stage);
    asm volatile("cp.async.commit_group;" ::: "memory");
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    __syncthreads();
    const int R0 = (int)(v0 / No), x0 = (int)(v0 - (long)R0 * No), left = (int)(v1 - v0 < V ? v1 - v0 : V);
    const unsigned ib = base + cur * stage + (unsigned)(boct * np) * 16;
    const unsigned db = base + cur * stage + (unsigned)(np * 32) + (unsigned)(aoct * V + ak) * 16;
    for (int j = 16 * chain; j < left; j += 64) {
      uint32_t af[4];
      ldsm4t(af, db + (unsigned)j * 16);
      // the lane's voxel (past the end: dpre is 0 there, any staged voxel serves)
      const int l = x0 + (j + bk < left ? j + bk : left - 1), lr = l / No, x = l - lr * No;
      const int xo = row_origin(lr == 0, x0);
      const unsigned row = ib + (unsigned)(lr * P) * 16;
#pragma unroll
      for (int tx = 0; tx < 3; ++tx) {
        uint32_t bf[4];
        ldsm4t(bf, row + (unsigned)(along(x, tx - 1) - xo) * 16);
        const uint32_t b0[2] = {bf[0], bf[1]}, b1[2] = {bf[2], bf[3]};
        mma_bf16(acc[tx][0], af, b0);
        mma_bf16(acc[tx][1], af, b1);
      }
    }
    __syncthreads();
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  float* red = reinterpret_cast<float*>(st_sm);  // [3][16 ncb][16]
  for (int q = 0; q < 4; ++q) {
    __syncthreads();
    if (chain != q) continue;
#pragma unroll
    for (int t = 0; t < 3; ++t)
#pragma unroll
      for (int n = 0; n < 2; ++n)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int co = 16 * cob + g + 8 * (e >> 1), ci = 8 * n + 2 * tig + (e & 1);
          float* r = red + (t * 16 * ncb + co) * 16 + ci;
          const float v = q > 0 ? *r + acc[t][n][e] : acc[t][n][e];
          if (q < 3) *r = v;
          else atomicAdd(a.dW + ((long)(3 * blockIdx.y + t) * a.Cout + co0 + co) * a.Cin + 16 * slice + ci, v);
        }
  }
}

// bias gradient: db[co] += sum_v dpre(v)[co]; a block takes 8 channels, 16 bytes a voxel (one channel after the
// other, 2 bytes a load: 0.27 ms of a 64^3 training step)
__global__ void k_bgrad(const bf16* dpre, long nvox, int Cout, float* db) {
  __shared__ float red[8][256];
  float s[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  for (long v = blockIdx.x * (long)blockDim.x + threadIdx.x; v < nvox; v += (long)gridDim.x * blockDim.x) {
    const uint4 u = *reinterpret_cast<const uint4*>(dpre + v * Cout + 8 * blockIdx.y);
    const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      s[2 * c] += __uint_as_float(w[c] << 16);
      s[2 * c + 1] += __uint_as_float(w[c] & 0xFFFF0000u);
    }
  }
#pragma unroll
  for (int c = 0; c < 8; ++c) red[c][threadIdx.x] = s[c];
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    for (int q = threadIdx.x; q < 8 * o; q += blockDim.x) red[q / o][q % o] += red[q / o][q % o + o];
    __syncthreads();
  }
  if (threadIdx.x < 8) atomicAdd(&db[8 * blockIdx.y + threadIdx.x], red[threadIdx.x][0]);
}

// min_taps: the smallest group of weights worth running this tile with
template <int NT, int MT>
static bool conv_st(const ConvArgs& a, int min_taps, cudaStream_t st) {
  const int limit = (NT * MT <= 16 ? 113 : 227) * 1024;  // the resident blocks its registers allow
  int taps = 27;
  while (taps > min_taps && st_bytes(a, MT, taps) > limit) taps /= 3;
  const int bytes = st_bytes(a, MT, taps);
  if (bytes > limit) return false;
  const int nx = (a.No + st_tx(MT) - 1) / st_tx(MT), ny = (a.No + st_ty(MT) - 1) / st_ty(MT),
            nz = (a.No + kStTz - 1) / kStTz;
  ConvArgs arg = a;
  void* args[] = {&arg, &taps};
  // the limit is one value per kernel and device, whoever launches it: always the most it may be
  if (cudaFuncSetAttribute(k_conv_st<NT, MT>, cudaFuncAttributeMaxDynamicSharedMemorySize, limit) != cudaSuccess ||
      cudaLaunchKernel((const void*)k_conv_st<NT, MT>, dim3(nx * ny * nz), dim3(kStThreads), args, bytes, st) !=
          cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return true;
}

// The staged kernel where its modes fit; the largest tile (least staging per voxel, most reuse of the
// weights) whose accumulators and staged input leave room for two blocks per SM, if the grid still gives
// every SM one.  The tile counts for more than the group of weights it leaves room for: 48 input
// channels at 128^3 369 us tap by tap on 32 x 8 x 4, 416 us with all taps staged on 16 x 8 x 4; 96 at 64^3
// 147 us on 16 x 8 x 4, 161 us in threes on 16 x 4 x 4.
static bool launch_conv_st(const UNet& U, const ConvArgs& a, cudaStream_t st) {
  auto fits = [&](const Src& s) {
    if (s.C == 0) return true;
    if (s.C != 16 && s.C != 32 && s.C != 64) return false;
    if (s.mode == G_SAME || s.mode == G_SAME_T) return s.n == a.No;
    if (s.mode == G_UP) return 2 * s.n == a.No;
    return s.mode == G_DOWN && s.n == 2 * a.No;
  };
  if (a.accumulate || !fits(a.s0) || !fits(a.s1)) return false;
  if (a.s1.C && (a.s0.mode == G_SAME_T || a.s1.mode == G_SAME_T)) return false;
  auto blocks = [&](int mt) {
    return (long)((a.No + st_tx(mt) - 1) / st_tx(mt)) * ((a.No + st_ty(mt) - 1) / st_ty(mt)) *
           ((a.No + kStTz - 1) / kStTz);
  };
  const bool big = blocks(8) >= U.nsm, mid = blocks(4) >= U.nsm;
  switch (a.Cout / 8) {
    case 2: return (big && conv_st<2, 8>(a, 1, st)) || (mid && conv_st<2, 4>(a, 1, st)) || conv_st<2, 2>(a, 1, st);
    case 4: return (mid && conv_st<4, 4>(a, 1, st)) || conv_st<4, 2>(a, 1, st);
    case 6: return (mid && conv_st<6, 4>(a, 1, st)) || conv_st<6, 2>(a, 1, st);
    case 8: return conv_st<8, 2>(a, 1, st);
    case 12: return conv_st<12, 2>(a, 1, st);
  }
  return false;
}

static void launch_conv(const UNet& U, const ConvArgs& a, cudaStream_t st) {
  // stride-1 gathers (same grid, nearest upsampling) go to the tensor-memory kernel when it fits
  auto tc_mode = [&](const Src& s, int& m) {
    if (s.C == 0) return true;
    if (s.mode == G_SAME && s.n == a.No) return (m = 0, true);
    if (s.mode == G_UP && 2 * s.n == a.No) return (m = 1, true);
    return false;
  };
  int m0 = 0, m1 = 0;
  if (U.use_tc && !a.accumulate && (a.out32 == nullptr || a.out32_ch == 1) && tc_mode(a.s0, m0) &&
      tc_mode(a.s1, m1)) {
    TcConvArgs t{a.s0.ptr, a.s1.ptr, a.s0.C, a.s1.C, m0, m1, a.No, a.W, a.bias, a.out, a.out32, a.relu, U.err};
    if (conv_tc(t, a.Cout, U.nsm, st)) return;
  }
  if (launch_conv_st(U, a, st)) return;
  const long nvox = cube(a.No);
  const int grid = (int)((nvox + 16 * CONV_MT * CONV_WARPS - 1) / (16 * CONV_MT * CONV_WARPS));
  const int threads = CONV_WARPS * 32;
  const bool down_t = a.s0.mode == G_DOWN_T;  // data gradients of the stride-2 layers: into 16 or 32 channels
  switch (a.Cout / 8) {
    case 2:
      if (down_t) k_conv<2, true><<<grid, threads, 0, st>>>(a);
      else k_conv<2, false><<<grid, threads, 0, st>>>(a);
      break;
    case 4:
      if (down_t) k_conv<4, true><<<grid, threads, 0, st>>>(a);
      else k_conv<4, false><<<grid, threads, 0, st>>>(a);
      break;
    case 6: k_conv<6, false><<<grid, threads, 0, st>>>(a); break;
    case 8: k_conv<8, false><<<grid, threads, 0, st>>>(a); break;
    case 12: k_conv<12, false><<<grid, threads, 0, st>>>(a); break;
  }
}

static Src src(const bf16* p, int C, int mode, int n) { return Src{p, C, mode, n}; }

// forward conv of layer l
static void fwd(UNet& U, int l, Src s0, Src s1, bf16* out, float* out32, int relu, cudaStream_t st) {
  Layer& y = U.L[l];
  ConvArgs a;
  memset(&a, 0, sizeof(a));
  a.s0 = s0;
  a.s1 = s1;
  a.Cin = s0.C + s1.C;
  a.Cout = y.cout;
  a.No = U.N >> y.level_out;
  a.W = y.wf;
  a.bias = y.b;
  a.out = out;
  a.out32 = out32;
  a.out32_ch = 1;
  a.relu = relu;
  launch_conv(U, a, st);
}

// Forward pass on the packed input; output channel 0 in U.out32.
static void unet_forward(UNet& U, cudaStream_t st) {
  const int n0 = U.N, n1 = U.N / 2, n2 = U.N / 4;
  Src none = src(nullptr, 0, G_SAME, 0);
  fwd(U, 0, src(U.in16, 16, G_SAME, n0), none, U.e1a, nullptr, 1, st);
  fwd(U, 1, src(U.e1a, 16, G_SAME, n0), none, U.e1b, nullptr, 1, st);
  fwd(U, 2, src(U.e1b, 16, G_DOWN, n0), none, U.d1, nullptr, 1, st);
  fwd(U, 3, src(U.d1, 32, G_SAME, n1), none, U.e2, nullptr, 1, st);
  fwd(U, 4, src(U.e2, 32, G_DOWN, n1), none, U.d2, nullptr, 1, st);
  fwd(U, 5, src(U.d2, 64, G_SAME, n2), none, U.e3, nullptr, 1, st);
  fwd(U, 6, src(U.e3, 64, G_UP, n2), src(U.e2, 32, G_SAME, n1), U.u2, nullptr, 1, st);
  fwd(U, 7, src(U.u2, 32, G_UP, n1), src(U.e1b, 16, G_SAME, n0), U.u1, nullptr, 1, st);
  fwd(U, 8, src(U.u1, 16, G_SAME, n0), none, nullptr, U.out32, 0, st);
}

// Data gradient of layer l: dIn (fp32, [n_in^3][Cin]) from dpre ([n_out^3][Cout] bf16).
static void bwd_data(UNet& U, int l, int n_in, float* dIn, cudaStream_t st) {
  Layer& y = U.L[l];
  ConvArgs a;
  memset(&a, 0, sizeof(a));
  const int n_out = U.N >> y.level_out;
  a.s0 = src(U.dpre, y.cout, y.stride == 2 ? G_DOWN_T : G_SAME_T, n_out);
  a.s1 = src(nullptr, 0, G_SAME, 0);
  a.Cin = y.cout;
  a.Cout = y.cin;
  a.No = n_in;
  a.W = y.wt;  // [27][cin][cout]: rows = input channels, k = output channels
  a.out32 = dIn;
  a.out32_ch = y.cin;
  launch_conv(U, a, st);
}

// most shared memory of k_wgrad over output grids of 2 to 512 cells a side
static int wg_limit() {
  int most = 0;
  for (int N = 2; N <= 512; ++N)
    for (int mode : {G_SAME, G_DOWN, G_UP}) most = std::max(most, 2 * wg_stage_bytes(mode, N, 32));
  return most;
}

// false: the launch was refused
static bool wgrad(UNet& U, int l, Src s0, Src s1, cudaStream_t st) {
  Layer& y = U.L[l];
  WgradArgs a{s0, s1, y.cin, y.cout, U.N >> y.level_out, U.dpre, y.gw, 0};
  const long nvox = cube(a.No);
  a.chunk = ((nvox + 63) / 64 + 15) / 16 * 16;
  const int co = y.cout < 32 ? y.cout : 32;
  int bytes = wg_stage_bytes(s0.mode, a.No, co);
  if (s1.C) bytes = std::max(bytes, wg_stage_bytes(s1.mode, a.No, co));
  bytes = std::max(2 * bytes, 3 * co * 16 * 4);
  static const int limit = wg_limit();
  void* args[] = {&a};
  const bool ok =
      cudaFuncSetAttribute(k_wgrad, cudaFuncAttributeMaxDynamicSharedMemorySize, limit) == cudaSuccess &&
      cudaLaunchKernel((const void*)k_wgrad, dim3((unsigned)((nvox + a.chunk - 1) / a.chunk), 9, y.cin / 16 * (y.cout / co)),
                       dim3(8 * co), args, bytes, st) == cudaSuccess;
  k_bgrad<<<dim3(64, y.cout / 8), 256, 0, st>>>(U.dpre, nvox, y.cout, y.gb);
  return ok;
}

}  // namespace fe

namespace fe {

// Network input for the current residual of a solve: rms(r)^2 = rr / n with
// rr read from the box scalar rr_slot, dt from SC_KDT (the solve's operator);
// the output scale rms(r) d0 of the direction goes to SC_NSCALE.  The scales, five FP64 divisions and a root, are
// formed by one thread of a block, and the fields converted off the FP64 pipe (per thread and by the conversion
// instruction they bound the kernel: 53 us at 128^3, 40 now).
template <typename T>
__global__ void __launch_bounds__(256) k_pack_fcg(const T* __restrict__ r, const T* __restrict__ dinv, long n, double* sc,
                                                  int rr_slot, double ih, bf16* __restrict__ in16) {
  __shared__ double sa, sc3;
  if (threadIdx.x == 0) {
    const double rr = sc[rr_slot], dt = sc[SC_KDT];
    const double c3 = 3.0 * dt * ih * ih, d0 = 1.0 / (1.0 / dt + c3);
    const double rms = rr > 0.0 ? sqrt(rr / (double)n) : 0.0;
    sa = rms > 0.0 ? 1.0 / (rms * d0) : 0.0;
    sc3 = c3;
    if (blockIdx.x == 0) sc[SC_NSCALE] = rms * d0;
  }
  __syncthreads();
  const double a = sa, c3 = sc3;
#pragma unroll 4
  for (long q = blockIdx.x * (long)blockDim.x + threadIdx.x; q < n; q += (long)gridDim.x * blockDim.x) {
    const double dq = widen(dinv[q]);
    pack_voxel(in16 + q * 16, narrow(widen(r[q]) * dq * a), narrow(dq * c3));
  }
}

// mean-square of a field (two-level, fixed order): part[block] partial sums
template <typename T>
__global__ void k_sumsq(const T* a, long n, double* part) {
  __shared__ double red[256];
  double s = 0.0;
  for (long q = blockIdx.x * (long)blockDim.x + threadIdx.x; q < n; q += (long)gridDim.x * blockDim.x)
    s += (double)a[q] * (double)a[q];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.x] = red[0];
}

template <typename T>
__global__ void k_scale_to_f32(const T* a, long n, double s, float* out) {
  for (long q = blockIdx.x * (long)blockDim.x + threadIdx.x; q < n; q += (long)gridDim.x * blockDim.x)
    out[q] = (float)((double)a[q] * s);
}

// Queue the copy of the flag behind the work on st; after the stream has been waited for, unet_failed says whether
// a convolution of that work gave up, and clears the flag.
void unet_queue_error(UNet* U, cudaStream_t st) {
  cudaMemcpyAsync(U->herr, U->err, sizeof(int), cudaMemcpyDeviceToHost, st);
}
bool unet_failed(UNet* U, cudaStream_t st) {
  if (*U->herr == 0) return false;
  cudaMemsetAsync(U->err, 0, sizeof(int), st);
  *U->herr = 0;
  return true;
}

// Sum of the nb = ew(N^3) block sums in U.part, added in order; *failed: whether a convolution gave up (unet_failed).
static double host_sum(UNet& U, int nb, cudaStream_t st, bool* failed = nullptr) {
  std::vector<double> h(nb + 1);
  cudaMemcpyAsync(h.data(), U.part, (nb + 1) * sizeof(double), cudaMemcpyDeviceToHost, st);
  cudaStreamSynchronize(st);
  if (failed) {
    memcpy(U.herr, &h[nb], sizeof(int));
    *failed = unet_failed(&U, st);
  }
  double s = 0.0;
  for (int b = 0; b < nb; ++b) s += h[b];
  return s;
}

UNet* unet_create(int N, bool training, int* rc) {
  UNet* U = new UNet();
  *rc = unet_alloc(*U, N, training);
  if (*rc != FE_OK) {
    cudaGetLastError();  // of the refused allocation
    unet_free(*U);
    delete U;
    return nullptr;
  }
  return U;
}

void unet_destroy(UNet* U) {
  if (!U) return;
  unet_free(*U);
  delete U;
}

// host layout per layer: W[27][cin_real][cout_real] then b[cout_real]
int unet_set_weights(UNet* U, const float* host, cudaStream_t st) {
  long off = 0;
  for (int l = 0; l < kNL; ++l) {
    Layer& y = U->L[l];
    const long nw = 27L * y.cin * y.cout;
    std::vector<float> w(nw, 0.f), b(y.cout, 0.f);
    for (int t = 0; t < 27; ++t)
      for (int ci = 0; ci < y.cin_real; ++ci)
        for (int co = 0; co < y.cout_real; ++co)
          w[((long)t * y.cout + co) * y.cin + ci] = host[off + ((long)t * y.cin_real + ci) * y.cout_real + co];
    off += 27L * y.cin_real * y.cout_real;
    for (int co = 0; co < y.cout_real; ++co) b[co] = host[off + co];
    off += y.cout_real;
    cudaMemcpyAsync(y.w, w.data(), nw * 4, cudaMemcpyHostToDevice, st);
    cudaMemcpyAsync(y.b, b.data(), y.cout * 4, cudaMemcpyHostToDevice, st);
    cudaMemsetAsync(y.mw, 0, nw * 4, st);
    cudaMemsetAsync(y.vw, 0, nw * 4, st);
    cudaMemsetAsync(y.mb, 0, y.cout * 4, st);
    cudaMemsetAsync(y.vb, 0, y.cout * 4, st);
    k_cast_weights<<<ew(nw), 256, 0, st>>>(y.w, nw, y.cout, y.cin, y.wf, y.wt);
    cudaStreamSynchronize(st);  // host vectors go out of scope
  }
  U->adam_step = 0;
  U->trained = true;
  return cudaGetLastError() == cudaSuccess ? FE_OK : FE_ERR_CUDA;
}

// One layer's parameters (or gradients) from [27][cout][cin] and [cout] to the host's order, without the padding.
__global__ void k_export(const float* __restrict__ w, const float* __restrict__ b, int cin, int cout, int cin_real,
                         int cout_real, float* __restrict__ out) {
  const int nw = 27 * cin_real * cout_real, n = nw + cout_real;
  for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < n; q += gridDim.x * blockDim.x) {
    const int co = q % cout_real, r = q / cout_real, ci = r % cin_real, t = r / cin_real;
    out[q] = q < nw ? w[((long)t * cout + co) * cin + ci] : b[q - nw];
  }
}

// which = 0: weights and biases, 1: their gradients.  Put into the host's order on the device and copied at once
// (a copy and a wait per layer array and the reordering on the host took 0.5 ms of the 64^3 training step's 2.4 ms
// for each of the two).
int unet_get_weights(UNet* U, float* host, int which, cudaStream_t st) {
  long off = 0;
  for (int l = 0; l < kNL; ++l) {
    Layer& y = U->L[l];
    const long n = 27L * y.cin_real * y.cout_real + y.cout_real;
    k_export<<<ew(n), 256, 0, st>>>(which ? y.gw : y.w, which ? y.gb : y.b, y.cin, y.cout, y.cin_real, y.cout_real,
                                    U->xfer + off);
    off += n;
  }
  cudaMemcpyAsync(host, U->xfer, off * 4, cudaMemcpyDeviceToHost, st);
  cudaStreamSynchronize(st);
  return cudaGetLastError() == cudaSuccess ? FE_OK : FE_ERR_CUDA;
}

// Network pass for the current residual of a solve (input as k_pack_fcg);
// the output y stays in U->out32 and its scale in sc[SC_NSCALE].
template <typename T>
void unet_apply_sc(UNet* U, const T* r, const T* dinv, double* sc, int rr_slot, double ih, cudaStream_t st) {
  const long n = cube(U->N);
  const int blocks = ew(n) < 4 * U->nsm ? ew(n) : 4 * U->nsm;
  k_pack_fcg<T><<<blocks, 256, 0, st>>>(r, dinv, n, sc, rr_slot, ih, U->in16);
  unet_forward(*U, st);
}

// Preconditioner scales of a residual: rms(r) from a fixed-order reduction, d0 from dt.
template <typename T>
static void precond_scales(UNet* U, const T* r, double dt, double ih, cudaStream_t st, double* rms, double* d0) {
  const long n = cube(U->N);
  const int nb = ew(n);
  k_sumsq<T><<<nb, 256, 0, st>>>(r, n, U->part);
  const double rr = host_sum(*U, nb, st);
  *rms = rr > 0.0 ? sqrt(rr / (double)n) : 0.0;
  *d0 = 1.0 / (1.0 / dt + 3.0 * dt * ih * ih);
}

// z = r dinv + rms(r) d0 net(input): the residual-form direction.
template <typename T>
int unet_apply(UNet* U, const T* r, const T* dinv, double dt, double ih, float* z, cudaStream_t st) {
  const long n = cube(U->N);
  double rms, d0;
  precond_scales<T>(U, r, dt, ih, st, &rms, &d0);
  k_pack_input<T><<<ew(n), 256, 0, st>>>(r, dinv, n, rms > 0.0 ? 1.0 / (rms * d0) : 0.0, 3.0 * dt * ih * ih,
                                         U->in16);
  unet_forward(*U, st);
  k_direction<T><<<ew(n), 256, 0, st>>>(r, dinv, U->out32, rms * d0, n, z);
  unet_queue_error(U, st);
  cudaStreamSynchronize(st);
  if (unet_failed(U, st)) return FE_ERR_CUDA;
  return cudaGetLastError() == cudaSuccess ? FE_OK : FE_ERR_CUDA;
}

// One training step on the pair (r, e) with M e = r (M of this dt): input as
// unet_apply, target t = (e - r dinv) / (rms(r) d0), loss ||y - t||^2 /
// ||t||^2, backward through every layer, Adam.  lr <= 0: gradients only.
template <typename T>
int unet_train_step(UNet* U, const T* r, const T* e, const T* dinv, double dt, double ih, double lr, double* loss,
                    cudaStream_t st) {
  if (!U->g0) return FE_ERR_UNSUPPORTED;
  const int n0 = U->N, n1 = U->N / 2, n2 = U->N / 4;
  const long v0 = cube(n0), v1 = cube(n1), v2 = cube(n2);
  const int nb = ew(v0);
  double rms, d0;
  precond_scales<T>(U, r, dt, ih, st, &rms, &d0);
  if (!(rms > 0.0)) return FE_ERR_INVALID_ARG;
  k_pack_input<T><<<ew(v0), 256, 0, st>>>(r, dinv, v0, 1.0 / (rms * d0), 3.0 * dt * ih * ih, U->in16);
  unet_forward(*U, st);
  // target into gsk0 (fp32 scratch), its norm, then loss and dL/dy
  float* tgt = U->gsk0;
  k_target<T><<<nb, 256, 0, st>>>(r, e, dinv, v0, 1.0 / (rms * d0), tgt, U->part);
  bool failed = false;
  const double tt = host_sum(*U, nb, st, &failed);
  if (failed) return FE_ERR_CUDA;  // before any weight moves
  if (!(tt > 0.0)) return FE_ERR_INVALID_ARG;
  k_loss_grad<<<nb, 256, 0, st>>>(U->out32, tgt, v0, 1.0 / tt, U->dy8, U->part);
  *loss = host_sum(*U, nb, st) / tt;
  for (int l = 0; l < kNL; ++l) {
    cudaMemsetAsync(U->L[l].gw, 0, 27L * U->L[l].cin * U->L[l].cout * 4, st);
    cudaMemsetAsync(U->L[l].gb, 0, U->L[l].cout * 4, st);
  }
  Src none = src(nullptr, 0, G_SAME, 0);
  bool ok = true;
  // out (linear)
  k_mask<<<ew(v0 * 16), 256, 0, st>>>(U->dy8, nullptr, nullptr, v0 * 16, U->dpre);
  ok = ok && wgrad(*U, 8, src(U->u1, 16, G_SAME, n0), none, st);
  bwd_data(*U, 8, n0, U->g0, st);
  // u1
  k_mask<<<ew(v0 * 16), 256, 0, st>>>(U->g0, nullptr, U->u1, v0 * 16, U->dpre);
  ok = ok && wgrad(*U, 7, src(U->u2, 32, G_UP, n1), src(U->e1b, 16, G_SAME, n0), st);
  bwd_data(*U, 7, n0, U->g0, st);
  k_up2_back<<<ew(v1 * 32), 256, 0, st>>>(U->g0, n0, 48, 32, U->g1);
  k_slice<<<ew(v0 * 16), 256, 0, st>>>(U->g0, v0, 48, 32, 16, U->gsk0);
  // u2
  k_mask<<<ew(v1 * 32), 256, 0, st>>>(U->g1, nullptr, U->u2, v1 * 32, U->dpre);
  ok = ok && wgrad(*U, 6, src(U->e3, 64, G_UP, n2), src(U->e2, 32, G_SAME, n1), st);
  bwd_data(*U, 6, n1, U->g1, st);
  k_up2_back<<<ew(v2 * 64), 256, 0, st>>>(U->g1, n1, 96, 64, U->g2);
  k_slice<<<ew(v1 * 32), 256, 0, st>>>(U->g1, v1, 96, 64, 32, U->gsk1);
  // e3
  k_mask<<<ew(v2 * 64), 256, 0, st>>>(U->g2, nullptr, U->e3, v2 * 64, U->dpre);
  ok = ok && wgrad(*U, 5, src(U->d2, 64, G_SAME, n2), none, st);
  bwd_data(*U, 5, n2, U->g2, st);
  // d2
  k_mask<<<ew(v2 * 64), 256, 0, st>>>(U->g2, nullptr, U->d2, v2 * 64, U->dpre);
  ok = ok && wgrad(*U, 4, src(U->e2, 32, G_DOWN, n1), none, st);
  bwd_data(*U, 4, n1, U->g1, st);
  // e2 (+ skip from u2)
  k_mask<<<ew(v1 * 32), 256, 0, st>>>(U->g1, U->gsk1, U->e2, v1 * 32, U->dpre);
  ok = ok && wgrad(*U, 3, src(U->d1, 32, G_SAME, n1), none, st);
  bwd_data(*U, 3, n1, U->g1, st);
  // d1
  k_mask<<<ew(v1 * 32), 256, 0, st>>>(U->g1, nullptr, U->d1, v1 * 32, U->dpre);
  ok = ok && wgrad(*U, 2, src(U->e1b, 16, G_DOWN, n0), none, st);
  bwd_data(*U, 2, n0, U->g0, st);
  // e1b (+ skip from u1)
  k_mask<<<ew(v0 * 16), 256, 0, st>>>(U->g0, U->gsk0, U->e1b, v0 * 16, U->dpre);
  ok = ok && wgrad(*U, 1, src(U->e1a, 16, G_SAME, n0), none, st);
  bwd_data(*U, 1, n0, U->g0, st);
  // e1a
  k_mask<<<ew(v0 * 16), 256, 0, st>>>(U->g0, nullptr, U->e1a, v0 * 16, U->dpre);
  ok = ok && wgrad(*U, 0, src(U->in16, 16, G_SAME, n0), none, st);
  if (cudaGetLastError() != cudaSuccess || !ok) return FE_ERR_CUDA;  // a launch was refused: no weight moves
  if (lr > 0.0) {
    U->adam_step += 1;
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.f - powf(b1, (float)U->adam_step), c2 = 1.f - powf(b2, (float)U->adam_step);
    for (int l = 0; l < kNL; ++l) {
      Layer& y = U->L[l];
      const long nw = 27L * y.cin * y.cout;
      k_adam<<<ew(nw), 256, 0, st>>>(y.w, y.gw, y.mw, y.vw, nw, (float)lr, b1, b2, 1e-8f, c1, c2, 27, y.cout, y.cin,
                                     y.wf, y.wt, y.cin_real, y.cout_real);
      k_adam<<<1, 256, 0, st>>>(y.b, y.gb, y.mb, y.vb, y.cout, (float)lr, b1, b2, 1e-8f, c1, c2, 0, y.cout, 1,
                                nullptr, nullptr, 1, y.cout_real);
    }
  }
  cudaStreamSynchronize(st);
  return cudaGetLastError() == cudaSuccess ? FE_OK : FE_ERR_CUDA;
}

float* unet_output(UNet* U) { return U->out32; }
int unet_N(const UNet* U) { return U->N; }
void unet_set_kernels(UNet* U, int tc) { U->use_tc = tc; }

#define INST(T)                                                                                         \
  template void unet_apply_sc<T>(UNet*, const T*, const T*, double*, int, double, cudaStream_t);         \
  template int unet_apply<T>(UNet*, const T*, const T*, double, double, float*, cudaStream_t);          \
  template int unet_train_step<T>(UNet*, const T*, const T*, const T*, double, double, double, double*, \
                                  cudaStream_t);
INST(double)
INST(float)

}  // namespace fe

namespace fe {
__global__ void k_bf16_to_f32(const bf16* a, long n, float* out) {
  for (long q = blockIdx.x * (long)blockDim.x + threadIdx.x; q < n; q += (long)gridDim.x * blockDim.x)
    out[q] = __bfloat162float(a[q]);
}

// Activation of layer l (0..8; 9 = packed input) after the last forward pass,
// channels-last, as floats: count = n_l^3 * C_l.
int unet_activation(UNet* U, int l, float* host, long count, cudaStream_t st) {
  const int n0 = U->N, n1 = U->N / 2, n2 = U->N / 4;
  const bf16* p = nullptr;
  long n = 0;
  switch (l) {
    case 0: p = U->e1a; n = cube(n0) * 16; break;
    case 1: p = U->e1b; n = cube(n0) * 16; break;
    case 2: p = U->d1; n = cube(n1) * 32; break;
    case 3: p = U->e2; n = cube(n1) * 32; break;
    case 4: p = U->d2; n = cube(n2) * 64; break;
    case 5: p = U->e3; n = cube(n2) * 64; break;
    case 6: p = U->u2; n = cube(n1) * 32; break;
    case 7: p = U->u1; n = cube(n0) * 16; break;
    case 8:
      if (count != cube(n0)) return FE_ERR_INVALID_ARG;
      cudaMemcpyAsync(host, U->out32, cube(n0) * 4, cudaMemcpyDeviceToHost, st);
      cudaStreamSynchronize(st);
      return FE_OK;
    case 9: p = U->in16; n = cube(n0) * 16; break;
    default: return FE_ERR_INVALID_ARG;
  }
  if (count != n) return FE_ERR_INVALID_ARG;
  float* d = nullptr;
  if (cudaMalloc(&d, n * 4) != cudaSuccess) {
    cudaGetLastError();
    return FE_ERR_OOM;
  }
  k_bf16_to_f32<<<ew(n), 256, 0, st>>>(p, n, d);
  cudaMemcpyAsync(host, d, n * 4, cudaMemcpyDeviceToHost, st);
  cudaStreamSynchronize(st);
  cudaFree(d);
  return cudaGetLastError() == cudaSuccess ? FE_OK : FE_ERR_CUDA;
}
}  // namespace fe
