// unet_tc.cu -- 3x3x3 convolutions of the U-Net preconditioner on the
// fifth-generation tensor cores (tcgen05.mma, accumulators in tensor memory).
//
// Implicit GEMM: D[voxel][co] = sum_{tap, ci} A_tap[voxel][ci] W[tap][co][ci].
// A CTA computes tiles of kR = 4 output rows of 128 voxels (x-runs at fixed
// z, rows y0..y0+3).  For each 16-channel slice of the input it stages the
// (kR + 2) x 3 input rows the tile touches (periodic wrap; nearest upsampling
// of a half-resolution source is applied while staging) in shared memory in
// the no-swizzle K-major core-matrix layout
//   [8-channel half][voxel][8 channels]   (16 bytes per voxel and half)
// so the A operand of every tap is the staged row shifted by whole voxels
// (one descriptor, no im2col copy).  An input row feeds up to three output
// rows (dy = +1, 0, -1), so the weights of one (dz, dx) are stacked along N
// ([W(dy=+1); W(dy=0); W(dy=-1)], 3 Cout rows) and one MMA with N up to
// 3 Cout updates those three rows at once: measured on this part the cost
// of an M = 128, K = 16 MMA is set by reading A from shared memory and does
// not grow with N up to 128, so wider N means fewer MMAs per voxel.
// One elected thread issues the MMAs and commits to mbarriers that release
// the staging buffers and hand finished accumulators to the epilogue
// (tcgen05.ld, bias, ReLU, BF16 stores).  Staging uses cp.async (16-byte
// chunks; the gather wraps per chunk).  Two forms: k_conv_ring keeps the
// planes that consecutive tiles share in shared memory, where they and the
// weights fit; k_conv_tc stages both per tile and slice (96 -> 32 channels).
#include <cuda_bf16.h>

#include "zbulk.cuh"
#include "zring.cuh"

namespace fe {

typedef __nv_bfloat16 bf16;

struct TcConvArgs {
  const bf16* s0;  // source 0 (channels-last), channels c0, mode 0 = same grid, 1 = half grid (upsampled)
  const bf16* s1;
  int c0, c1, m0, m1;
  int No;          // output grid side (multiple of 128)
  const bf16* W;   // [27][Cout][Cin], Cin = c0 + c1
  const float* bias;
  bf16* out;       // [No^3][Cout] or null
  float* out32;    // [No^3] channel 0, or null
  int relu;
  int* err;        // set when a bounded wait gave up
};

namespace tc {

constexpr int kR = 4;                             // output rows per tile
constexpr int kRowVox = 130;                      // 128 + halo of 1 on each side
constexpr int kRowBytes = 2 * kRowVox * 16;       // two 8-channel halves
constexpr int kRows = (kR + 2) * 3;               // input rows: kR + 2 in y, 3 in z
constexpr int kInBytes = kRows * kRowBytes;       // input slice of one stage
constexpr int kThreads = 256;

__device__ __forceinline__ uint64_t desc(unsigned saddr, unsigned lbo, unsigned sbo) {
  // no-swizzle shared-memory matrix descriptor: start, leading and stride byte
  // offsets in 16-byte units, descriptor version 1 (bits 46-47), layout 0
  return (uint64_t)((saddr >> 4) & 0x3FFF) | ((uint64_t)((lbo >> 4) & 0x3FFF) << 16) |
         ((uint64_t)((sbo >> 4) & 0x3FFF) << 32) | ((uint64_t)1 << 46);
}
// kind::f16 instruction descriptor: FP32 accumulate, BF16 A and B, both K-major
__host__ __device__ constexpr uint32_t idesc(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}
__device__ __forceinline__ void mma(uint32_t tmem, uint64_t a, uint64_t b, uint32_t id, int accum) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
      "l"(a), "l"(b), "r"(id), "r"(accum)
      : "memory");
}
// The same from converged code: the warp computes the operands, its `leader` lane issues.  hi: the high words of
// both descriptors (they differ in the start address alone, in the low words).
__device__ __forceinline__ uint32_t elect() {
  uint32_t p;
  asm volatile("{\n .reg .pred q;\n elect.sync _|q, 0xffffffff;\n selp.b32 %0, 1, 0, q;\n}\n" : "=r"(p));
  return p;
}
__device__ __forceinline__ void mma_by(uint32_t leader, uint32_t tmem, uint32_t alo, uint32_t blo, uint32_t hi,
                                       uint32_t id, int accum) {
  asm volatile(
      "{\n .reg .pred p, q;\n .reg .b64 a, b;\n setp.ne.b32 q, %0, 0;\n setp.ne.b32 p, %6, 0;\n"
      " mov.b64 a, {%2, %4};\n mov.b64 b, {%3, %4};\n"
      " @q tcgen05.mma.cta_group::1.kind::f16 [%1], a, b, %5, p;\n}\n" ::"r"(leader),
      "r"(tmem), "r"(alo), "r"(blo), "r"(hi), "r"(id), "r"(accum)
      : "memory");
}
__device__ __forceinline__ void commit_by(uint32_t leader, uint64_t* bar) {
  asm volatile(
      "{\n .reg .pred q;\n setp.ne.b32 q, %0, 0;\n"
      " @q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%1];\n}\n" ::"r"(leader),
      "r"(smem_u32(bar))
      : "memory");
}
__device__ __forceinline__ void commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}
__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void cp16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}

// NC (a multiple of 16) accumulator columns of the warp's 32 lanes: all reads in flight behind one wait
template <int NC>
__device__ __forceinline__ void tmem_ld_cols(uint32_t t, float (&v)[NC]) {
  uint32_t r[NC];
#pragma unroll
  for (int q = 0; q < NC; q += 16)
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[q]), "=r"(r[q + 1]), "=r"(r[q + 2]), "=r"(r[q + 3]), "=r"(r[q + 4]), "=r"(r[q + 5]), "=r"(r[q + 6]),
          "=r"(r[q + 7]), "=r"(r[q + 8]), "=r"(r[q + 9]), "=r"(r[q + 10]), "=r"(r[q + 11]), "=r"(r[q + 12]),
          "=r"(r[q + 13]), "=r"(r[q + 14]), "=r"(r[q + 15])
        : "r"(t + q));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int q = 0; q < NC; ++q) {
    asm volatile("" : "+r"(r[q]));  // not read before the wait
    v[q] = __uint_as_float(r[q]);
  }
}

__device__ __forceinline__ int wrapc(int v, int n) { return v < 0 ? v + n : (v >= n ? v - n : v); }

}  // namespace tc

// Shared memory: [barriers 128 B][zero operand][NS stages of input and weights]
template <int COUT, int NSTAGE>
struct TcPlan {
  static constexpr int NS = NSTAGE;
  static constexpr int wslice = 27 * COUT * 32;      // weights of one 16-channel slice (9 stacked blocks)
  static constexpr int wblock = 3 * COUT * 32;       // one (dz, dx) block: 3 Cout rows x K = 16
  static constexpr int zbytes = tc::kR * COUT * 32;  // zero B operand that clears an accumulator
  static constexpr int stage_bytes = tc::kInBytes + wslice;
  static constexpr int bytes() { return 128 + zbytes + NS * stage_bytes; }
};

// offset of W[t][co][8 h .. 8 h + 7] of one slice in the stacked layout
template <int COUT>
__device__ __forceinline__ int wofs(int t, int co, int h) {
  const int dz = t / 9 - 1, dy = (t / 3) % 3 - 1, dx = t % 3 - 1;
  const int blk = (dz + 1) * 3 + (dx + 1), n = (1 - dy) * COUT + co;
  return blk * (3 * COUT * 32) + h * (3 * COUT * 16) + n * 16;
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// Warp-specialised pipeline.  Warp 0 (one lane) issues the MMAs; warps 1-7
// stage input slices (cp.async, kLook steps ahead) and publish them on
// full[stage]; the MMA warp releases a stage with a tcgen05.commit on
// empty[stage] and hands a finished tile to the epilogue warps (4-7) on
// acc_full[buf]; they free the accumulator on acc_empty[buf].
template <int COUT, int NSTAGE>
__global__ void __launch_bounds__(tc::kThreads, 1) k_conv_tc(TcConvArgs a) {
  using P = TcPlan<COUT, NSTAGE>;
  constexpr int NS = P::NS, LOOK = NS - 1, NPROD = tc::kThreads - 32, NEPI = 128;
  extern __shared__ __align__(1024) unsigned char sm[];
  static_assert(NS >= 2 && NS <= 4, "2 to 4 stages");
  uint64_t* full = reinterpret_cast<uint64_t*>(sm);  // NS (<= 4)
  uint64_t* empty = full + 4;                        // NS
  uint64_t* acc_full = full + 8;                     // 2
  uint64_t* acc_empty = full + 10;                   // 2
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(sm + 96);
  int* abort_flag = reinterpret_cast<int*>(sm + 100);
  const int Cin = a.c0 + a.c1, nsl = Cin / 16;
  constexpr int R = tc::kR;
  unsigned char* zb = sm + 128;
  unsigned char* stage0 = zb + P::zbytes;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int No = a.No, nseg = No / 128;
  const long ntiles = (long)nseg * (No / R) * No;
  const long t0 = ntiles * blockIdx.x / gridDim.x, t1 = ntiles * (blockIdx.x + 1) / gridDim.x;
  const int ntile = (int)(t1 - t0), nsteps = ntile * nsl;
  constexpr int TCOLS = 2 * R * COUT;  // two tiles x kR rows x COUT fp32 columns (a power of two)
  static_assert((TCOLS & (TCOLS - 1)) == 0 && TCOLS >= 32 && TCOLS <= 512, "tensor memory columns");

  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(TCOLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 0) {
    for (int q = 0; q < NS; ++q) {
      mbar_init(full + q, NPROD);
      mbar_init(empty + q, 1);
    }
    for (int q = 0; q < 2; ++q) {
      mbar_init(acc_full + q, 1);
      mbar_init(acc_empty + q, NEPI);
    }
    *abort_flag = 0;
    mbar_fence_init();
  }
  for (int q = tid; q < P::zbytes / 16; q += tc::kThreads) reinterpret_cast<uint4*>(zb)[q] = make_uint4(0u, 0u, 0u, 0u);
  tc::fence_proxy_async();
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  const uint32_t tmem = *tmem_slot;

  // tiles march in z for a fixed (x segment, row group): consecutive tiles of
  // a CTA share two of their three z-planes of input rows, so the re-reads hit L2
  auto tile_of = [&](int i, int& x0, int& y0, int& z) {
    const long t = t0 + i;
    z = (int)(t % No);
    const long r = t / No;
    x0 = 128 * (int)(r % nseg);
    y0 = R * (int)(r / nseg);
  };
  auto fail = [&]() { atomicExch(abort_flag, 1); };
  auto aborted = [&]() { return *(volatile int*)abort_flag != 0; };

  if (warp == 0) {
    // ---------------- MMA issuer (the warp waits together, lane 0 issues) ----------------
    constexpr uint32_t id1 = tc::idesc(128, COUT), id2 = tc::idesc(128, 2 * COUT), id3 = tc::idesc(128, 3 * COUT),
                       idz = tc::idesc(128, R * COUT);
    int s = 0;
    for (; s < nsteps; ++s) {
      const int i = s / nsl, sl = s % nsl;
      bool w = true;
      if (sl == 0 && i >= 2) w = mbar_wait(acc_empty + (i & 1), (unsigned)(((i - 2) >> 1) & 1));
      if (w) w = mbar_wait(full + (s % NS), (unsigned)((s / NS) & 1));
      if (!__all_sync(0xffffffffu, w && !aborted())) break;  // warp-uniform decision
      tc::fence_after();
      if (lane == 0) {
        const unsigned st = smem_u32(stage0 + (s % NS) * P::stage_bytes);
        const unsigned wb = st + tc::kInBytes;
        const uint64_t abase = tc::desc(st, tc::kRowVox * 16, 128), bbase = tc::desc(wb, 3 * COUT * 16, 128);
        const uint32_t d0 = tmem + (uint32_t)((i & 1) * R * COUT);
        if (sl == 0) tc::mma(d0, abase, tc::desc(smem_u32(zb), R * COUT * 16, 128), idz, 0);  // D = 0
#pragma unroll
        for (int yy = 0; yy < R + 2; ++yy)
#pragma unroll
          for (int zz = 0; zz < 3; ++zz)
#pragma unroll
            for (int dx = 0; dx < 3; ++dx) {
              // output rows fed by input row yy: j = yy-2 .. yy (dy = +1, 0, -1) inside [0, R)
              const int jlo = yy - 2 < 0 ? 0 : yy - 2, jhi = yy > R - 1 ? R - 1 : yy;
              const int n = jhi - jlo + 1, dyi0 = jlo - (yy - 2);  // first stacked block row used
              const uint64_t aoff = (uint64_t)(((yy * 3 + zz) * tc::kRowBytes + dx * 16) >> 4);
              const uint64_t boff = (uint64_t)(((zz * 3 + dx) * (3 * COUT * 32) + dyi0 * COUT * 16) >> 4);
              const uint32_t dc = d0 + (uint32_t)(jlo * COUT);
              tc::mma(dc, abase + aoff, bbase + boff, n == 3 ? id3 : (n == 2 ? id2 : id1), 1);
            }
        tc::commit(empty + (s % NS));
        if (sl == nsl - 1) tc::commit(acc_full + (i & 1));
      }
      __syncwarp();
    }
    if (s < nsteps && lane == 0) fail();
    // every MMA issued has completed before the accumulator memory is released
    if (s > 0) mbar_wait(empty + ((s - 1) % NS), (unsigned)(((s - 1) / NS) & 1));
    __syncwarp();
  } else {
    // ---------------- producers (warps 1-7) and epilogue (warps 4-7) ----------------
    const int ptid = tid - 32;
    auto stage = [&](int s) {
      const int i = s / nsl, sl = s % nsl;
      int x0, y0, z;
      tile_of(i, x0, y0, z);
      unsigned char* st = stage0 + (s % NS) * P::stage_bytes;
      for (int q = ptid; q < tc::kRows * tc::kRowVox * 2; q += NPROD) {
        const int r = q / (tc::kRowVox * 2), rem = q - r * (tc::kRowVox * 2), v = rem >> 1, h = rem & 1;
        const int yy = tc::wrapc(y0 - 1 + r / 3, No), zz = tc::wrapc(z - 1 + r % 3, No),
                  xx = tc::wrapc(x0 - 1 + v, No);  // row r = yy * 3 + zz of the stage
        const int ch = 16 * sl + 8 * h;
        const bf16* src;
        if (ch < a.c0) {
          const int n = a.m0 ? No / 2 : No, sh = a.m0;
          src = a.s0 + ((long)(xx >> sh) + (long)n * ((yy >> sh) + (long)n * (zz >> sh))) * a.c0 + ch;
        } else {
          const int n = a.m1 ? No / 2 : No, sh = a.m1;
          src = a.s1 + ((long)(xx >> sh) + (long)n * ((yy >> sh) + (long)n * (zz >> sh))) * a.c1 + (ch - a.c0);
        }
        tc::cp16(st + r * tc::kRowBytes + h * (tc::kRowVox * 16) + v * 16, src);
      }
      unsigned char* wst = st + tc::kInBytes;
      for (int q = ptid; q < 27 * COUT * 2; q += NPROD) {
        const int h = q & 1, co = (q >> 1) % COUT, t = (q >> 1) / COUT;
        tc::cp16(wst + wofs<COUT>(t, co, h), a.W + ((long)t * COUT + co) * Cin + 16 * sl + 8 * h);
      }
    };
    auto epilogue = [&](int i) -> bool {
      if (!__all_sync(0xffffffffu, mbar_wait(acc_full + (i & 1), (unsigned)((i >> 1) & 1)))) return false;
      tc::fence_after();
      int x0, y0, z;
      tile_of(i, x0, y0, z);
      const int sub = warp & 3;
      const int x = x0 + 32 * sub + lane;
#pragma unroll 1
      for (int j = 0; j < R; ++j) {
        float v[COUT];
        tc::tmem_ld_cols<COUT>(tmem + ((uint32_t)(32 * sub) << 16) + (uint32_t)((i & 1) * R * COUT + j * COUT), v);
        const long vox = (long)x + (long)No * ((y0 + j) + (long)No * z);
#pragma unroll
        for (int c = 0; c < COUT; ++c) {
          const float u = v[c] + (a.bias ? a.bias[c] : 0.f);
          v[c] = a.relu ? fmaxf(u, 0.f) : u;
        }
        if (a.out) {
          uint4* o = reinterpret_cast<uint4*>(a.out + vox * COUT);
#pragma unroll
          for (int q = 0; q < COUT / 8; ++q) {
            __nv_bfloat162 p0 = __floats2bfloat162_rn(v[8 * q], v[8 * q + 1]);
            __nv_bfloat162 p1 = __floats2bfloat162_rn(v[8 * q + 2], v[8 * q + 3]);
            __nv_bfloat162 p2 = __floats2bfloat162_rn(v[8 * q + 4], v[8 * q + 5]);
            __nv_bfloat162 p3 = __floats2bfloat162_rn(v[8 * q + 6], v[8 * q + 7]);
            uint4 u;
            u.x = *reinterpret_cast<uint32_t*>(&p0);
            u.y = *reinterpret_cast<uint32_t*>(&p1);
            u.z = *reinterpret_cast<uint32_t*>(&p2);
            u.w = *reinterpret_cast<uint32_t*>(&p3);
            o[q] = u;
          }
        }
        if (a.out32) a.out32[vox] = v[0];
      }
      tc::fence_before();
      mbar_arrive(acc_empty + (i & 1));
      return true;
    };
    const bool epi = warp >= 4;
    for (int q = 0; q < LOOK; ++q) {
      if (q < nsteps) stage(q);
      asm volatile("cp.async.commit_group;" ::: "memory");
    }
    bool ok = true;
    for (int s = 0; s < nsteps && ok; ++s) {
      // publish step s (its group is the oldest of the LOOK outstanding ones)
      asm volatile("cp.async.wait_group %0;" ::"n"(LOOK - 1) : "memory");
      tc::fence_proxy_async();
      mbar_arrive(full + (s % NS));
      // refill: step s + LOOK reuses the stage of step s + LOOK - NS = s - 1
      const int s2 = s + LOOK;
      if (s2 < nsteps) {
        if (s2 >= NS) ok = mbar_wait(empty + (s2 % NS), (unsigned)(((s2 - NS) / NS) & 1));
        if (ok) stage(s2);
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
      const int i = s / nsl;
      if (ok && epi && s % nsl == 0 && i > 0) ok = epilogue(i - 1);
      if (aborted()) ok = false;
    }
    if (ok && epi && ntile > 0) ok = epilogue(ntile - 1);
    if (!ok) fail();
    asm volatile("cp.async.wait_group 0;" ::: "memory");
  }
  tc::fence_before();
  __syncthreads();
  if (tid == 0 && *abort_flag) atomicExch(a.err, 1);
  if (warp == 0) {
    tc::fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TCOLS) : "memory");
  }
}

// ---- resident planes: the staged input planes stay in shared memory for the three tiles that read them ----
// The streamed form (k_conv_tc) stages all three z planes of rows for every tile and waits for its own copies:
// 4.4 us per (tile, slice) at 128^3.  Here one ring of units -- unit = the R + 2 rows of one z plane and one
// 16-channel slice -- holds the planes z-1 .. z+1 of all slices plus what is staged ahead, so a tile needs one
// new plane (a third of the copies and of the L2 reads), the copies run two units ahead behind their own warps,
// and the epilogue has warps of its own.  What bounds it then is the issue of the MMAs (47 clocks each when
// nothing else holds them up): 107 clocks with the operands formed by the issuing lane alone, 85 with the whole
// warp computing them in converged code, 58 with four warps issuing for a tile each.  16 -> 16 channels at 128^3:
// 121 us streamed, then 85, 69, 56; 48 -> 16 (two rows a tile): 302, then 332, 252, 180; 32 -> 32 at 128^3 of a
// 256^3 network: 245, then 229, 191, 135.
// The MMAs are issued in the order of the streamed form, so the results are the same bits.
// Warps 0-3: epilogue (warp % 4 selects the tensor memory lanes); the next `issuers` warps issue the MMAs of every
// issuers-th tile into an accumulator of their own; then the producers, one warp per row of a unit.  A unit is free
// when the three tiles that read it have committed (`empty` counts three; tiles at the ends of a run of planes
// commit for the missing ones).
// A wait for a unit tells its fill from the one before by the parity of the slot's turn, so an issuer may wait for
// unit u only once it has seen some unit >= u - NU arrive: units are published in order, so the slot's earlier
// fills are then over, and the next one needs this tile's commit.  From unit to unit of a tile, and from an
// issuer's tile to its next, that holds (at most 4 nsl units further, 2 nsl more where a run of planes ends
// between, against 3 nsl - 1 seen and NU >= 3 nsl + 2).  An issuer's first tile can begin beyond the first NU units, where the block's first run is
// short (which runs a block gets follows from the number of blocks, that is of SMs): it waits for `primed` before,
// which the producers complete once, with unit NU - 1 (0.5 us a launch).
template <int COUT, int R>
struct TcRing {
  static constexpr int rows = R + 2, unit = rows * tc::kRowBytes;
  static constexpr int issuers = 4;
  static constexpr int threads = 32 * (4 + issuers + rows), ahead = 2;  // copy groups in flight per producer thread
  static constexpr int wslice = 27 * COUT * 32, zbytes = R * COUT * 32, head = 384, max_units = 12;
  static constexpr int room = 227 * 1024;
  // units of the ring for nsl slices: all that fit (at most max_units); 0: fewer than three planes and `ahead` units
  static __host__ __device__ int units(int nsl) {
    int n = (room - head - zbytes - nsl * wslice) / unit;
    if (n > max_units) n = max_units;
    return n >= 3 * nsl + ahead ? n : 0;
  }
  static int bytes(int nsl) { return head + zbytes + nsl * wslice + units(nsl) * unit; }
};

template <int COUT, int R>
__global__ void __launch_bounds__((TcRing<COUT, R>::threads), 1) k_conv_ring(TcConvArgs a) {
  using P = TcRing<COUT, R>;
  extern __shared__ __align__(1024) unsigned char sm[];
  uint64_t* full = reinterpret_cast<uint64_t*>(sm);  // max_units
  uint64_t* empty = full + P::max_units;             // max_units
  constexpr int NB = P::issuers;
  uint64_t* acc_full = empty + P::max_units;         // NB
  uint64_t* acc_empty = acc_full + NB;               // NB
  uint64_t* done = acc_empty + NB;                   // NB
  uint64_t* primed = done + NB;                      // 1
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(primed + 1);
  int* abort_flag = reinterpret_cast<int*>(tmem_slot + 1);
  static_assert((2 * P::max_units + 3 * NB + 1) * 8 + 8 <= P::head, "barriers fit");
  const int nsl = (a.c0 + a.c1) / 16, NU = P::units(nsl);
  unsigned char* zb = sm + P::head;
  unsigned char* wres = zb + P::zbytes;
  unsigned char* unit0 = wres + nsl * P::wslice;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int No = a.No, nseg = No / 128;
  const long ntiles = (long)nseg * (No / R) * No;
  const long t0 = ntiles * blockIdx.x / gridDim.x, t1 = ntiles * (blockIdx.x + 1) / gridDim.x;
  constexpr int TCOLS = NB * R * COUT;  // NB tiles x R rows x COUT fp32 columns (a power of two)
  static_assert((TCOLS & (TCOLS - 1)) == 0 && TCOLS >= 32 && TCOLS <= 512, "tensor memory columns");

  if (warp == 4) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(TCOLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 0) {
    for (int q = 0; q < NU; ++q) {
      mbar_init(full + q, P::rows);
      mbar_init(empty + q, 3);
    }
    for (int q = 0; q < NB; ++q) {
      mbar_init(acc_full + q, 1);
      mbar_init(acc_empty + q, 4);
      mbar_init(done + q, 1);
    }
    mbar_init(primed, P::rows);
    *abort_flag = 0;
    mbar_fence_init();
  }
  for (int q = tid; q < P::zbytes / 16; q += P::threads) reinterpret_cast<uint4*>(zb)[q] = make_uint4(0u, 0u, 0u, 0u);
  tc::fence_proxy_async();
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  const uint32_t tmem = *tmem_slot;
  auto fail = [&]() { atomicExch(abort_flag, 1); };
  auto aborted = [&]() { return *(volatile int*)abort_flag != 0; };
  // A block's tiles are runs of consecutive z in one column of (x segment, row group); a run of n tiles from zs
  // takes the planes zs - 1 .. zs + n, nsl units each.
  auto run_of = [&](long t, int& x0, int& y0, int& zs) -> int {
    zs = (int)(t % No);
    const long r = t / No;
    x0 = 128 * (int)(r % nseg);
    y0 = R * (int)(r / nseg);
    return (int)((t1 - t) < (long)(No - zs) ? (t1 - t) : (long)(No - zs));
  };

  if (warp >= 4 && warp < 4 + NB) {
    // ---------------- MMA issuers: the warp waits and computes the operands together, one lane issues ----------
    constexpr uint32_t id1 = tc::idesc(128, COUT), id2 = tc::idesc(128, 2 * COUT), id3 = tc::idesc(128, 3 * COUT),
                       idz = tc::idesc(128, R * COUT);
    const int me = warp - 4;
    const uint32_t leader = tc::elect();
    const uint32_t d0 = tmem + (uint32_t)(me * R * COUT);
    const uint64_t da = tc::desc(smem_u32(unit0), tc::kRowVox * 16, 128);
    const uint32_t hi = (uint32_t)(da >> 32), a0 = (uint32_t)da;
    const uint32_t b0 = (uint32_t)tc::desc(smem_u32(wres), 3 * COUT * 16, 128);
    const uint32_t z0 = (uint32_t)tc::desc(smem_u32(zb), R * COUT * 16, 128);
    constexpr int ustep = P::unit >> 4;
    int i = 0;        // tile of the block
    unsigned ub = 0;  // first unit of the tile's lower plane
    bool ok = true;
    if (t0 + me < t1) {  // this warp's first tile begins with unit me nsl, 2 nsl further in the second run
      const int first = me * nsl + ((int)(t0 % No) + me < No ? 0 : 2 * nsl);
      ok = __all_sync(0xffffffffu, first < NU || mbar_wait(primed, 0));
    }
    for (long t = t0; t < t1 && ok;) {
      int x0, y0, zs;
      const int n = run_of(t, x0, y0, zs);
      for (int j = 0; j < n && ok; ++j, ++i, ub += nsl) {
        if (i % NB != me) continue;
        bool w = i < NB || mbar_wait(acc_empty + me, (unsigned)((i / NB - 1) & 1));
        for (int sl = 0; sl < nsl && ok; ++sl) {
          unsigned slot[3];
#pragma unroll
          for (int zz = 0; zz < 3; ++zz) {
            const unsigned u = ub + zz * nsl + sl, q = u / NU;
            slot[zz] = u - q * NU;
            if (w) w = mbar_wait(full + slot[zz], q & 1);
          }
          ok = __all_sync(0xffffffffu, w && !aborted());  // warp-uniform decision
          if (!ok) break;
          tc::fence_after();
          uint32_t ab[3];
#pragma unroll
          for (int zz = 0; zz < 3; ++zz) ab[zz] = a0 + slot[zz] * ustep;
          const uint32_t bb = b0 + (uint32_t)(sl * (P::wslice >> 4));
          if (sl == 0) tc::mma_by(leader, d0, ab[0], z0, hi, idz, 0);  // D = 0
#pragma unroll
          for (int yy = 0; yy < R + 2; ++yy)
#pragma unroll
            for (int zz = 0; zz < 3; ++zz)
#pragma unroll
              for (int dx = 0; dx < 3; ++dx) {
                // output rows fed by input row yy: yy-2 .. yy (dy = +1, 0, -1) inside [0, R)
                const int jlo = yy - 2 < 0 ? 0 : yy - 2, jhi = yy > R - 1 ? R - 1 : yy;
                const int nj = jhi - jlo + 1, dyi0 = jlo - (yy - 2);  // first stacked block row used
                tc::mma_by(leader, d0 + (uint32_t)(jlo * COUT), ab[zz] + (uint32_t)((yy * tc::kRowBytes + dx * 16) >> 4),
                           bb + (uint32_t)(((zz * 3 + dx) * (3 * COUT * 32) + dyi0 * COUT * 16) >> 4), hi,
                           nj == 3 ? id3 : (nj == 2 ? id2 : id1), 1);
              }
          const int uses[3] = {j == 0 ? 3 : 1, 1 + (j == 0) + (j == n - 1), j == n - 1 ? 3 : 1};
#pragma unroll
          for (int zz = 0; zz < 3; ++zz)
            for (int q = 0; q < uses[zz]; ++q) tc::commit_by(leader, empty + slot[zz]);
          if (sl == nsl - 1) tc::commit_by(leader, acc_full + me);
          __syncwarp();
        }
      }
      t += n;
      ub += 2 * nsl;
    }
    if (!ok && lane == 0) fail();
    // every MMA issued has completed before the accumulator memory is released
    tc::commit_by(leader, done + me);
    __syncwarp();
    mbar_wait(done + me, 0);
  } else if (warp >= 4 + NB) {
    // ---------------- producers: warp 4 + NB + r copies row r of each unit ----------------
    const int r = warp - 4 - NB;
    for (int q = tid - 32 * (4 + NB); q < nsl * 27 * COUT * 2; q += 32 * P::rows) {  // weights, part of the first group
      const int h = q & 1, co = (q >> 1) % COUT, r2 = (q >> 1) / COUT, t = r2 % 27, sl = r2 / 27;
      tc::cp16(wres + sl * P::wslice + wofs<COUT>(t, co, h),
               a.W + ((long)t * COUT + co) * (a.c0 + a.c1) + 16 * sl + 8 * h);
    }
    unsigned v = 0, slot = 0, turn = 0;    // unit to copy, its place and how often that was filled
    unsigned vp = 0, slotp = 0;            // unit to publish
    bool ok = true;
    auto publish = [&]() {
      tc::fence_proxy_async();
      __syncwarp();
      if (lane == 0) mbar_arrive(full + slotp);
      if (lane == 0 && vp == (unsigned)NU - 1) mbar_arrive(primed);
      ++vp;
      if (++slotp == (unsigned)NU) slotp = 0;
    };
    for (long t = t0; t < t1 && ok;) {
      int x0, y0, zs;
      const int n = run_of(t, x0, y0, zs);
      const int yy = tc::wrapc(y0 - 1 + r, No);
      for (int p = -1; p <= n && ok; ++p) {
        const int zz = tc::wrapc(zs + p, No);
        for (int sl = 0; sl < nsl; ++sl) {
          if (turn > 0) ok = mbar_wait(empty + slot, (turn - 1) & 1);
          ok = __all_sync(0xffffffffu, ok && !aborted());
          if (!ok) break;
          const bool first = 16 * sl < a.c0;
          const int C = first ? a.c0 : a.c1, sh = first ? a.m0 : a.m1, nn = No >> sh;
          const bf16* row = (first ? a.s0 + 16 * sl : a.s1 + (16 * sl - a.c0)) +
                            (long)nn * ((yy >> sh) + (long)nn * (zz >> sh)) * C;
          unsigned char* dst = unit0 + slot * P::unit + r * tc::kRowBytes;
          // voxels x0 .. x0 + 127 (16 at a time, two 8-channel halves each), then the two at the ends
          const int h = lane & 1, vx = lane >> 1;
          const bf16* src = row + (long)((x0 + vx) >> sh) * C + 8 * h;
          unsigned char* d = dst + h * (tc::kRowVox * 16) + (vx + 1) * 16;
          const int sstep = (16 >> sh) * C;
#pragma unroll
          for (int q = 0; q < 8; ++q) tc::cp16(d + q * 256, src + q * sstep);
          if (lane < 4) {
            const int e = lane >> 1, xx = e ? tc::wrapc(x0 + 128, No) : tc::wrapc(x0 - 1, No);
            tc::cp16(dst + h * (tc::kRowVox * 16) + e * 129 * 16, row + (long)(xx >> sh) * C + 8 * h);
          }
          asm volatile("cp.async.commit_group;" ::: "memory");
          ++v;
          if (++slot == (unsigned)NU) {
            slot = 0;
            ++turn;
          }
          if (v > (unsigned)P::ahead) {
            asm volatile("cp.async.wait_group %0;" ::"n"(P::ahead) : "memory");
            publish();
          }
        }
      }
      t += n;
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    if (ok)
      while (vp < v) publish();
    else if (lane == 0)
      fail();
  } else {
    // ---------------- epilogue ----------------
    constexpr int JB = R * COUT <= 64 ? R : 64 / COUT;  // rows read together: 64 columns
    int i = 0;
    bool ok = true;
    for (long t = t0; t < t1 && ok;) {
      int x0, y0, zs;
      const int n = run_of(t, x0, y0, zs);
      const int x = x0 + 32 * warp + lane;
      for (int j = 0; j < n; ++j, ++i) {
        ok = __all_sync(0xffffffffu, mbar_wait(acc_full + i % NB, (unsigned)((i / NB) & 1)));
        if (!ok) break;
        tc::fence_after();
        const uint32_t tb = tmem + ((uint32_t)(32 * warp) << 16) + (uint32_t)((i % NB) * R * COUT);
#pragma unroll 1
        for (int j0 = 0; j0 < R; j0 += JB) {
          float v[JB * COUT];
          tc::tmem_ld_cols<JB * COUT>(tb + (uint32_t)(j0 * COUT), v);
#pragma unroll
          for (int jj = 0; jj < JB; ++jj) {
            const long vox = (long)x + (long)No * ((y0 + j0 + jj) + (long)No * (zs + j));
            float* w = v + jj * COUT;
#pragma unroll
            for (int c = 0; c < COUT; ++c) {
              const float u = w[c] + (a.bias ? __ldg(a.bias + c) : 0.f);
              w[c] = a.relu ? fmaxf(u, 0.f) : u;
            }
            if (a.out) {
              uint4* o = reinterpret_cast<uint4*>(a.out + vox * COUT);
#pragma unroll
              for (int q = 0; q < COUT / 8; ++q) {
                __nv_bfloat162 p[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) p[e] = __floats2bfloat162_rn(w[8 * q + 2 * e], w[8 * q + 2 * e + 1]);
                o[q] = make_uint4(*reinterpret_cast<uint32_t*>(&p[0]), *reinterpret_cast<uint32_t*>(&p[1]),
                                  *reinterpret_cast<uint32_t*>(&p[2]), *reinterpret_cast<uint32_t*>(&p[3]));
              }
            }
            if (a.out32) a.out32[vox] = w[0];
          }
        }
        tc::fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(acc_empty + i % NB);
        if (aborted()) ok = false;
      }
      t += n;
    }
    if (!ok && lane == 0) fail();
  }
  tc::fence_before();
  __syncthreads();
  if (tid == 0 && *abort_flag) atomicExch(a.err, 1);
  if (warp == 4) {
    tc::fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TCOLS) : "memory");
  }
}

// ---- host ----------------------------------------------------------------------------------------
// Launch if the layer fits (stride 1, output grid a multiple of 128, Cout 16 or 32, source channels
// multiples of 16); returns 0 otherwise.  Resident planes where three planes of all slices, two units ahead and
// the weights fit in shared memory (rows of four where they do, else of two); else the streamed form.
// limit: the most shared memory of any layer, since it is one value per kernel and device, whoever launches it.
template <typename K>
static int tc_launch(K kernel, TcConvArgs a, int rows, int threads, int limit, int bytes, int nsm, cudaStream_t st) {
  const long ntiles = (long)(a.No / 128) * (a.No / rows) * a.No;
  void* args[] = {&a};
  if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, limit) != cudaSuccess ||
      cudaLaunchKernel((const void*)kernel, dim3((unsigned)(ntiles < nsm ? ntiles : nsm)), dim3(threads), args, bytes,
                       st) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return 1;
}

template <int COUT, int R>
static int ring_launch(const TcConvArgs& a, int nsm, cudaStream_t st) {
  using P = TcRing<COUT, R>;
  const int nsl = (a.c0 + a.c1) / 16;
  return P::units(nsl) ? tc_launch(k_conv_ring<COUT, R>, a, R, P::threads, P::room, P::bytes(nsl), nsm, st) : 0;
}


int conv_tc(const TcConvArgs& a, int Cout, int nsm, cudaStream_t st) {
  const int cin = a.c0 + a.c1;
  if (a.No < 128 || a.No % 128 || (a.c0 % 16) || (a.c1 % 16) || cin == 0 || !a.err) return 0;
  switch (Cout) {
    case 16: return ring_launch<16, 4>(a, nsm, st) || ring_launch<16, 2>(a, nsm, st);
    case 32: {
      using P = TcPlan<32, 2>;
      return ring_launch<32, 2>(a, nsm, st) ||
             tc_launch(k_conv_tc<32, 2>, a, tc::kR, tc::kThreads, P::bytes(), P::bytes(), nsm, st);
    }
  }
  return 0;
}

}  // namespace fe
