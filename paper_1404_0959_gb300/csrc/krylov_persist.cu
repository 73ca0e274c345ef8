// krylov_persist.cu -- the FP64 pressure solves of small boxes in one launch.
//
// A box of 32^3 cells gives an iteration of Jacobi-PCG two kernels of a few
// microseconds each; what the host-driven solve paid for was their launches,
// their ramps and the host's look at the convergence flag (25 us per iteration
// at 32^3, 92 us per BiCGStab iteration at 45^3).  Here one cooperative launch
// runs the whole solve: every block keeps its cells' vectors in registers, only
// the vectors that neighbours read go through global memory (L2), and the blocks
// of a box meet once per inner product.
//
// Units and sums: unit u of a box is its cells [128 u, 128 u + 128); a block owns
// 1, 2, 4 or 8 consecutive units, aligned.  A box's sum is one binary tree over its
// units (adjacent pairs, then pairs of pairs): a block publishes the sum of its
// subtree, and every block adds those of its box up the rest of the tree.  So the
// sums (and the iterates) of a box do not depend on how many blocks it was given,
// in an ensemble or alone, and no block waits for a coordinator's value.  Boxes that the device
// cannot hold at once are launched in groups, one after the other.
//
// A meeting: publish, count up the box's counter, wait until all blocks have (one
// thread per block polls), read the published sums.  Two sets of sums alternate: a
// block can be at most one meeting ahead of another.  A meeting alone, in a probe
// with 256 threads per block (the kernels have 128): 3.2 us for 54 blocks, 3.4 us for
// 152, 4.1 us for 304, against 3.3, 5.7 and 10.9 us where every block polls every
// other's sum, and 3.2 us at 152 through clusters of eight.  The counters are cleared before each launch.  Waits are
// bounded: a block that gives up sets SC_KERR, finishes, and leaves the others to
// their own limits.
#include <algorithm>
#include <new>
#include <vector>

#include "fe_internal.cuh"

namespace fe {

constexpr int kPkThreads = 128;  // cells of a unit, threads of a block
constexpr int kPkWarps = kPkThreads / 32;
constexpr int kPkPerSm = 4;      // resident blocks per SM asked for (128 registers)
constexpr int kPkMaxUnits = 8;   // units per block, at most
constexpr int kPkLeaves = 8;     // published sums per thread, at most: 1024 blocks of a box
#ifndef FE_PK_SPINS
#define FE_PK_SPINS (1 << 22)  // polls of a meeting's counter before a block gives up: seconds
#endif
constexpr int kPkSpins = FE_PK_SPINS;
constexpr int kPkLine = 32;      // words between the counters of two boxes (one line each)

// A block's place: box, its first unit, its units, the box's first block and first cell among all boxes.
struct PkBlock {
  int box, u0, mine, b0;
  long cell0;
};

template <typename T>
__device__ __forceinline__ T* Fp(const BoxDev& B, int slot) {
  return reinterpret_cast<T*>(B.f[slot]);
}
// The meetings of the blocks of one box.
struct Meet {
  double* sums;        // published sums of the box: [2 sets][2 values][blocks]
  unsigned* counter;
  int blocks, me, mine;  // blocks of the box, this one, its units
  unsigned epoch = 0;
  bool failed = false;
};

struct MeetShared {
  double val[2][kPkMaxUnits][kPkThreads];
  double unit[2][kPkMaxUnits];
  double sum[2][kPkThreads];
  double out[4];  // the solver's scalars after a meeting
  int go;         // 0: finished
  int bad;
};

// the binary tree over 128 values in shared memory, adjacent pairs first (one warp)
__device__ __forceinline__ double pk_tree(const double* e, int lane) {
  e += 4 * lane;
  double a = (e[0] + e[1]) + (e[2] + e[3]);
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
  return a;
}

// One thread: count this block in and wait for the others.
__device__ __forceinline__ void pk_wait(Meet& m, MeetShared& sh) {
  __threadfence();  // this block's stores before the count
  atomicAdd(m.counter, 1u);
  const unsigned all = m.epoch * (unsigned)m.blocks;
  int spins = 0;
  bool ok = !m.failed;
  while (ok && *(volatile unsigned*)m.counter < all) ok = ++spins < kPkSpins;
  __threadfence();  // the other blocks' stores after it
  sh.bad = ok ? 0 : 1;
}

// Sums LV t .. LV t + LV - 1 of value k (zeros beyond the box's blocks), added up the tree.
template <int LV>
__device__ __forceinline__ double pk_gather(const Meet& m, const double* set) {
  double l[LV];
#pragma unroll
  for (int j = 0; j < LV; ++j) l[j] = (int)threadIdx.x * LV + j < m.blocks ? __ldcg(set + threadIdx.x * LV + j) : 0.0;
#pragma unroll
  for (int o = 1; o < LV; o <<= 1)
#pragma unroll
    for (int j = 0; j < LV; j += 2 * o) l[j] += l[j + o];
  return l[0];
}

// v[k][s]: this thread's share of value k in unit s of the block.  Afterwards everything the blocks of
// the box stored to global memory before is visible, and fin(totals) has run in one thread: the scalars it
// leaves in shared memory are for all.  The FP64 pipe takes 16 clocks per warp instruction and 68 from one
// add to the next, so sums and scalars are left to one warp (all warps forming them took 5 of 14 us per
// iteration at 32^3).
template <int K, int UPC, typename Fin>
__device__ __forceinline__ void meet(Meet& m, MeetShared& sh, const double (&v)[K][UPC], Fin fin) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  ++m.epoch;
  double* set = m.sums + (size_t)(m.epoch & 1u) * 2 * m.blocks;
#pragma unroll
  for (int k = 0; k < K; ++k)
#pragma unroll
    for (int s = 0; s < UPC; ++s) sh.val[k][s][tid] = v[k][s];
  __syncthreads();
#pragma unroll
  for (int q = 0; q < (K * UPC + kPkWarps - 1) / kPkWarps; ++q) {
    const int i = q * kPkWarps + warp;
    if (i < K * UPC) {
      const double a = pk_tree(sh.val[i % K][i / K], lane);
      if (lane == 0) sh.unit[i % K][i / K] = a;
    }
  }
  if (K * UPC > 1) __syncthreads();
  if (tid == 0) {
#pragma unroll
    for (int k = 0; k < K; ++k) {
      double e[UPC];
#pragma unroll
      for (int s = 0; s < UPC; ++s) e[s] = sh.unit[k][s];
#pragma unroll
      for (int o = 1; o < UPC; o <<= 1)
#pragma unroll
        for (int s = 0; s < UPC; s += 2 * o) e[s] += e[s + o];
      set[(size_t)k * m.blocks + m.me] = e[0];
    }
    pk_wait(m, sh);
  }
  __syncthreads();
  m.failed = sh.bad != 0;
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const double* p = set + (size_t)k * m.blocks;
    sh.sum[k][tid] = m.blocks <= kPkThreads       ? pk_gather<1>(m, p)
                     : m.blocks <= 2 * kPkThreads ? pk_gather<2>(m, p)
                     : m.blocks <= 4 * kPkThreads ? pk_gather<4>(m, p)
                                                  : pk_gather<kPkLeaves>(m, p);
  }
  __syncthreads();
  if (warp == 0) {
    double t[K];
#pragma unroll
    for (int k = 0; k < K; ++k) t[k] = pk_tree(sh.sum[k], lane);
    if (lane == 0) fin(t);
  }
  __syncthreads();
}

// The same without a value: the blocks' stores become visible to each other.
__device__ __forceinline__ void meet_plain(Meet& m, MeetShared& sh) {
  ++m.epoch;
  __syncthreads();
  if (threadIdx.x == 0) pk_wait(m, sh);
  __syncthreads();
  m.failed = sh.bad != 0;
}

// Flat offsets of the six neighbours of a cell.
struct PkNbr {
  int c;
  int xm, xp, ym, yp, zm, zp;
  __device__ __forceinline__ PkNbr(int cell, int N) {
    const int NN = N * N, n3 = NN * N;
    c = cell;
    const int i = cell % N, j = (cell / N) % N;
    xm = i == 0 ? cell + N - 1 : cell - 1;
    xp = i == N - 1 ? cell - N + 1 : cell + 1;
    ym = j == 0 ? cell + NN - N : cell - N;
    yp = j == N - 1 ? cell - NN + N : cell + N;
    zm = cell < NN ? cell + n3 - NN : cell - NN;
    zp = cell >= n3 - NN ? cell - n3 + NN : cell + NN;
  }
};

// Jacobi-PCG (the iteration of kz_cg_dirmatvec and k_cg_rupdate): z = D^{-1} r and the directions
// alternating between K_PD and K_PP are what neighbours read; x, r, pd and q stay in registers.  Two
// meetings per iteration.  FP64 work per cell and iteration: about 25 operations, on as many SMs as the
// box has units.
template <int UPC>
__global__ void __launch_bounds__(kPkThreads, kPkPerSm) kc_cg(const BoxDev* boxes, const PkBlock* work,
                                                              double* sums, unsigned* counters, double*) {
  __shared__ MeetShared sh;
  const PkBlock w = work[blockIdx.x];
  const BoxDev& B = boxes[w.box];
  Meet m;
  m.me = w.u0 / UPC;
  m.mine = w.mine;
  m.sums = sums + (size_t)w.b0 * 4;
  m.counter = counters + w.box * kPkLine;
  const int N = B.N, n3 = N * N * N;
  m.blocks = (n3 + kPkThreads * UPC - 1) / (kPkThreads * UPC);
  const double* __restrict__ b = Fp<double>(B, K_B);
  const double* __restrict__ dinv = Fp<double>(B, W_DINV);
  const double* __restrict__ psi = Fp<double>(B, W_PSI);
  double* z = Fp<double>(B, K_AUX);
  double *pa = Fp<double>(B, K_PD), *pb = Fp<double>(B, K_PP);
  const double dt = B.sc[SC_KDT], ih = B.ih, idt = 1.0 / dt, lapc = 0.5 * dt * ih * ih;
  const double tol = B.sc[SC_TOL];
  const int maxit = (int)B.sc[SC_MAXIT];
  const int tid = threadIdx.x;
  // the operator as (psi / dt + 6 lapc) pd - lapc (sum of neighbours)
  auto diag = [&](int c) { return fma(psi[c], idt, 6.0 * lapc); };
  constexpr bool KEEP = UPC <= 2;  // D^{-1} and the diagonal of more cells are read again
  double x[UPC], r[UPC], zo[UPC], pd[UPC], q[UPC], di[UPC], dg[UPC], v1[1][UPC], v2[2][UPC];
  auto cell = [&](int s) { return (w.u0 + s) * kPkThreads + tid; };
  auto on = [&](int s) { return s < m.mine && cell(s) < n3; };
#pragma unroll
  for (int s = 0; s < UPC; ++s) {
    x[s] = r[s] = zo[s] = pd[s] = q[s] = di[s] = dg[s] = v2[0][s] = v2[1][s] = v1[0][s] = 0.0;
    if (on(s)) {
      const int c = cell(s);
      if (KEEP) {
        di[s] = dinv[c];
        dg[s] = diag(c);
      }
      r[s] = b[c];
      zo[s] = r[s] * dinv[c];
      z[c] = zo[s];
      v2[0][s] = r[s] * zo[s];
      v2[1][s] = r[s] * r[s];
    }
  }
  // one thread's scalars: rz, ||r||^2 and the stopping bound stay with it, alpha and beta go to all
  double rz = 0.0, rr = 0.0, bb = 0.0, stop = 0.0, alpha = 0.0, beta = 0.0;
  int it = 0;
  bool conv = false;
  meet<2, UPC>(m, sh, v2, [&](const double* t) {
    rz = t[0];
    bb = rr = t[1];
    stop = (tol * sqrt(bb)) * (tol * sqrt(bb));
    conv = !(bb > 0.0);
    sh.go = conv ? 0 : 1;
  });
  while (sh.go != 0 && !m.failed) {
    const double* po = (it & 1) ? pb : pa;
    double* pn = (it & 1) ? pa : pb;
#pragma unroll
    for (int s = 0; s < UPC; ++s) {
      if (!on(s)) continue;
      const PkNbr n(cell(s), N);
      auto dir = [&](int c) {
        const double zc = __ldcg(&z[c]);
        return it == 0 ? zc : fma(beta, __ldcg(&po[c]), zc);
      };
      const double pc = it == 0 ? zo[s] : fma(beta, pd[s], zo[s]);
      const double nb = (dir(n.xm) + dir(n.xp)) + (dir(n.ym) + dir(n.yp)) + (dir(n.zm) + dir(n.zp));
      const double y = fma(KEEP ? dg[s] : diag(n.c), pc, -lapc * nb);
      pn[n.c] = pc;
      pd[s] = pc;
      q[s] = y;
      v1[0][s] = pc * y;
    }
    meet<1, UPC>(m, sh, v1, [&](const double* t) { sh.out[0] = rz / t[0]; });
    alpha = sh.out[0];
#pragma unroll
    for (int s = 0; s < UPC; ++s) {
      if (!on(s)) continue;
      const int c = cell(s);
      x[s] = fma(alpha, pd[s], x[s]);
      r[s] = fma(-alpha, q[s], r[s]);
      zo[s] = r[s] * (KEEP ? di[s] : dinv[c]);
      z[c] = zo[s];
      v2[0][s] = r[s] * zo[s];
      v2[1][s] = r[s] * r[s];
    }
    ++it;
    meet<2, UPC>(m, sh, v2, [&](const double* t) {
      rr = t[1];
      if (rr <= stop) conv = true, sh.go = 0;
      else if (it >= maxit) sh.go = 0;
      else {
        sh.out[1] = t[0] / rz;
        rz = t[0];
      }
    });
    beta = sh.out[1];
  }
  double* X = Fp<double>(B, K_X);
#pragma unroll
  for (int s = 0; s < UPC; ++s)
    if (on(s)) X[cell(s)] = x[s];
  if (w.u0 == 0 && tid == 0) {
    double* sc = B.sc;
    sc[SC_RZ] = rz;
    sc[SC_BB] = bb;
    sc[SC_RR] = rr;
    sc[SC_ALPHA] = alpha;
    sc[SC_BETA] = beta;
    sc[SC_ITERS] = it;
    sc[SC_DONE] = 1.0;
    sc[SC_CONV] = conv ? 1.0 : 0.0;
  }
  if (m.failed && tid == 0) B.sc[SC_KERR] = 1.0;
}

// Right-preconditioned BiCGStab for any operator (the iteration of k_bicg_p .. k_bicg_x).  Neighbours
// read the preconditioned vector of the operator (K_PD).  The operator is formed once as coefficients per
// cell, own, then -2, -1, +1, +2 along x, y, z (the transonic term reaches two cells): 13 FP64
// multiply-adds per application where evaluating psi, the interpolations and the face products took 36
// (BiCGStab at 45^3 92 us per iteration kernel by kernel, 32 us here).  x, r (s between the two operators), p, v and t stay in
// registers; five meetings per iteration.
constexpr int kPkCoef = 13;
template <int UPC>
__global__ void __launch_bounds__(kPkThreads, kPkPerSm) kc_bicg(const BoxDev* boxes, const PkBlock* work,
                                                                double* sums, unsigned* counters, double* coef) {
  __shared__ MeetShared sh;
  const PkBlock w = work[blockIdx.x];
  const BoxDev& B = boxes[w.box];
  Meet m;
  m.me = w.u0 / UPC;
  m.mine = w.mine;
  m.sums = sums + (size_t)w.b0 * 4;
  m.counter = counters + w.box * kPkLine;
  const int N = B.N, NN = N * N, n3 = NN * N;
  m.blocks = (n3 + kPkThreads * UPC - 1) / (kPkThreads * UPC);
  const bool transonic = B.transonic != 0;
  const double* __restrict__ b = Fp<double>(B, K_B);
  const double* __restrict__ dinv = Fp<double>(B, W_DINV);
  const double* __restrict__ psi = Fp<double>(B, W_PSI);
  double* A1 = Fp<double>(B, K_PD);
  double* C = coef + w.cell0 * kPkCoef;
  const double dt = B.sc[SC_KDT], ih = B.ih, idt = 1.0 / dt, lapc = 0.5 * dt * ih * ih, ct = 0.03125 * ih;
  const double tol = B.sc[SC_TOL];
  const int maxit = (int)B.sc[SC_MAXIT];
  const int tid = threadIdx.x;
  double x[UPC], r[UPC], p[UPC], v[UPC], t[UPC], d1[1][UPC], d2[2][UPC];
  auto cell = [&](int s) { return (w.u0 + s) * kPkThreads + tid; };
  auto on = [&](int s) { return s < m.mine && cell(s) < n3; };
  // offsets of the cells at -2, -1, 1, 2 along axis d
  auto line = [&](int c, int d, int (&o)[4]) {
    const int i = d == 0 ? c % N : d == 1 ? (c / N) % N : c / NN, st = d == 0 ? 1 : d == 1 ? N : NN, base = c - i * st;
    o[0] = base + st * (i >= 2 ? i - 2 : i - 2 + N);
    o[1] = base + st * (i >= 1 ? i - 1 : i - 1 + N);
    o[2] = base + st * (i < N - 1 ? i + 1 : i + 1 - N);
    o[3] = base + st * (i < N - 2 ? i + 2 : i + 2 - N);
  };
  // M applied to the vector in K_PD (own value a)
  auto apply = [&](int c, double a) {
    double y[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      int o[4];
      line(c, d, o);
      const double* q = C + (long)(1 + 4 * d) * n3 + c;
      y[d] = q[n3] * __ldcg(&A1[o[1]]);
      y[d] = fma(q[2 * (long)n3], __ldcg(&A1[o[2]]), y[d]);
      if (transonic) {
        y[d] = fma(q[0], __ldcg(&A1[o[0]]), y[d]);
        y[d] = fma(q[3 * (long)n3], __ldcg(&A1[o[3]]), y[d]);
      }
    }
    return fma(C[c], a, (y[0] + y[1]) + y[2]);
  };
#pragma unroll
  for (int s = 0; s < UPC; ++s) {
    x[s] = r[s] = p[s] = v[s] = t[s] = d1[0][s] = d2[0][s] = d2[1][s] = 0.0;
    if (on(s)) {
      const int c = cell(s);
      r[s] = b[c];
      d1[0][s] = r[s] * r[s];
      // (1/2) D(I4(psi x) I4(HbyA)) with f, g = I4(HbyA) at the +1/2, -1/2 faces:
      // f (9 (w_0 + w_1) - (w_-1 + w_2)) - g (9 (w_-1 + w_0) - (w_-2 + w_1)), w = psi x
      double own = fma(psi[c], idt, 6.0 * lapc);
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        int o[4];
        line(c, d, o);
        double* q = C + (long)(1 + 4 * d) * n3 + c;
        double m1 = -lapc, p1 = -lapc;
        if (transonic) {
          const double* hb = Fp<double>(B, W_HB0 + d);
          const double h0 = hb[c], hm1 = hb[o[1]], hp1 = hb[o[2]];
          const double f = ct * 0.0625 * (9.0 * (h0 + hp1) - (hm1 + hb[o[3]]));
          const double g = ct * 0.0625 * (9.0 * (hm1 + h0) - (hb[o[0]] + hp1));
          own += 9.0 * (f - g) * psi[c];
          m1 -= (f + 9.0 * g) * psi[o[1]];
          p1 += (9.0 * f + g) * psi[o[2]];
          q[0] = g * psi[o[0]];
          q[3 * (long)n3] = -f * psi[o[3]];
        }
        q[n3] = m1;
        q[2 * (long)n3] = p1;
      }
      C[c] = own;
    }
  }
  // one thread's scalars; beta, omega and alpha go to all
  double rho = 0.0, rho_old = 1.0, rr = 0.0, bb = 0.0, stop = 0.0, alpha = 1.0, omega = 1.0;
  int it = 0;
  bool conv = false;
  meet<1, UPC>(m, sh, d1, [&](const double* q) {
    bb = rho = rr = q[0];
    stop = (tol * sqrt(bb)) * (tol * sqrt(bb));
    conv = !(bb > 0.0);
    sh.go = conv ? 0 : 1;
    sh.out[0] = rho;  // beta = (rho / rho_old)(alpha / omega)
  });
  while (sh.go != 0 && !m.failed) {
    const double beta = sh.out[0];
#pragma unroll
    for (int s = 0; s < UPC; ++s)
      if (on(s)) {
        p[s] = r[s] + beta * (p[s] - omega * v[s]);
        A1[cell(s)] = p[s] * dinv[cell(s)];
      }
    meet_plain(m, sh);
#pragma unroll
    for (int s = 0; s < UPC; ++s)
      if (on(s)) {
        const int c = cell(s);
        v[s] = apply(c, p[s] * dinv[c]);
        d1[0][s] = b[c] * v[s];
      }
    meet<1, UPC>(m, sh, d1, [&](const double* q) { sh.out[1] = rho / q[0]; });
    alpha = sh.out[1];
#pragma unroll
    for (int s = 0; s < UPC; ++s)
      if (on(s)) {
        r[s] = r[s] - alpha * v[s];
        A1[cell(s)] = r[s] * dinv[cell(s)];
      }
    meet_plain(m, sh);
#pragma unroll
    for (int s = 0; s < UPC; ++s)
      if (on(s)) {
        const int c = cell(s);
        t[s] = apply(c, r[s] * dinv[c]);
        d2[0][s] = t[s] * r[s];
        d2[1][s] = t[s] * t[s];
      }
    meet<2, UPC>(m, sh, d2, [&](const double* q) { sh.out[2] = q[0] / q[1]; });
    omega = sh.out[2];
#pragma unroll
    for (int s = 0; s < UPC; ++s)
      if (on(s)) {
        const int c = cell(s);
        const double di = dinv[c];
        x[s] = x[s] + alpha * (p[s] * di) + omega * (r[s] * di);
        r[s] = r[s] - omega * t[s];
        d2[0][s] = r[s] * r[s];
        d2[1][s] = b[c] * r[s];
      }
    ++it;
    meet<2, UPC>(m, sh, d2, [&](const double* q) {
      rr = q[0];
      rho_old = rho;
      rho = q[1];
      if (rr <= stop) conv = true, sh.go = 0;
      else if (it >= maxit) sh.go = 0;
      else sh.out[0] = (rho / rho_old) * (alpha / omega);
    });
  }
  double* X = Fp<double>(B, K_X);
#pragma unroll
  for (int s = 0; s < UPC; ++s)
    if (on(s)) X[cell(s)] = x[s];
  if (w.u0 == 0 && tid == 0) {
    double* sc = B.sc;
    sc[SC_BB] = bb;
    sc[SC_RZ] = rho;
    sc[SC_RHO_OLD] = rho_old;
    sc[SC_RR] = rr;
    sc[SC_ALPHA] = alpha;
    sc[SC_OMEGA] = omega;
    sc[SC_ITERS] = it;
    sc[SC_DONE] = 1.0;
    sc[SC_CONV] = conv ? 1.0 : 0.0;
  }
  if (m.failed && tid == 0) B.sc[SC_KERR] = 1.0;
}

// ---- launch ---------------------------------------------------------------------------
constexpr int kPkBicgUnits = 4;  // units per block of BiCGStab (its five register vectors)

typedef void (*PkKernel)(const BoxDev*, const PkBlock*, double*, unsigned*, double*);
static PkKernel pk_kernel(bool bicg, int upc) {
  if (bicg) return upc == 1 ? kc_bicg<1> : upc == 2 ? kc_bicg<2> : kc_bicg<4>;
  return upc == 1 ? kc_cg<1> : upc == 2 ? kc_cg<2> : upc == 4 ? kc_cg<4> : kc_cg<8>;
}

// The one-launch solves of a context: the blocks of the boxes that take one, in groups that the device holds at
// once (one launch each), their counters, sums and BiCGStab coefficients, in one allocation.
struct PkGroup {
  int first, blocks, upc;
};
struct Persist {
  std::vector<PkGroup> groups;
  std::vector<char> takes;  // per box
  size_t counter_bytes = 0;
  PkBlock* work = nullptr;
  unsigned* counters = nullptr;
  double* sums = nullptr;
  double* coef = nullptr;
  bool bicg = false;
};

void persist_free(Persist* P) {
  if (!P) return;
  cudaFree(P->work);
  delete P;
}

bool persist_takes(const Persist* P, int box) { return P && P->takes[box]; }

// A box takes the one-launch solve where the device holds its blocks at once: a function of the box alone, since
// the kernel-by-kernel solve adds its sums in another order.  The boxes that do are filled into groups at the most
// units per block; a group then runs with the fewest that fit.  Against the kernel-by-kernel solve of all boxes of a
// context that is too large for one launch, ms per step: CG, where that solve is bound by the FP64 pipe too and forms
// each direction once, 3 boxes of 64^3 4.48 -> 4.66, 8 of them 9.97 -> 11.5, 64 of 32^3 to 96^3 82.0 -> 90.6;
// BiCGStab, 8 boxes of 48^3 16.3 -> 7.8, 48 of 32^3 24.8 -> 13.1.
// null with *rc = FE_OK: no box does, the device has no cooperative launches or no memory for the solves (the boxes
// then iterate kernel by kernel).  No CUDA error is left behind in that case.
Persist* persist_create(const int* N, int nb, int nsm, bool bicg, cudaStream_t st, int* rc) {
  *rc = FE_OK;
  int dev = 0, coop = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess || !coop) {
    cudaGetLastError();
    return nullptr;
  }
  const int most = bicg ? kPkBicgUnits : kPkMaxUnits;
  long cap[kPkMaxUnits + 1];  // resident blocks of the device, per units of a block
  for (int upc = 1; upc <= most; upc *= 2) {
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, pk_kernel(bicg, upc), kPkThreads, 0) != cudaSuccess) {
      cudaGetLastError();
      return nullptr;
    }
    cap[upc] = (long)std::min(per_sm, kPkPerSm) * nsm;
  }
  auto units = [&](int b) { return ((long)N[b] * N[b] * N[b] + kPkThreads - 1) / kPkThreads; };
  auto blocks = [&](int b, int upc) { return (units(b) + upc - 1) / upc; };
  auto fits = [&](const std::vector<int>& g, int upc) {
    long sum = 0, largest = 0;
    for (int b : g) {
      sum += blocks(b, upc);
      largest = std::max(largest, blocks(b, upc));
    }
    return sum <= cap[upc] && largest <= (long)kPkLeaves * kPkThreads;
  };
  std::vector<char> takes(nb, 0);
  std::vector<std::vector<int>> groups;
  for (int b = 0; b < nb; ++b) {
    if (!fits({b}, most)) continue;
    takes[b] = 1;
    if (!groups.empty()) {
      groups.back().push_back(b);
      if (fits(groups.back(), most)) continue;
      groups.back().pop_back();
    }
    groups.push_back({b});
  }
  if (groups.empty()) return nullptr;
  Persist* P = new (std::nothrow) Persist();
  if (!P) {
    *rc = FE_ERR_OOM;
    return nullptr;
  }
  P->bicg = bicg;
  P->takes = takes;
  std::vector<PkBlock> work;
  long cells = 0;
  for (const std::vector<int>& g : groups) {
    int upc = 1;
    while (!fits(g, upc)) upc *= 2;
    const int first = (int)work.size();
    for (int b : g) {
      const int b0 = (int)work.size();
      for (long q = 0; q < units(b); q += upc)
        work.push_back(PkBlock{b, (int)q, (int)std::min<long>(upc, units(b) - q), b0, cells});
      cells += (long)N[b] * N[b] * N[b];
    }
    P->groups.push_back(PkGroup{first, (int)work.size() - first, upc});
  }
  P->counter_bytes = ((size_t)nb * kPkLine * sizeof(unsigned) + 255) / 256 * 256;
  const size_t wb = (work.size() * sizeof(PkBlock) + 255) / 256 * 256;
  const size_t sb = (work.size() * 4 * sizeof(double) + 255) / 256 * 256;
  const size_t cb = bicg ? (size_t)cells * kPkCoef * sizeof(double) : 0;
  if (cudaMalloc(&P->work, wb + P->counter_bytes + sb + cb) != cudaSuccess) {
    cudaGetLastError();
    P->work = nullptr;
    persist_free(P);
    return nullptr;
  }
  char* base = reinterpret_cast<char*>(P->work) + wb;
  P->counters = reinterpret_cast<unsigned*>(base);
  P->sums = reinterpret_cast<double*>(base + P->counter_bytes);
  P->coef = bicg ? reinterpret_cast<double*>(base + P->counter_bytes + sb) : nullptr;
  if (cudaMemcpyAsync(P->work, work.data(), work.size() * sizeof(PkBlock), cudaMemcpyHostToDevice, st) != cudaSuccess ||
      cudaStreamSynchronize(st) != cudaSuccess) {
    persist_free(P);
    *rc = FE_ERR_CUDA;
    return nullptr;
  }
  return P;
}

// The whole solve of every box that takes one, from K_B into K_X (FP64 fields; psi, D^{-1} and the scalars in place).
int launch_persist(const Launch& L) {
  Persist* P = L.persist;
  if (cudaMemsetAsync(P->counters, 0, P->counter_bytes, L.st) != cudaSuccess) return FE_ERR_CUDA;
  for (const PkGroup& g : P->groups) {
    const BoxDev* boxes = L.boxes;
    PkBlock* work = P->work + g.first;
    void* args[] = {&boxes, &work, &P->sums, &P->counters, &P->coef};
    cudaError_t e = cudaSuccess;
    FE_LAUNCH(L, KID_SOLVE,
              (e = cudaLaunchCooperativeKernel((const void*)pk_kernel(P->bicg, g.upc), dim3(g.blocks),
                                               dim3(kPkThreads), args, 0, L.st)));
    if (e != cudaSuccess) return FE_ERR_CUDA;
  }
  return FE_OK;
}

}  // namespace fe
