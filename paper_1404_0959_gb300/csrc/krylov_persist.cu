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
// Units and sums: unit u of a box is its cells [256 u, 256 u + 256); a block owns
// consecutive units.  Every unit's partial sum is formed by one fixed tree and
// published as a packet, and every block adds the packets of all units of its box
// in the same fixed order, so the sums (and the iterates) of a box do not depend
// on how many blocks it was given, in an ensemble or alone, and no block needs a
// value from a coordinator.
//
// A packet is the two halves of the double, each with the number of the meeting
// (epoch) in its other 32 bits, so that a reader sees whether it has arrived; the
// writer's fence before it orders the vectors that the next phase reads.  Two
// packet sets alternate: a block can be at most one meeting ahead of another.
// The packets are cleared before each launch.  Waits are bounded: a block that
// gives up sets SC_KERR, finishes, and leaves the others to their own limits.
#include <algorithm>
#include <vector>

#include "fe_internal.cuh"

namespace fe {

constexpr int kPkThreads = 256;
constexpr int kPkWarps = kPkThreads / 32;
constexpr int kPkPerSm = 2;     // resident blocks per SM asked for (128 registers)
constexpr int kPkMaxUnits = 8;  // units per block, at most
constexpr int kPkWords = 4;     // words of a packet: two values
constexpr long kPkSpins = 1L << 21;

template <typename T>
__device__ __forceinline__ T* Fp(const BoxDev& B, int slot) {
  return reinterpret_cast<T*>(B.f[slot]);
}
__device__ __forceinline__ void st_packet(unsigned long long* p, unsigned long long v) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ unsigned long long ld_packet(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}

// The meetings of the blocks of one box.
struct Meet {
  unsigned long long* set0;  // packets of the box: [2][units][kPkWords]
  long stride;               // words of one set
  int units, u0, mine;       // units of the box; first one and number of this block
  unsigned epoch = 0;
  bool failed = false;
};

struct MeetShared {
  double val[2][kPkMaxUnits][kPkThreads];
  double warp[2][kPkWarps];
  int bad;
};

// v[k][s]: this thread's share of value k in unit s of the block.  On return tot[k] is the box's sum in
// every thread, and everything the blocks of the box stored to global memory before is visible.
template <int K, int UPC>
__device__ __forceinline__ void meet(Meet& m, MeetShared& sh, const double (&v)[K][UPC], double (&tot)[K]) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  ++m.epoch;
  unsigned long long* set = m.set0 + (m.epoch & 1u) * m.stride;
#pragma unroll
  for (int k = 0; k < K; ++k)
#pragma unroll
    for (int s = 0; s < UPC; ++s) sh.val[k][s][tid] = v[k][s];
  if (tid == 0) sh.bad = 0;
  __syncthreads();
  for (int q = warp; q < K * m.mine; q += kPkWarps) {
    const int k = q % K, s = q / K;
    double a = sh.val[k][s][lane];
#pragma unroll
    for (int j = 1; j < kPkWarps; ++j) a += sh.val[k][s][lane + 32 * j];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) a += __shfl_down_sync(0xffffffffu, a, o);
    if (lane == 0) {
      __threadfence();
      unsigned long long* p = set + (long)(m.u0 + s) * kPkWords + 2 * k;
      const unsigned long long bits = (unsigned long long)__double_as_longlong(a), e = m.epoch;
      st_packet(p, (bits << 32) | e);
      st_packet(p + 1, (bits & 0xffffffff00000000ull) | e);
    }
  }
  double a[K];
#pragma unroll
  for (int k = 0; k < K; ++k) a[k] = 0.0;
  long spins = 0;
  bool bad = m.failed;
  constexpr int AT = 4;  // packets requested at once
  for (int q0 = tid; q0 < m.units; q0 += AT * kPkThreads) {
    unsigned long long w[AT][2 * K];
#pragma unroll
    for (int j = 0; j < AT; ++j)
      if (q0 + j * kPkThreads < m.units) {
        const unsigned long long* p = set + (long)(q0 + j * kPkThreads) * kPkWords;
#pragma unroll
        for (int x = 0; x < 2 * K; ++x) w[j][x] = ld_packet(p + x);
      }
#pragma unroll
    for (int j = 0; j < AT; ++j)
      if (q0 + j * kPkThreads < m.units) {
        const unsigned long long* p = set + (long)(q0 + j * kPkThreads) * kPkWords;
#pragma unroll
        for (int x = 0; x < 2 * K; ++x)
          while ((unsigned)w[j][x] != m.epoch && !bad) {
            w[j][x] = ld_packet(p + x);
            bad = ++spins > kPkSpins;
          }
#pragma unroll
        for (int k = 0; k < K; ++k)
          a[k] += __longlong_as_double((long long)((w[j][2 * k] >> 32) | (w[j][2 * k + 1] & 0xffffffff00000000ull)));
      }
  }
  if (bad) sh.bad = 1;
#pragma unroll
  for (int k = 0; k < K; ++k) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) a[k] += __shfl_down_sync(0xffffffffu, a[k], o);
    if (lane == 0) sh.warp[k][warp] = a[k];
  }
  __syncthreads();
  m.failed = sh.bad != 0;
#pragma unroll
  for (int k = 0; k < K; ++k) {
    double t = sh.warp[k][0];
#pragma unroll
    for (int j = 1; j < kPkWarps; ++j) t += sh.warp[k][j];
    tot[k] = t;
  }
  __syncthreads();
}

// The same without a value: the blocks' stores become visible to each other.
__device__ __forceinline__ void meet_plain(Meet& m, MeetShared& sh) {
  const int tid = threadIdx.x;
  ++m.epoch;
  unsigned long long* set = m.set0 + (m.epoch & 1u) * m.stride;
  if (tid == 0) sh.bad = 0;
  __syncthreads();
  if (tid < m.mine) {
    __threadfence();
    st_packet(set + (long)(m.u0 + tid) * kPkWords, m.epoch);
  }
  long spins = 0;
  bool bad = m.failed;
  for (int q = tid; q < m.units; q += kPkThreads)
    while ((unsigned)ld_packet(set + (long)q * kPkWords) != m.epoch && !bad) bad = ++spins > kPkSpins;
  if (bad) sh.bad = 1;
  __syncthreads();
  m.failed = sh.bad != 0;
  __syncthreads();
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
__global__ void __launch_bounds__(kPkThreads, kPkPerSm) kc_cg(const BoxDev* boxes, const int4* work,
                                                              unsigned long long* packets, long set_stride) {
  __shared__ MeetShared sh;
  const int4 w = work[blockIdx.x];
  const BoxDev& B = boxes[w.x];
  Meet m;
  m.u0 = w.y;
  m.mine = w.z;
  m.set0 = packets + (long)w.w * kPkWords;
  m.stride = set_stride;
  const int N = B.N, n3 = N * N * N;
  m.units = (n3 + kPkThreads - 1) / kPkThreads;
  const double* __restrict__ b = Fp<double>(B, K_B);
  const double* __restrict__ dinv = Fp<double>(B, W_DINV);
  const double* __restrict__ psi = Fp<double>(B, W_PSI);
  double* z = Fp<double>(B, K_AUX);
  double *pa = Fp<double>(B, K_PD), *pb = Fp<double>(B, K_PP);
  const double dt = B.sc[SC_KDT], ih = B.ih, idt = 1.0 / dt, lapc = 0.5 * dt * ih * ih;
  const double tol = B.sc[SC_TOL];
  const int maxit = (int)B.sc[SC_MAXIT];
  const int tid = threadIdx.x;
  double x[UPC], r[UPC], pd[UPC], q[UPC], v1[1][UPC], v2[2][UPC], t1[1], t2[2];
  auto cell = [&](int s) { return (m.u0 + s) * kPkThreads + tid; };
  auto on = [&](int s) { return s < m.mine && cell(s) < n3; };
#pragma unroll
  for (int s = 0; s < UPC; ++s) {
    x[s] = r[s] = pd[s] = q[s] = v2[0][s] = v2[1][s] = v1[0][s] = 0.0;
    if (on(s)) {
      const int c = cell(s);
      r[s] = b[c];
      const double zc = r[s] * dinv[c];
      z[c] = zc;
      v2[0][s] = r[s] * zc;
      v2[1][s] = r[s] * r[s];
    }
  }
  meet<2, UPC>(m, sh, v2, t2);
  double rz = t2[0], rr = t2[1], alpha = 0.0, beta = 0.0;
  const double bb = t2[1];
  int it = 0;
  bool conv = !(bb > 0.0), run = !conv && !m.failed;
  while (run) {
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
      const double pc = it == 0 ? r[s] * dinv[n.c] : fma(beta, pd[s], r[s] * dinv[n.c]);
      const double nb = (dir(n.xm) + dir(n.xp)) + (dir(n.ym) + dir(n.yp)) + (dir(n.zm) + dir(n.zp));
      const double y = psi[n.c] * pc * idt - lapc * (nb - 6.0 * pc);
      pn[n.c] = pc;
      pd[s] = pc;
      q[s] = y;
      v1[0][s] = pc * y;
    }
    meet<1, UPC>(m, sh, v1, t1);
    alpha = rz / t1[0];
#pragma unroll
    for (int s = 0; s < UPC; ++s) {
      if (!on(s)) continue;
      const int c = cell(s);
      x[s] = fma(alpha, pd[s], x[s]);
      r[s] = fma(-alpha, q[s], r[s]);
      const double zc = r[s] * dinv[c];
      z[c] = zc;
      v2[0][s] = r[s] * zc;
      v2[1][s] = r[s] * r[s];
    }
    meet<2, UPC>(m, sh, v2, t2);
    ++it;
    rr = t2[1];
    if (sqrt(rr) <= tol * sqrt(bb)) conv = true, run = false;
    else if (it >= maxit) run = false;
    else {
      beta = t2[0] / rz;
      rz = t2[0];
    }
    run = run && !m.failed;
  }
  double* X = Fp<double>(B, K_X);
#pragma unroll
  for (int s = 0; s < UPC; ++s)
    if (on(s)) X[cell(s)] = x[s];
  if (m.u0 == 0 && tid == 0) {
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
// read the preconditioned vector of the operator (K_PD) and, for the transonic term, psi times it (K_Q);
// the velocity interpolated to the faces is formed once (K_V, K_S, K_T: +1/2 faces along x, y, z).
// x, r (s between the two operators), p, v and t stay in registers; five meetings per iteration.
template <int UPC>
__global__ void __launch_bounds__(kPkThreads, kPkPerSm) kc_bicg(const BoxDev* boxes, const int4* work,
                                                                unsigned long long* packets, long set_stride) {
  __shared__ MeetShared sh;
  const int4 w = work[blockIdx.x];
  const BoxDev& B = boxes[w.x];
  Meet m;
  m.u0 = w.y;
  m.mine = w.z;
  m.set0 = packets + (long)w.w * kPkWords;
  m.stride = set_stride;
  const int N = B.N, NN = N * N, n3 = NN * N;
  m.units = (n3 + kPkThreads - 1) / kPkThreads;
  const bool transonic = B.transonic != 0;
  const double* __restrict__ b = Fp<double>(B, K_B);
  const double* __restrict__ dinv = Fp<double>(B, W_DINV);
  const double* __restrict__ psi = Fp<double>(B, W_PSI);
  double* A1 = Fp<double>(B, K_PD);
  double* A2 = Fp<double>(B, K_Q);
  double* FH[3] = {Fp<double>(B, K_V), Fp<double>(B, K_S), Fp<double>(B, K_T)};
  const double dt = B.sc[SC_KDT], ih = B.ih, idt = 1.0 / dt, lapc = 0.5 * dt * ih * ih, ct = 0.03125 * ih;
  const double tol = B.sc[SC_TOL];
  const int maxit = (int)B.sc[SC_MAXIT];
  const int tid = threadIdx.x;
  double x[UPC], r[UPC], p[UPC], v[UPC], t[UPC], d1[1][UPC], d2[2][UPC], t1[1], t2[2];
  auto cell = [&](int s) { return (m.u0 + s) * kPkThreads + tid; };
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
    const double ps = psi[c], wc = ps * a;
    double nb = 0.0, tr = 0.0;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      int o[4];
      line(c, d, o);
      nb += __ldcg(&A1[o[1]]) + __ldcg(&A1[o[2]]);
      if (transonic) {
        const double m2 = __ldcg(&A2[o[0]]), m1 = __ldcg(&A2[o[1]]), p1 = __ldcg(&A2[o[2]]), p2 = __ldcg(&A2[o[3]]);
        tr += (9.0 * (wc + p1) - (m1 + p2)) * __ldcg(&FH[d][c]) - (9.0 * (m1 + wc) - (m2 + p1)) * __ldcg(&FH[d][o[1]]);
      }
    }
    double y = wc * idt - lapc * (nb - 6.0 * a);
    if (transonic) y += ct * tr;
    return y;
  };
  auto publish = [&](int c, double a) {
    A1[c] = a;
    if (transonic) A2[c] = psi[c] * a;
  };
#pragma unroll
  for (int s = 0; s < UPC; ++s) {
    x[s] = r[s] = p[s] = v[s] = t[s] = d1[0][s] = d2[0][s] = d2[1][s] = 0.0;
    if (on(s)) {
      const int c = cell(s);
      r[s] = b[c];
      d1[0][s] = r[s] * r[s];
      if (transonic) {
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          const double* hb = Fp<double>(B, W_HB0 + d);
          int o[4];
          line(c, d, o);
          FH[d][c] = (9.0 * (hb[c] + hb[o[2]]) - (hb[o[1]] + hb[o[3]])) * 0.0625;
        }
      }
    }
  }
  meet<1, UPC>(m, sh, d1, t1);
  const double bb = t1[0];
  double rho = bb, rho_old = 1.0, alpha = 1.0, omega = 1.0, rr = bb;
  int it = 0;
  bool conv = !(bb > 0.0), run = !conv && !m.failed;
  while (run) {
    const double beta = (rho / rho_old) * (alpha / omega);
#pragma unroll
    for (int s = 0; s < UPC; ++s)
      if (on(s)) {
        p[s] = r[s] + beta * (p[s] - omega * v[s]);
        publish(cell(s), p[s] * dinv[cell(s)]);
      }
    meet_plain(m, sh);
#pragma unroll
    for (int s = 0; s < UPC; ++s)
      if (on(s)) {
        const int c = cell(s);
        v[s] = apply(c, p[s] * dinv[c]);
        d1[0][s] = b[c] * v[s];
      }
    meet<1, UPC>(m, sh, d1, t1);
    alpha = rho / t1[0];
#pragma unroll
    for (int s = 0; s < UPC; ++s)
      if (on(s)) {
        r[s] = r[s] - alpha * v[s];
        publish(cell(s), r[s] * dinv[cell(s)]);
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
    meet<2, UPC>(m, sh, d2, t2);
    omega = t2[0] / t2[1];
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
    meet<2, UPC>(m, sh, d2, t2);
    ++it;
    rr = t2[0];
    rho_old = rho;
    rho = t2[1];
    if (sqrt(rr) <= tol * sqrt(bb)) conv = true, run = false;
    else if (it >= maxit) run = false;
    run = run && !m.failed;
  }
  double* X = Fp<double>(B, K_X);
#pragma unroll
  for (int s = 0; s < UPC; ++s)
    if (on(s)) X[cell(s)] = x[s];
  if (m.u0 == 0 && tid == 0) {
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

typedef void (*PkKernel)(const BoxDev*, const int4*, unsigned long long*, long);
static PkKernel pk_kernel(bool bicg, int upc) {
  if (bicg) return upc == 1 ? kc_bicg<1> : upc == 2 ? kc_bicg<2> : kc_bicg<4>;
  return upc == 1 ? kc_cg<1> : upc == 2 ? kc_cg<2> : upc == 4 ? kc_cg<4> : kc_cg<8>;
}

// Blocks of a context's boxes (box, first unit, units, units of the boxes before); none if they do not
// fit the device at once or it has no cooperative launches.
int persist_plan(const int* N, int nb, int nsm, bool bicg, std::vector<int4>& work, long* units, int* upc) {
  work.clear();
  *units = 0;
  int dev = 0, coop = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess || !coop)
    return 0;
  std::vector<long> u(nb);
  for (int b = 0; b < nb; ++b) {
    u[b] = ((long)N[b] * N[b] * N[b] + kPkThreads - 1) / kPkThreads;
    *units += u[b];
  }
  const int most = bicg ? kPkBicgUnits : kPkMaxUnits;
  for (*upc = 1; *upc <= most; *upc *= 2) {
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, pk_kernel(bicg, *upc), kPkThreads, 0) != cudaSuccess)
      return 0;
    const long cap = (long)std::min(per_sm, kPkPerSm) * nsm;
    long blocks = 0;
    for (int b = 0; b < nb; ++b) blocks += (u[b] + *upc - 1) / *upc;
    if (blocks <= cap) break;
  }
  if (*upc > most) return 0;
  long before = 0;
  for (int b = 0; b < nb; ++b) {
    for (long q = 0; q < u[b]; q += *upc)
      work.push_back(make_int4(b, (int)q, (int)std::min<long>(*upc, u[b] - q), (int)before));
    before += u[b];
  }
  return (int)work.size();
}
size_t persist_packet_bytes(long units) { return (size_t)2 * units * kPkWords * sizeof(unsigned long long); }

// The whole solve of every box from K_B into K_X (FP64 fields; psi, D^{-1} and the scalars in place).
int launch_persist(const Launch& L, bool bicg) {
  if (cudaMemsetAsync(L.packets, 0, persist_packet_bytes(L.punits), L.st) != cudaSuccess) return FE_ERR_CUDA;
  const BoxDev* boxes = L.boxes;
  const int4* work = L.pwork;
  unsigned long long* packets = L.packets;
  long stride = L.punits * kPkWords;
  void* args[] = {&boxes, &work, &packets, &stride};
  cudaError_t e = cudaSuccess;
  FE_LAUNCH(L, KID_SOLVE,
            (e = cudaLaunchCooperativeKernel((const void*)pk_kernel(bicg, L.pupc), dim3(L.npblocks), dim3(kPkThreads),
                                             args, 0, L.st)));
  return e == cudaSuccess ? FE_OK : FE_ERR_CUDA;
}

}  // namespace fe
