// jz_stage_d.cu -- the FP64 fused Runge-Kutta stage kernel: residual
// evaluation and stage update in one pass over HBM.
//
// Paper: arXiv 2003.09926, Section 3 and Section 4.2: per Runge-Kutta
// sub-step, the centred inviscid flux in general curvilinear coordinates, the
// Turkel-Vatsa anisotropic scalar artificial dissipation (pressure sensor,
// five-point stencil, Section 4.3), the viscous flux (Stokes stress, Fourier
// heat flux, Sutherland viscosity) plus a Smagorinsky (or Vreman) eddy
// viscosity, then the update Q^(l) = Q^(0) - alpha_l dt J R(Q^(l-1)) of the
// 5-stage scheme, in face form as in the FP32 kernel (jz_stage_v.cu), whose
// organisation this kernel shares: a CTA marches a TI x TJ tile in k over a
// chunk of planes, TMA stages the planes, one thread per node of the tile and
// its one-node i and j halo forms the node fluxes, faces go through shared
// memory, and what only the thread itself reads again stays in tensor memory.
//
// What bounds it: GB300's FP64 pipe, which passes two lanes per cycle and SM
// (1.25 TFLOP/s); HBM is idle beside it.  So every choice here is about the
// number of FP64 instructions per point:
//  - conserved records beside the primitive ones: the faces difference what is
//    stored instead of forming rho u again at four nodes per face;
//  - twice the face flux, with l2 = 2 lam e2 and l4 = 2 lam e4 formed once per
//    face, and half the time step in the update;
//  - gradients left without their factor J/2, which multiplies the two
//    viscosities instead of twelve gradients;
//  - reciprocals, square roots and J^(-2/3) from the hardware's 20-bit (FP64)
//    or FP32 approximations and one fourth-order step each (4, 7 and 7
//    instructions: 6% of a step less than the library's forms, as precise);
//  - the planes below and above a chunk and its halo nodes there, which only
//    build up the march, form their k quantities only.
// All FP64 arithmetic is written as explicit rounded operations, so that a
// node's values are the same bits whether its thread is a tile or a halo
// thread, in whichever tile, chunk or build.
#include <cmath>
#include <cstdint>

#include "jz_stage_common.cuh"

namespace jz {

using namespace stg;

namespace {

__device__ __forceinline__ double mul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double add(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double sub(double a, double b) { return __dsub_rn(a, b); }

// the larger of two numbers, compared by their bits (an order-preserving map
// to signed integers); a NaN of either sign is larger than any number
__device__ __forceinline__ long long order_bits(double a) {
  const long long x = __double_as_longlong(a);
  return (__double2hiint(a) & 0x7fffffff) > 0x7ff00000 ? 0x7fffffffffffffffLL : x ^ ((x >> 63) & 0x7fffffffffffffffLL);
}
__device__ __forceinline__ double max_bits(double a, double b) { return order_bits(a) > order_bits(b) ? a : b; }

template <int TI_, int TJ_>
struct Cfg {
  static constexpr int TI = TI_, TJ = TJ_;
  static constexpr int NTILE = TI * TJ, NJH = 2 * TI, NIH = 2 * TJ;  // tile, j-halo and i-halo nodes
  static constexpr int NT = NTILE + NJH + NIH;
  static_assert(NTILE % 32 == 0 && NT % 32 == 0, "whole warps of one role");
  static constexpr int RW = TI + 4, RH = TJ + 4, PL = RW * RH;  // staged plane: tile plus two-node halo
  static constexpr int MH = TJ + 2, MPL = RW * MH;              // metric box: rows -1 .. TJ
  static constexpr int UPL = RW * TJ;                           // Q^(0) box: tile rows
  static constexpr int NSQ = 3, NSP = 2;  // ring planes: conserved t+1 .. t+3, primitive t+1, t+2
  static constexpr int GIW = TI + 2, GJH = TJ + 2, HIW = TI + 1, HJH = TJ + 1;
  static constexpr size_t al(size_t x) { return (x + 127) / 128 * 128; }
  static constexpr size_t RAW_B = al(8 * 5 * PL), MET_B = al(8 * 10 * MPL), Q0_B = al(8 * 5 * UPL);
  static constexpr size_t O_RAW = 0;
  static constexpr size_t O_Q = O_RAW + RAW_B;             // conserved ring [slot][v][PL]
  static constexpr size_t O_P = O_Q + al(8 * NSQ * 5 * PL);  // primitive ring (u, v, w, T, p)
  static constexpr size_t O_MET = O_P + al(8 * NSP * 5 * PL);
  static constexpr size_t O_Q0 = O_MET + 2 * MET_B;
  static constexpr size_t O_GI = O_Q0 + Q0_B;              // node fluxes and (lambda~, nu) [v][.]
  static constexpr size_t O_GJ = O_GI + al(8 * 7 * TJ * GIW);
  static constexpr size_t O_HI = O_GJ + al(8 * 7 * GJH * TI);  // face fluxes
  static constexpr size_t O_HJ = O_HI + al(8 * 5 * TJ * HIW);
  static constexpr size_t O_SCR = O_GI;  // a chunk's first three planes are staged over the node and face buffers
  static constexpr size_t O_END = O_HJ + al(8 * 5 * HJH * TI);
  static constexpr size_t O_BAR = O_END > O_SCR + 3 * RAW_B ? O_END : O_SCR + 3 * RAW_B;
  static constexpr size_t O_TMEM = O_BAR + 64;
  static constexpr size_t BYTES = O_BAR + 128;
  static_assert(BYTES <= 232448, "shared memory");
  static constexpr uint32_t RAW_TX = 8 * 5 * PL, MET_TX = 8 * 10 * MPL, Q0_TX = 8 * 5 * UPL;
  // tensor memory, 32-bit columns per warp group: four records of the own
  // column (primitive 5, conserved 5), the march (G^k 5, low k face flux 5,
  // lambda~, nu, J), the own low i and j face fluxes (10); two columns a number
  static constexpr int T_REC = 20, T_MARCH = 4 * T_REC, T_FACE = T_MARCH + 26, T_COLS = T_FACE + 20;
  static constexpr int T_GROUPS = (NT / 32 + 3) / 4;
  static constexpr int T_ALLOC = T_GROUPS * T_COLS <= 128 ? 128 : 512;
  static_assert(T_GROUPS * T_COLS <= T_ALLOC, "tensor memory");
  // CTAs per SM: shared memory (228 KB, 1 KB reserved each) and tensor memory
  static constexpr int MINB_S = (int)(228 * 1024 / (BYTES + 1024 + 64)), MINB_T = 512 / T_ALLOC;
  static constexpr int MINB = MINB_S < MINB_T ? MINB_S : MINB_T;
  static constexpr int B_RAW = 0, B_MET = 4, B_Q0 = 6, NBAR = 7;  // mbarriers (1..3: prologue staging)
};

// N numbers to / from 2 N tensor-memory columns.  Loads are asynchronous:
// issue them, tm_wait_ld, then tie() and combine.
__device__ __forceinline__ void tm_ld4(uint32_t a, uint32_t* r) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a));
}
__device__ __forceinline__ void tm_ld2(uint32_t a, uint32_t* r) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0, %1}, [%2];" : "=r"(r[0]), "=r"(r[1]) : "r"(a));
}
__device__ __forceinline__ void tm_st4(uint32_t a, const uint32_t* r) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(r[0]), "r"(r[1]),
               "r"(r[2]), "r"(r[3]));
}
__device__ __forceinline__ void tm_st2(uint32_t a, const uint32_t* r) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x2.b32 [%0], {%1, %2};" ::"r"(a), "r"(r[0]), "r"(r[1]));
}
template <int N>
struct Words {
  uint32_t w[2 * N];
  __device__ __forceinline__ void load(uint32_t a) {
#pragma unroll
    for (int q = 0; q + 4 <= 2 * N; q += 4) tm_ld4(a + q, w + q);
    if (N % 2) tm_ld2(a + 2 * N - 2, w + 2 * N - 2);
  }
  __device__ __forceinline__ void get(double* r) {  // after the wait
#pragma unroll
    for (int q = 0; q < 2 * N; ++q) asm volatile("" : "+r"(w[q]));
#pragma unroll
    for (int v = 0; v < N; ++v) r[v] = __hiloint2double((int)w[2 * v + 1], (int)w[2 * v]);
  }
  __device__ __forceinline__ void store(uint32_t a, const double* r) {
#pragma unroll
    for (int v = 0; v < N; ++v) {
      w[2 * v] = (uint32_t)__double2loint(r[v]);
      w[2 * v + 1] = (uint32_t)__double2hiint(r[v]);
    }
#pragma unroll
    for (int q = 0; q + 4 <= 2 * N; q += 4) tm_st4(a + q, w + q);
    if (N % 2) tm_st2(a + 2 * N - 2, w + 2 * N - 2);
  }
};
__device__ __forceinline__ void tm_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tm_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
template <class C>
__device__ __forceinline__ void tm_alloc(unsigned char* smem) {
  if (threadIdx.x < 32) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(smem + C::O_TMEM)),
                 "r"(C::T_ALLOC)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  __syncthreads();
}
template <class C>
__device__ __forceinline__ void tm_free(unsigned char* smem) {
  __syncthreads();  // every warp is past its last access
  if (threadIdx.x < 32)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(
                     *reinterpret_cast<volatile uint32_t*>(smem + C::O_TMEM)),
                 "r"(C::T_ALLOC));
}

// flow constants combined once per thread
struct Consts {
  double muc, kpr, kprt;  // mu_inf (1 + S1), Cp / Pr, Cp / Pr_t
};

// Vreman's eddy viscosity (the formula of eddy_nu) from the gradients without
// their factor J/2
__device__ __forceinline__ double vreman_nu(const KConst<double>& c, const double g[4][3], double hJ, double J) {
  double gj[3][3], b[3][3];
#pragma unroll
  for (int q = 0; q < 3; ++q)
#pragma unroll
    for (int m = 0; m < 3; ++m) gj[q][m] = mul(hJ, g[q][m]);
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int d = a; d < 3; ++d)
      b[a][d] = fma(gj[a][2], gj[d][2], fma(gj[a][1], gj[d][1], mul(gj[a][0], gj[d][0])));
  const double aa = add(add(b[0][0], b[1][1]), b[2][2]);
  if (!(aa > 0.0)) return 0.0;
  double B = fma(-b[0][1], b[0][1], mul(b[0][0], b[1][1]));
  B = fma(-b[0][2], b[0][2], fma(b[0][0], b[2][2], B));
  B = fma(-b[1][2], b[1][2], fma(b[1][1], b[2][2], B));
  return mul(mul(mul(2.5, c.cs2), jm23_d(J)), __dsqrt_rn(__ddiv_rn(rmax(B, 0.0), aa)));
}

// A node before its directions: metrics, velocities, viscous flux vectors,
// radii.  pm, pc, pp: primitive records (u, v, w, T, p) of the own column
// below / at / above; P: the plane's primitive ring slot, o the node in it.
template <int MD, int PL, int RW, int MPL>
struct Node {
  double S[9], J, U[3], lam[3], sq[3], Fv[3][4];
  __device__ __forceinline__ void form(const KConst<double>& c, const Consts& k, const double* P, const double* met,
                                       int o, int mo, const double pm[5], const double pc[5], const double pp[5],
                                       double rho) {
#pragma unroll
    for (int f = 0; f < 9; ++f) S[f] = met[f * MPL + mo];
    J = met[9 * MPL + mo];
    const double u = pc[0], v = pc[1], w = pc[2], T = pc[3];
    const double cson = sqrt_d(T);
#pragma unroll
    for (int m = 0; m < 3; ++m)
#pragma unroll
      for (int q = 0; q < 4; ++q) Fv[m][q] = 0.0;
    if (ModelFlags<MD>::viscous(c)) {
      // Cartesian gradients of u, v, w, T without their factor J/2
      double g[4][3];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const double d0 = sub(P[q * PL + o + 1], P[q * PL + o - 1]);
        const double d1 = sub(P[q * PL + o + RW], P[q * PL + o - RW]);
        const double d2 = sub(pp[q], pm[q]);
#pragma unroll
        for (int m = 0; m < 3; ++m) g[q][m] = fma(S[6 + m], d2, fma(S[3 + m], d1, mul(S[m], d0)));
      }
      const double hJ = mul(0.5, J);
      const double mu = mul(mul(k.muc, mul(T, cson)), rcp_d(add(T, c.s1)));  // Sutherland
      const double s01 = add(g[0][1], g[1][0]), s02 = add(g[0][2], g[2][0]), s12 = add(g[1][2], g[2][1]);
      double mu_t = 0.0;
      if (ModelFlags<MD>::sgs(c)) {
        double nu_t;
        if (MD == kModelRuntime && c.vreman) {
          nu_t = vreman_nu(c, g, hJ, J);
        } else {  // Smagorinsky: (C_s Delta)^2 sqrt(2 S_ij S_ij), Delta^2 = J^(-2/3)
          const double dd = fma(g[2][2], g[2][2], fma(g[1][1], g[1][1], mul(g[0][0], g[0][0])));
          const double ss = fma(2.0, dd, fma(s12, s12, fma(s02, s02, mul(s01, s01))));
          nu_t = mul(mul(c.cs2, mul(sqrt_d(ss), hJ)), jm23_d(J));
        }
        mu_t = mul(rho, nu_t);
      }
      const double mue = mul(add(mu, mu_t), hJ), kap = mul(fma(mu_t, k.kprt, mul(mu, k.kpr)), hJ);
      const double div3 = mul(add(add(g[0][0], g[1][1]), g[2][2]), 2.0 / 3.0);
      const double t01 = mul(mue, s01), t02 = mul(mue, s02), t12 = mul(mue, s12);
      Fv[0][0] = mul(mue, fma(2.0, g[0][0], -div3)); Fv[0][1] = t01; Fv[0][2] = t02;
      Fv[1][0] = t01; Fv[1][1] = mul(mue, fma(2.0, g[1][1], -div3)); Fv[1][2] = t12;
      Fv[2][0] = t02; Fv[2][1] = t12; Fv[2][2] = mul(mue, fma(2.0, g[2][2], -div3));
#pragma unroll
      for (int m = 0; m < 3; ++m) Fv[m][3] = fma(kap, g[3][m], fma(w, Fv[m][2], fma(v, Fv[m][1], mul(u, Fv[m][0]))));
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      U[d] = fma(S[3 * d + 2], w, fma(S[3 * d + 1], v, mul(S[3 * d], u)));
      const double s2 = fma(S[3 * d + 2], S[3 * d + 2], fma(S[3 * d + 1], S[3 * d + 1], mul(S[3 * d], S[3 * d])));
      lam[d] = fma(cson, sqrt_d(s2), fabs(U[d]));
      sq[d] = ModelFlags<MD>::sig_half(c) ? sqrt_d(lam[d]) : 0.0;
    }
  }
  // G^d = E^d - F^d, lambda~^d and nu^d of one direction with face vector
  // (Sx, Sy, Sz), contravariant velocity Ud, its radius and the other two's;
  // q the conserved record, p, pm, pp the pressures along the direction
  __device__ __forceinline__ void direction(const KConst<double>& c, double Sx, double Sy, double Sz, double Ud,
                                            double l, double la, double lb, double sl, double sa, double sb,
                                            const double q[5], double p, double pm, double pp, double G[7]) const {
    double F[4];
#pragma unroll
    for (int n = 0; n < 4; ++n) F[n] = fma(Sz, Fv[2][n], fma(Sy, Fv[1][n], mul(Sx, Fv[0][n])));
    G[0] = mul(q[0], Ud);
    G[1] = fma(q[1], Ud, fma(Sx, p, -F[0]));
    G[2] = fma(q[2], Ud, fma(Sy, p, -F[1]));
    G[3] = fma(q[3], Ud, fma(Sz, p, -F[2]));
    G[4] = fma(add(q[4], p), Ud, -F[3]);
    if (ModelFlags<MD>::sig_half(c))  // lambda + sqrt(lambda) (sqrt(la) + sqrt(lb))
      G[5] = fma(sl, add(sa, sb), l);
    else
      G[5] = l > 0.0 ? mul(l, add(add(1.0, pow(la / l, c.sigma)), pow(lb / l, c.sigma))) : 0.0;
    G[6] = mul(fabs(add(fma(-2.0, p, pp), pm)), rcp_d(add(fma(2.0, p, pp), pm)));
  }
};

// twice the dissipative face flux between nodes a and b of a line m, a, b, p:
// 2h = Ga + Gb - 2 lam [e2 (qb - qa) - e4 (qp - 3 qb + 3 qa - qm)]; Ga, Gb hold
// (G 5, lambda~, nu)
__device__ __forceinline__ void face_d(const KConst<double>& c, const double Ga[7], const double Gb[7],
                                       const double qm[5], const double qa[5], const double qb[5], const double qp[5],
                                       double h[5]) {
  const double lam = add(Ga[5], Gb[5]);
  const double e2 = mul(c.k2, max_bits(Ga[6], Gb[6]));
  const double e4 = sub(c.k4, e2);
  const double l2 = mul(lam, e2), l4 = __double2hiint(e4) < 0 ? 0.0 : mul(lam, e4);
#pragma unroll
  for (int v = 0; v < 5; ++v) {
    const double d1 = sub(qb[v], qa[v]);
    const double d3 = fma(-3.0, d1, sub(qp[v], qm[v]));
    // only the last rounding at the size of the sum (added to Ga + Gb, the two
    // parts of the dissipation rounded there as well: a step's momenta erred by
    // 0.5% more)
    h[v] = add(fma(-l2, d1, Ga[v]), fma(l4, d3, Gb[v]));
  }
}

// One work item: tile (bx, by), k-chunk bz of grid X, stage st, for the tile
// threads (ROLE 0) or the halo threads (ROLE 1: rows -1 and TJ, columns -1 and
// TI, one direction each).  On a bounded-wait timeout the item records where
// it gave up, lets its copies in flight land and returns false.
template <class C, int MD, int ROLE>
__device__ __forceinline__ bool item_d(const StageCtx<double, double>& X, const StageSel& st, int bx, int by, int bz,
                                       unsigned char* smem, bool first) {
  constexpr int TI = C::TI, TJ = C::TJ, RW = C::RW, PL = C::PL, MPL = C::MPL;
  double* const raw = reinterpret_cast<double*>(smem + C::O_RAW);
  double* const Qr = reinterpret_cast<double*>(smem + C::O_Q);
  double* const Pr = reinterpret_cast<double*>(smem + C::O_P);
  double* const Gi = reinterpret_cast<double*>(smem + C::O_GI);
  double* const Gj = reinterpret_cast<double*>(smem + C::O_GJ);
  double* const Hi = reinterpret_cast<double*>(smem + C::O_HI);
  double* const Hj = reinterpret_cast<double*>(smem + C::O_HJ);
  uint64_t* const bar = reinterpret_cast<uint64_t*>(smem + C::O_BAR);
  const Layout& L = X.L;
  const KConst<double> c = X.k;
  const int tid = threadIdx.x;
  const int i0 = bx * TI, j0 = by * TJ;
  const int t0 = L.lo[2] + bz * X.kc, t1 = min(t0 + X.kc, L.hi[2] + 1);
  const uint32_t xtx = st.stall ? kStallBytes : 0u;
  const long long wlim = st.stall ? kStallLimit : kWaitLimit;

  int nx, ny;
  bool dj = false;  // halo thread of the j direction
  if constexpr (ROLE == 0) {
    nx = tid % TI;
    ny = tid / TI;
  } else {
    const int h = tid - C::NTILE;
    dj = h < C::NJH;
    nx = dj ? h % TI : (((h - C::NJH) / TJ) ? TI : -1);
    ny = dj ? ((h / TI) ? TJ : -1) : (h - C::NJH) % TJ;
  }
  const int gi = i0 + nx, gj = j0 + ny;
  const bool own = ROLE == 0 && gi >= L.lo[0] && gi <= L.hi[0] && gj >= L.lo[1] && gj <= L.hi[1];

  __syncthreads();
  if (tid == 0) {
    for (int b = 0; b < C::NBAR; ++b) {
      if (!first) asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(smem_addr(&bar[b])) : "memory");
      mbar_init(&bar[b], 1);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  fence_async_shared();  // generic-proxy writes to the buffers the prologue stages into, then the barrier
  __syncthreads();

  // thread 0's record of its copies: bit b of pend = barrier b has had one,
  // bit b of ppar = the parity of the last one's phase
  uint32_t pend = 0, ppar = 0;
  auto begin_copy = [&](int b, uint32_t parity, uint32_t bytes) {
    pend |= 1u << b;
    ppar = (ppar & ~(1u << b)) | (parity << b);
    fence_async_shared();
    mbar_expect_tx(&bar[b], bytes + xtx);
  };
  auto issue_raw = [&](int p, int b, void* dst, uint32_t parity) {
    if (ROLE == 0 && tid == 0) {
      begin_copy(b, parity, C::RAW_TX);
      tma_load_4d(dst, &X.tmQ[st.qin], &bar[b], i0, j0, p + NG, 0);
    }
  };
  auto raw_parity = [&](int p) { return (uint32_t)((p - t0 - 1) & 1); };
  auto met_sel = [&](int p) { return (p - t0 + 1) & 1; };
  auto met_parity = [&](int p) { return (uint32_t)(((p - t0 + 1) >> 1) & 1); };
  auto met_buf = [&](int p) { return reinterpret_cast<double*>(smem + C::O_MET + met_sel(p) * C::MET_B); };
  auto issue_met = [&](int p) {
    if (ROLE == 0 && tid == 0) {
      const int b = C::B_MET + met_sel(p);
      begin_copy(b, met_parity(p), C::MET_TX);
      tma_load_4d(met_buf(p), &X.tmMv, &bar[b], i0, j0 + 1, p + NG, 0);
    }
  };
  const bool q0_own = st.qin == 0;  // the first stage's Q^(0) is its input
  auto issue_q0 = [&](int p) {
    if (ROLE == 0 && tid == 0 && !q0_own) {
      begin_copy(C::B_Q0, (uint32_t)((p - t0) & 1), C::Q0_TX);
      tma_load_4d(smem + C::O_Q0, &X.tmQ0u, &bar[C::B_Q0], i0, j0 + 2, p + NG, 0);
    }
  };
  bool ok = true;
  auto wait = [&](int b, uint32_t parity, int p) {
    if (mbar_try_wait(&bar[b], parity) || mbar_wait_bounded(&bar[b], parity, wlim)) return;
    ok = false;
    if (ROLE == 0 && tid == 0 && atomicCAS(X.err, 0, 1) == 0) {
      int* info = X.err + 1;
      info[0] = b; info[1] = (int)parity; info[2] = p; info[3] = bx; info[4] = by; info[5] = bz; info[6] = st.qin;
    }
  };

  const int oo = (ny + 2) * RW + nx + 2;  // this thread's node in a staged or ring plane
  const int mo = (ny + 1) * RW + nx + 2;  // ... in the metric box
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
  const uint32_t tm = __shfl_sync(0xffffffffu, *reinterpret_cast<volatile uint32_t*>(smem + C::O_TMEM), 0) +
                      ((uint32_t)(warp & 3) << 21) + (uint32_t)((warp >> 2) * C::T_COLS);

  // records of a staged plane: every thread its own node (which also goes to
  // tensor memory), halo threads the next node outwards too, four of them the
  // corners of the one-node halo
  auto convert = [&](const double* src, int sq, int sp, int rec) {
    int e = oo;
    constexpr int NC = ROLE == 0 ? 1 : 3;
    bool on = true;
#pragma unroll 1
    for (int b = 0; b < NC; ++b) {
      double r[10];
      if (on) {
#pragma unroll
        for (int v = 0; v < 5; ++v) r[5 + v] = src[v * PL + e];
        const double ri = rcp_d(r[5]);
#pragma unroll
        for (int m = 0; m < 3; ++m) r[m] = mul(r[6 + m], ri);
        const double k2 = fma(r[2], r[8], fma(r[1], r[7], mul(r[0], r[6])));  // rho |u|^2
        r[4] = mul(c.gm1, fma(-0.5, k2, r[9]));
        r[3] = mul(mul(c.gamma, r[4]), ri);
#pragma unroll
        for (int v = 0; v < 5; ++v) {
          Qr[(sq * 5 + v) * PL + e] = r[5 + v];
          Pr[(sp * 5 + v) * PL + e] = r[v];
        }
      }
      if (b == 0) {
        __syncwarp();
        Words<10> w;
        w.store(tm + rec, r);
      }
      if constexpr (ROLE == 1) {
        if (b == 0) {
          e += dj ? (ny < 0 ? -RW : RW) : (nx < 0 ? -1 : 1);
        } else {
          const int h = tid - C::NTILE;
          on = h < 4;
          e = ((h & 2) ? TJ + 2 : 1) * RW + ((h & 1) ? TI + 2 : 1);
        }
      }
    }
  };

  Consts k;
  k.muc = mul(c.mu_inf, c.s1p1);
  k.kpr = mul(c.cp, c.inv_pr);
  k.kprt = mul(c.cp, c.inv_prt);
  const double hadt = mul(0.5, mul(st.alpha, X.sc->dt));  // half: the residual is formed of twice the face fluxes
  const long long npad = L.npad;
  double* const Qo = X.Q[st.qout];
  const double* const q0buf = reinterpret_cast<const double*>(smem + C::O_Q0);
  const long long n_t0 = own ? L.at(gi, gj, t0) : 0;
  unsigned char* const scr = smem + C::O_SCR;

  issue_raw(t0 - 2, 1, scr, 0);
  issue_raw(t0 - 1, 2, scr + C::RAW_B, 0);
  issue_raw(t0, 3, scr + 2 * C::RAW_B, 0);
  issue_met(t0 - 1);
  issue_raw(t0 + 1, C::B_RAW, raw, 0);
  issue_met(t0);
#pragma unroll 1
  for (int q = 0; q < 3; ++q) {
    wait(1 + q, 0, t0 - 2 + q);
    convert(reinterpret_cast<const double*>(scr + q * C::RAW_B), q, (q + 1) & 1, q * C::T_REC);
  }
  __syncwarp();
  tm_wait_st();
  if (__syncthreads_or(!ok)) goto fail;

  {
    // node data from the node pass to the face pass: (G 5, lambda~, nu) of the
    // own faces' directions (a halo thread has one)
    double Wi[7], Wj[7];
    const bool do_i = ROLE == 0 || (!dj && nx == TI);
    const bool do_j = ROLE == 0 || (dj && ny == TJ);
    int r0 = 0, r1 = 1, r2 = 2, k0 = 0;  // conserved ring slots of planes t, t+1, t+2; record of plane t
#pragma unroll 1
    for (int t = t0 - 2; t < t1; ++t) {
      const bool live = t + 1 >= t0 && t + 1 < t1;  // plane t+1 is updated
      const int sp1 = (t - t0) & 1;                 // primitive slot of plane t+1
      const int k1 = (k0 + 1) & 3, k2 = (k0 + 2) & 3, k3 = (k0 + 3) & 3;
      double qb[5], Gk[7], Jn = 0.0;
      wait(C::B_MET + met_sel(t + 1), met_parity(t + 1), t + 1);
      __syncwarp();
      {
        double pb[5], pt[5], pn[5];
        Words<5> a, d, e;
        Words<5> f;
        a.load(tm + k0 * C::T_REC);
        d.load(tm + k1 * C::T_REC);
        f.load(tm + k1 * C::T_REC + 10);
        e.load(tm + k2 * C::T_REC);
        tm_wait_ld();
        a.get(pb);
        d.get(pt);
        f.get(qb);
        e.get(pn);
        if (ROLE == 0 || live) {
          const double* const P = Pr + sp1 * 5 * PL;
          Node<MD, PL, RW, MPL> nd;
          nd.form(c, k, P, met_buf(t + 1), oo, mo, pb, pt, pn, qb[0]);
          const double* const pp4 = P + 4 * PL + oo;
          const double* S = nd.S;
          if constexpr (ROLE == 0) {
            Jn = nd.J;
            nd.direction(c, S[6], S[7], S[8], nd.U[2], nd.lam[2], nd.lam[0], nd.lam[1], nd.sq[2], nd.sq[0], nd.sq[1], qb,
                         pt[4], pb[4], pn[4], Gk);
            if (live) {
              nd.direction(c, S[0], S[1], S[2], nd.U[0], nd.lam[0], nd.lam[1], nd.lam[2], nd.sq[0], nd.sq[1], nd.sq[2],
                           qb, pt[4], pp4[-1], pp4[1], Wi);
              nd.direction(c, S[3], S[4], S[5], nd.U[1], nd.lam[1], nd.lam[2], nd.lam[0], nd.sq[1], nd.sq[2], nd.sq[0],
                           qb, pt[4], pp4[-RW], pp4[RW], Wj);
            }
          } else {  // one direction, chosen by the thread
            const int st1 = dj ? RW : 1;
            const double Sx = dj ? S[3] : S[0], Sy = dj ? S[4] : S[1], Sz = dj ? S[5] : S[2];
            nd.direction(c, Sx, Sy, Sz, dj ? nd.U[1] : nd.U[0], dj ? nd.lam[1] : nd.lam[0], dj ? nd.lam[2] : nd.lam[1],
                         dj ? nd.lam[0] : nd.lam[2], dj ? nd.sq[1] : nd.sq[0], dj ? nd.sq[2] : nd.sq[1],
                         dj ? nd.sq[0] : nd.sq[2], qb, pt[4], pp4[-st1], pp4[st1], Wi);
          }
        }
        if (live) {
          if (ROLE == 0 || !dj)
#pragma unroll
            for (int v = 0; v < 7; ++v) Gi[(v * TJ + ny) * C::GIW + nx + 1] = Wi[v];
          if (ROLE == 0 || dj)
#pragma unroll
            for (int v = 0; v < 7; ++v) Gj[(v * C::GJH + ny + 1) * TI + nx] = ROLE == 0 ? Wj[v] : Wi[v];
        }
      }
      if (!q0_own && t >= t0) wait(C::B_Q0, (uint32_t)((t - t0) & 1), t);
      if constexpr (ROLE == 0) {
        double mv[13], hl[10], qc[5], qd[5], qp[5], hk[5];
        __syncwarp();
        {
          Words<13> a;
          Words<5> b, d, e;
          Words<10> f;
          a.load(tm + C::T_MARCH);
          b.load(tm + k3 * C::T_REC + 10);  // plane t-1
          d.load(tm + k0 * C::T_REC + 10);
          e.load(tm + k2 * C::T_REC + 10);
          f.load(tm + C::T_FACE);
          tm_wait_ld();
          a.get(mv);
          b.get(qc);
          d.get(qd);
          e.get(qp);
          f.get(hl);
        }
        double Ga[7];
#pragma unroll
        for (int v = 0; v < 5; ++v) Ga[v] = mv[v];
        Ga[5] = mv[10];
        Ga[6] = mv[11];
        if (t >= t0 - 1) {
          face_d(c, Ga, Gk, qc, qd, qb, qp, hk);
        } else {
#pragma unroll
          for (int v = 0; v < 5; ++v) hk[v] = 0.0;
        }
        {
          double nv[13];
#pragma unroll
          for (int v = 0; v < 5; ++v) {
            nv[v] = Gk[v];
            nv[5 + v] = hk[v];
          }
          nv[10] = Gk[5];
          nv[11] = Gk[6];
          nv[12] = Jn;
          __syncwarp();
          Words<13> a;
          a.store(tm + C::T_MARCH, nv);
        }
        if (own && t >= t0) {
          const double aj = -mul(hadt, mv[12]);
          double* const dst = Qo + n_t0 + (long long)(t - t0) * L.plane;
#pragma unroll
          for (int v = 0; v < 5; ++v) {
            const double di = sub(Hi[(v * TJ + ny) * C::HIW + nx + 1], hl[v]);
            const double djv = sub(Hj[(v * C::HJH + ny + 1) * TI + nx], hl[5 + v]);
            const double q0 = q0_own ? qd[v] : q0buf[v * C::UPL + ny * RW + nx + 2];
            dst[v * npad] = fma(aj, add(add(di, djv), sub(hk[v], mv[5 + v])), q0);
          }
        }
      }
      __syncwarp();
      tm_wait_st();
      if (__syncthreads_or(!ok)) goto fail;
      if (t + 3 <= t1) issue_met(t + 3);
      if (live) {
        issue_q0(t + 1);
        const double* const Q = Qr + r1 * 5 * PL + oo;
        double qo[5], hij[10];
        __syncwarp();
        {
          Words<5> a;
          a.load(tm + k1 * C::T_REC + 10);
          tm_wait_ld();
          a.get(qo);
        }
        auto face = [&](const double* G, int gs, int step, const double W[7], double h[5]) {
          double Ga[7], qm[5], qa[5], qp[5];
#pragma unroll
          for (int v = 0; v < 7; ++v) Ga[v] = G[v * gs];
#pragma unroll
          for (int v = 0; v < 5; ++v) {
            qm[v] = Q[v * PL - 2 * step];
            qa[v] = Q[v * PL - step];
            qp[v] = Q[v * PL + step];
          }
          face_d(c, Ga, W, qm, qa, qo, qp, h);
        };
        if (do_i) {
          face(Gi + ny * C::GIW + nx, TJ * C::GIW, 1, Wi, hij);
#pragma unroll
          for (int v = 0; v < 5; ++v) Hi[(v * TJ + ny) * C::HIW + nx] = hij[v];
        }
        if (do_j) {
          face(Gj + ny * TI + nx, C::GJH * TI, RW, ROLE == 0 ? Wj : Wi, hij + 5);
#pragma unroll
          for (int v = 0; v < 5; ++v) Hj[(v * C::HJH + ny) * TI + nx] = hij[5 + v];
        }
        if constexpr (ROLE == 0) {
          __syncwarp();
          Words<10> a;
          a.store(tm + C::T_FACE, hij);
        }
      }
      if (t + 3 <= t1 + 1) {
        wait(C::B_RAW, raw_parity(t + 3), t + 3);
        convert(raw, r0, sp1, k3 * C::T_REC);
      }
      __syncwarp();
      tm_wait_st();
      if (__syncthreads_or(!ok)) goto fail;
      if (t + 4 <= t1 + 1) issue_raw(t + 4, C::B_RAW, raw, raw_parity(t + 4));
      const int r = r0;
      r0 = r1;
      r1 = r2;
      r2 = r;
      k0 = k1;
    }
  }
  return true;

fail:
  // let this item's copies in flight land before the shared memory is reused
  if (tid == 0) {
    atomicExch(X.err, 1);
    for (int b = 0; b < C::NBAR; ++b)
      if (pend & (1u << b)) {
        if (xtx) mbar_complete_tx(&bar[b], xtx);
        mbar_wait_bounded(&bar[b], (ppar >> b) & 1u);
      }
  }
  __syncthreads();
  return false;
}

template <class C, int MD>
__global__ void __launch_bounds__(C::NT, C::MINB)
    k_stage_d(const __grid_constant__ StageCtx<double, double> X, const StageSel st) {
  extern __shared__ __align__(128) unsigned char smem[];
  tm_alloc<C>(smem);
  wait_for_previous();
  if (threadIdx.x < C::NTILE)
    item_d<C, MD, 0>(X, st, blockIdx.x, blockIdx.y, blockIdx.z, smem, true);
  else
    item_d<C, MD, 1>(X, st, blockIdx.x, blockIdx.y, blockIdx.z, smem, true);
  tm_free<C>(smem);
}

template <class C, int MD>
__global__ void __launch_bounds__(C::NT, C::MINB)
    k_stage_d_batch(const StageCtx<double, double>* __restrict__ ctx, const int4* __restrict__ items, int nitems,
                    unsigned int* queue, const StageSel st) {
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ int next;
  bool first = true;
  tm_alloc<C>(smem);
  for (;;) {
    if (threadIdx.x == 0) next = (int)atomicAdd(queue, 1u);
    __syncthreads();
    const int it = next;
    __syncthreads();
    if (it >= nitems) break;
    const int4 w = items[it];
    const bool ok = threadIdx.x < C::NTILE ? item_d<C, MD, 0>(ctx[w.x], st, w.y, w.z, w.w, smem, first)
                                           : item_d<C, MD, 1>(ctx[w.x], st, w.y, w.z, w.w, smem, first);
    if (!ok) break;
    first = false;
  }
  tm_free<C>(smem);
}

// Tiles: 16 x 16 (one CTA per SM) costs 15.2 FP64 warp instructions per node
// and plane, halo included; 8 x 8 (three CTAs) 17.3, but cuts a small grid
// into enough CTAs for the whole chip.
using Big = Cfg<16, 16>;
using Small = Cfg<8, 8>;

template <class C, int MD>
cudaError_t configure() {
  const cudaFuncAttribute a = cudaFuncAttributeMaxDynamicSharedMemorySize;
  cudaError_t e = cudaFuncSetAttribute(k_stage_d<C, MD>, a, (int)C::BYTES);
  if constexpr (C::TI == 16) {  // batches run 16 x 16 tiles
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_stage_d_batch<C, MD>, a, (int)C::BYTES);
  }
  return e;
}

template <class C, int MD>
cudaError_t launch(const StageCtx<double, double>& X, const StageSel& st, cudaStream_t s) {
  const Layout& L = X.L;
  const int nz = L.hi[2] - L.lo[2] + 1;
  const dim3 grid((L.hi[0] + C::TI) / C::TI, (L.hi[1] + C::TJ) / C::TJ, (nz + X.kc - 1) / X.kc);
  count_launches(1);
  return launch_dep(k_stage_d<C, MD>, grid, C::NT, C::BYTES, s, X, st);
}

template <class C, int MD>
cudaError_t launch_batch(const void* ctx, const int4* items, int nitems, unsigned int* queue, const StageSel& st,
                         cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(queue, 0, sizeof(unsigned int), s);
  if (e != cudaSuccess) return e;
  const int slots = device_sm_count() * C::MINB;
  const int ctas = nitems < slots ? nitems : slots;
  k_stage_d_batch<C, MD><<<ctas, C::NT, C::BYTES, s>>>((const StageCtx<double, double>*)ctx, items, nitems, queue, st);
  count_launches(1);
  return cudaGetLastError();
}

}  // namespace

cudaError_t stage_d_configure() {
  cudaError_t e;
  if ((e = configure<Small, kModelSmagorinsky>()) != cudaSuccess) return e;
  if ((e = configure<Small, kModelRuntime>()) != cudaSuccess) return e;
  if ((e = configure<Big, kModelSmagorinsky>()) != cudaSuccess) return e;
  return configure<Big, kModelRuntime>();
}

int stage_d_ctas_per_sm(StageTiling t) { return t.ti == Small::TI ? Small::MINB : Big::MINB; }

// The tile and k-chunk length of a grid: the split with the least modelled time
// (microseconds, fitted to measured stages).
//   16 x 16: the CTAs of an SM run one after the other, a chunk of kc planes
//     takes 33.8 kc + 45 (45: its prologue and the two planes that build up the
//     march), the FP64 pipe 92% busy.
//   8 x 8: only while all CTAs are resident together; a plane takes
//     9.5 + 7 c for c CTAs per SM and 15.6 at least (one CTA's three warps
//     wait for one another's results half of the time).
// (Fitted before the reciprocals and square roots took another instruction or
// two; both tiles are 5% slower since.)  Measured, us per stage: 48x32x32, 8 x 8
// with chunks of 2 planes (chosen) 104, of 3 98, of 5 114, 16 x 16 with chunks of 2
// 121; 77x42x54, 16 x 16 with chunks of 6 (chosen) 263, 8 x 8 277 at best;
// 56x36x30, 8 x 8 with chunks of 4 (chosen) 120, 16 x 16 156.
void stage_d_split(const Layout& L, StageTiling& t, int& kc) {
  const int nz = L.hi[2] - L.lo[2] + 1;
  const long long sms = device_sm_count();
  auto tiles = [&](int n) { return (long long)((L.hi[0] + n) / n) * ((L.hi[1] + n) / n); };
  const long long big = tiles(Big::TI), small = tiles(Small::TI);
  double best = 1e300;
  auto take = [&](double cost, int n, int k) {
    if (cost >= best * (1.0 - 1e-9)) return;
    best = cost;
    t = {n, n};
    kc = k;
  };
  for (int k = 1; k <= nz; ++k) {
    const int chunks = (nz + k - 1) / k;
    take((double)((big * chunks + sms - 1) / sms) * (33.8 * k + 45.0), Big::TI, k);
    const double c = (double)(small * chunks) / (double)sms;
    if (small * chunks <= sms * Small::MINB) take(std::fmax(15.6, 9.5 + 7.0 * c) * (k + 1.7) + 8.0, Small::TI, k);
  }
}

cudaError_t launch_stage_d(const StageCtx<double, double>& X, const StageSel& st, StageTiling t, cudaStream_t s) {
  if (t.ti == Small::TI)
    return flow_model(X.k) == kModelSmagorinsky ? launch<Small, kModelSmagorinsky>(X, st, s)
                                                : launch<Small, kModelRuntime>(X, st, s);
  return flow_model(X.k) == kModelSmagorinsky ? launch<Big, kModelSmagorinsky>(X, st, s)
                                              : launch<Big, kModelRuntime>(X, st, s);
}

cudaError_t launch_stage_d_batch(const void* ctx, const int4* items, int nitems, unsigned int* queue,
                                 const StageSel& st, int model, cudaStream_t s) {
  return model == kModelSmagorinsky ? launch_batch<Big, kModelSmagorinsky>(ctx, items, nitems, queue, st, s)
                                    : launch_batch<Big, kModelRuntime>(ctx, items, nitems, queue, st, s);
}

}  // namespace jz
