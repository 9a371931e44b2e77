// jz_stage_v.cu -- the FP32 fused Runge-Kutta stage kernel with vector node
// records: residual evaluation and stage update in one pass over HBM.
//
// Paper: arXiv 2003.09926, Section 3 and Section 4.2: per Runge-Kutta
// sub-step, the centred inviscid flux in general curvilinear coordinates, the
// Turkel-Vatsa anisotropic scalar artificial dissipation (pressure sensor,
// five-point stencil, Section 4.3), the viscous flux (Stokes stress, Fourier
// heat flux, Sutherland viscosity) plus a Smagorinsky (or Vreman) eddy viscosity, then
// the update Q^(l) = Q^(0) - alpha_l dt J R(Q^(l-1)) of the 5-stage scheme.
// The residual is taken in face form, R_n = sum_k (h^k_{n+1/2} - h^k_{n-1/2})
// with h_{n+1/2} = (G_n + G_{n+1})/2 - d_{n+1/2}, G = E - F the contravariant
// inviscid minus viscous flux: the paper's central difference plus
// dissipation, telescoping exactly.
//
// Organisation (2.5-D streaming over a TI x TJ (i, j) tile and a chunk of
// k-planes; the file is compiled once per tile shape the autotuner chooses
// from: 16 x 16 (the default, two CTAs per SM), 32 x 16 and 16 x 32 (one CTA
// per SM), VR_TI / VR_TJ, and its entry points carry the shape in their
// names; within a shape, once per flow model with the model's flags as
// constants plus once with the flags read at run time, and within a build
// once per node role):
//  - TMA stages the conserved variables of one plane (tile plus a two-node
//    halo) into a planar buffer, and the metric fields of two planes (tile
//    plus a one-node halo) into two buffers; waits are bounded;
//  - each staged plane is converted once into two rings of node records:
//    conserved (rho, rho u, rho v, rho w | e) over three planes and primitive
//    (u, v, w, T | p) over two, each a float4 plus a float, so that a
//    neighbour's stencil values arrive with two shared-memory loads;
//  - one thread per node of the plus-shaped set (tile nodes plus the
//    one-node i and j halo) forms G^k, the dissipation radius lambda~^k and
//    the sensor nu^k of its node (tile threads in all three directions, halo
//    threads in their own direction);
//  - i and j face fluxes go through shared memory as float4 + float records;
//  - what only the thread itself reads again -- the records of its own column
//    (planes t-1 .. t+3), the state of its k march, its own low face fluxes --
//    is kept in tensor memory (tcgen05.ld / st), whose four lane quadrants
//    together move four times the bytes per cycle of shared memory;
//  - two block barriers per plane: node pass of plane t+1, k face, i/j
//    residual and update of plane t | i/j face fluxes of plane t+1 and the
//    conversion of the plane three ahead;
//  - one loop body serves the whole chunk, the two planes that build up the
//    k march included.
//
// What bounds it.  With the column in a shared-memory ring and a prologue of
// its own, the kernel moved 7.8 shared-memory wavefronts per point through a
// pipe 67% busy and stalled 0.9 cycles per instruction on instruction fetch
// (103 KB of code for the three roles).  The column in tensor memory took the
// wavefronts to 6.0, and the single loop body the code to 42 KB, the fetch
// stalls to 0.2 and the issue rate from 53% to 66%: 1.98 to 1.72 ms per step
// on 256x192x192.  Tensor memory alone, with the old code size, gained 1%: the
// fetch stalls rose by what the memory stalls fell.  Block barriers without a
// reduction and the set-up before the previous kernel's end took the step to
// 1.69 ms (a stage 0.361 to 0.302 ms).  Now issue slots (66%) and the shared-memory
// pipe (64%) bind together, with the barriers between.
#include <cmath>
#include <cstdint>

#include "jz_stage_common.cuh"

#ifndef VR_TI
#define VR_TI 32
#define VR_TJ 16
#endif
// face fluxes, node gradients and contravariant viscous fluxes on packed
// FP32x2 component pairs
#ifndef VR_PACKED_FACES
#define VR_PACKED_FACES 1
#endif
#define VR_CAT3(a, b, c) a##_##b##x##c
#define VR_CAT(a, b, c) VR_CAT3(a, b, c)
#define VR_FN(name) VR_CAT(name, VR_TI, VR_TJ)

namespace jz {

using namespace stg;

namespace {

namespace vr {
constexpr int TI = VR_TI, TJ = VR_TJ;
constexpr int MINB = vr_ctas_per_sm(TI, TJ);    // CTAs per SM
constexpr int NTILE = TI * TJ;                  // tile nodes
constexpr int NJH = 2 * TI, NIH = 2 * TJ;       // j-halo (rows -1, TJ) and i-halo (columns -1, TI) nodes
constexpr int NT = NTILE + NJH + NIH;           // threads (608 for 32 x 16 and 16 x 32)
static_assert(NT % 32 == 0, "whole warps");
constexpr int RW = TI + 4, RH = TJ + 4, PL = RW * RH;  // staged plane: tile + two-node halo (36 x 20)
constexpr int MH = TJ + 2, MPL = RW * MH;        // metric box: rows -1 .. TJ, 36 columns
// Warp layout of the tile threads.  A warp holds 32 nodes: a full row of a
// 32-wide tile, or two rows of a 16-wide tile.  In the 16 x 16 build the two
// rows of a warp are r and r + 4 (warps 0-3: rows 0-3 and 4-7, warps 4-7:
// rows 8-11 and 12-15), and every per-row buffer has a row stride of 20
// words, so the two half-warps of a scalar shared-memory access sit 80 = 16
// (mod 32) banks apart and never conflict.
constexpr bool ROWS4 = TI == 16 && TJ == 16;
// ring records: rows padded to 37 so that the column-wise accesses of the
// i-halo warp fall on distinct banks (unpadded rows of 20 in the 16 x 16
// build, for the warp layout above)
constexpr int RR = ROWS4 ? RW : RW + 1, RPL = RR * RH;
// ring depths (planes): conserved records 3 (plane t + 1 for the faces, t + 2
// for the own column's next record, t + 3 being converted), primitive
// records 2 (the node pass of plane t + 1 reads planes t + 1 and, of its own
// column, t + 2; t + 3 is converted after it)
constexpr int NSQ = 3, NSP = 2;
// node buffers: columns -1..TI / rows -1..TJ; face buffers: i faces 0..TI /
// j faces 0..TJ.  The i-direction rows are padded (distinct banks for the
// i-halo warp's column accesses; a stride of 20 in the 16 x 16 build).
constexpr int GIW = ROWS4 ? TI + 4 : TI + 3, GJH = TJ + 2;
constexpr int HIW = ROWS4 ? TI + 4 : TI + 3, HJH = TJ + 1;
constexpr size_t al(size_t x) { return (x + 127) / 128 * 128; }
constexpr size_t RAW_B = al(4 * 5 * PL);
constexpr size_t QV_B = al(16 * NSQ * RPL), QE_B = al(4 * NSQ * RPL);
constexpr size_t PV_B = al(16 * NSP * RPL), PP_B = al(4 * NSP * RPL);
constexpr size_t MET_B = al(4 * 10 * MPL);       // one plane; two are staged
constexpr int UPL = RW * TJ;                     // Q^(0) box: tile rows, 36 columns
constexpr size_t Q0_B = al(4 * 5 * UPL);
constexpr size_t GI4_B = al(16 * TJ * GIW), GI1_B = al(4 * TJ * GIW);
// the scalar part of the j-direction records: rows of 20 in the 16 x 16 build
// (the float4 / float2 parts are conflict-free at any row stride)
constexpr int JS1 = ROWS4 ? TI + 4 : TI;
constexpr size_t GJ4_B = al(16 * GJH * TI), GJ1_B = al(4 * GJH * JS1);
constexpr size_t LI_B = al(8 * TJ * GIW), LJ_B = al(8 * GJH * TI);
constexpr size_t HI4_B = al(16 * TJ * HIW), HI1_B = al(4 * TJ * HIW);
constexpr size_t HJ4_B = al(16 * HJH * TI), HJ1_B = al(4 * HJH * JS1);
constexpr size_t O_RAW = 0;
constexpr size_t O_QV = O_RAW + RAW_B;
constexpr size_t O_QE = O_QV + QV_B;
constexpr size_t O_PV = O_QE + QE_B;
constexpr size_t O_PP = O_PV + PV_B;
constexpr size_t O_MET = O_PP + PP_B;
constexpr size_t O_Q0 = O_MET + 2 * MET_B;
constexpr size_t O_GI4 = O_Q0 + Q0_B;
constexpr size_t O_GI1 = O_GI4 + GI4_B;
constexpr size_t O_GJ4 = O_GI1 + GI1_B;
constexpr size_t O_GJ1 = O_GJ4 + GJ4_B;
constexpr size_t O_LI = O_GJ1 + GJ1_B;
constexpr size_t O_LJ = O_LI + LI_B;
constexpr size_t O_HI4 = O_LJ + LJ_B;
constexpr size_t O_HI1 = O_HI4 + HI4_B;
constexpr size_t O_HJ4 = O_HI1 + HI1_B;
constexpr size_t O_HJ1 = O_HJ4 + HJ4_B;
constexpr size_t O_BAR = O_HJ1 + HJ1_B;
constexpr size_t O_TMEM = O_BAR + 64;  // tensor memory address (written by the allocation)
constexpr size_t BYTES = O_BAR + 128;
// during a chunk's prologue three more raw planes are staged over the node
// and face buffers, which are not in use yet
constexpr size_t O_SCR = O_GI4;
static_assert(O_BAR - O_SCR >= 3 * RAW_B, "prologue staging does not fit");
static_assert(BYTES <= 232448, "shared memory");
// two CTAs per SM: 228 KB per SM, 1 KB reserved per CTA, a few bytes of
// static shared memory in the batched kernel
static_assert(MINB == 1 || 2 * (BYTES + 128 + 1024) <= 228 * 1024, "two CTAs per SM do not fit");
constexpr uint32_t RAW_TX = 4 * 5 * PL;
constexpr uint32_t MET_TX = 4 * 10 * MPL;
constexpr uint32_t Q0_TX = 4 * 5 * UPL;
// mbarriers: 0 raw buffer, 1..3 prologue staging, 4, 5 metrics, 6 Q^(0)
constexpr int B_RAW = 0, B_MET = 4, B_Q0 = 6, NBAR = 7;
// Tensor memory as a per-thread scratchpad (32-bit columns of the thread's
// own lane; the warps that share a lane quadrant take T_COLS columns each):
// four records (primitive 5, conserved 5) of the thread's own column of
// nodes, the state of the k march (G^k 5, low k face flux 5, lambda~, nu, J)
// the node's own low i and j face fluxes (10) and, for an FP64 state between
// steps, the node's five values of it.
constexpr int T_REC = 10, T_MARCH = 4 * T_REC, T_FACE = T_MARCH + 13, T_Q0D = T_FACE + 10;
constexpr int T_COLS = T_Q0D + 10;
constexpr int T_GROUPS = (NT / 32 + 3) / 4;
constexpr int T_ALLOC = T_GROUPS * T_COLS <= 256 ? 256 : 512;  // columns per CTA
static_assert(T_GROUPS * T_COLS <= T_ALLOC && MINB * T_ALLOC <= 512, "tensor memory");
}  // namespace vr

__device__ __forceinline__ void ld5(const float4* v4, const float* v1, int i, float q[5]) {
  const float4 a = v4[i];
  q[0] = a.x; q[1] = a.y; q[2] = a.z; q[3] = a.w;
  q[4] = v1[i];
}
__device__ __forceinline__ void st5(float4* v4, float* v1, int i, const float q[5]) {
  v4[i] = make_float4(q[0], q[1], q[2], q[3]);
  v1[i] = q[4];
}
// a record whose two parts have different row strides: row y, column x
__device__ __forceinline__ void ld5j(const float4* v4, const float* v1, int y, int x, float q[5]) {
  const float4 a = v4[y * vr::TI + x];
  q[0] = a.x; q[1] = a.y; q[2] = a.z; q[3] = a.w;
  q[4] = v1[y * vr::JS1 + x];
}
__device__ __forceinline__ void st5j(float4* v4, float* v1, int y, int x, const float q[5]) {
  v4[y * vr::TI + x] = make_float4(q[0], q[1], q[2], q[3]);
  v1[y * vr::JS1 + x] = q[4];
}
__device__ __forceinline__ void prefetch_map(const CUtensorMap* m) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(m)) : "memory");
}
__device__ __forceinline__ void mbar_inval(uint64_t* bar) {
  asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(smem_addr(bar)) : "memory");
}
// bounded wait with a fast path (the copy has normally landed long before)
__device__ __forceinline__ bool wait_v(uint64_t* bar, uint32_t parity, long long limit) {
  return mbar_try_wait(bar, parity) || mbar_wait_bounded(bar, parity, limit);
}

// --- tensor memory (tcgen05.ld / st, 32 lanes x 32 bits) --------------------
// Every lane of a warp reads and writes its own lane of the warp's quadrant,
// so the columns are private to a thread.  Loads are asynchronous: issue
// them, then tm_wait, then tie() every loaded array before its first use
// (the empty asm makes the uses depend on a statement after the wait).
__device__ __forceinline__ void tm_ld5(uint32_t a, float r[5]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
               : "=f"(r[0]), "=f"(r[1]), "=f"(r[2]), "=f"(r[3]) : "r"(a));
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=f"(r[4]) : "r"(a + 4));
}
__device__ __forceinline__ void tm_ld8(uint32_t a, float r[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=f"(r[0]), "=f"(r[1]), "=f"(r[2]), "=f"(r[3]), "=f"(r[4]), "=f"(r[5]), "=f"(r[6]), "=f"(r[7])
               : "r"(a));
}
__device__ __forceinline__ void tm_ld10(uint32_t a, float r[10]) {
  tm_ld8(a, r);
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0, %1}, [%2];" : "=f"(r[8]), "=f"(r[9]) : "r"(a + 8));
}
__device__ __forceinline__ void tm_ld13(uint32_t a, float r[13]) {
  tm_ld8(a, r);
  tm_ld5(a + 8, r + 8);
}
__device__ __forceinline__ void tm_st5(uint32_t a, const float r[5]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};" ::"r"(a), "f"(r[0]), "f"(r[1]),
               "f"(r[2]), "f"(r[3]));
  asm volatile("tcgen05.st.sync.aligned.32x32b.x1.b32 [%0], {%1};" ::"r"(a + 4), "f"(r[4]));
}
__device__ __forceinline__ void tm_st8(uint32_t a, const float r[8]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(a), "f"(r[0]),
               "f"(r[1]), "f"(r[2]), "f"(r[3]), "f"(r[4]), "f"(r[5]), "f"(r[6]), "f"(r[7]));
}
__device__ __forceinline__ void tm_st10(uint32_t a, const float r[10]) {
  tm_st8(a, r);
  asm volatile("tcgen05.st.sync.aligned.32x32b.x2.b32 [%0], {%1, %2};" ::"r"(a + 8), "f"(r[8]), "f"(r[9]));
}
__device__ __forceinline__ void tm_st13(uint32_t a, const float r[13]) {
  tm_st8(a, r);
  tm_st5(a + 8, r + 8);
}
__device__ __forceinline__ void tm_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tm_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void tie(float (&r)[N]) {
#pragma unroll
  for (int v = 0; v < N; ++v) asm volatile("" : "+f"(r[v]));
}
// allocation by warp 0, published through shared memory; ends with a barrier
__device__ __forceinline__ void tm_alloc(unsigned char* smem) {
  if (threadIdx.x < 32) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(smem + vr::O_TMEM)),
                 "r"(vr::T_ALLOC)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  __syncthreads();
}
__device__ __forceinline__ void tm_free(unsigned char* smem) {
  __syncthreads();  // every warp is past its last access
  if (threadIdx.x < 32)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(
                     *reinterpret_cast<volatile uint32_t*>(smem + vr::O_TMEM)),
                 "r"(vr::T_ALLOC));
}

// Node quantities of node (x, y) of plane kk: G^k = E^k - F^k, lambda~^k,
// nu^k.  The node's own column comes in registers: primitive records of the
// planes below / at / above (pm, pc, pp: u, v, w, T, p) and rho and e; its i
// and j neighbours from the primitive ring slot sC of the plane.  DIR = 0:
// all three directions; DIR = 1 / 2: direction i / j only.
template <int DIR, int MD>
__device__ __forceinline__ void node_v(const float4* __restrict__ PV, const float* __restrict__ PP,
                                       const float* __restrict__ met, int sC, const float pm5[5], const float pc5[5],
                                       const float pp5[5], float rho, float e, int x, int y, const KConst<float>& c,
                                       float mu_inf, float G[3][5], float lt[3], float nu[3], float& Jn) {
  using namespace vr;
  const int o = (y + 2) * RR + x + 2;
  const int mo = (y + 1) * RW + x + 2;
  float S[9];
#pragma unroll
  for (int f = 0; f < 9; ++f) S[f] = met[f * MPL + mo];
  Jn = met[9 * MPL + mo];
  const float4* pc = PV + sC;
  const float u = pc5[0], v = pc5[1], w = pc5[2], T = pc5[3], p = pc5[4];
  constexpr int K0 = DIR == 0 ? 0 : DIR - 1;
  constexpr int K1 = DIR == 0 ? 3 : DIR;

  float Fv[3][4];  // viscous flux vectors F_m (m = x, y, z), components 1..4
#pragma unroll
  for (int m = 0; m < 3; ++m)
#pragma unroll
    for (int q = 0; q < 4; ++q) Fv[m][q] = 0.f;
  if (ModelFlags<MD>::viscous(c)) {
    // Cartesian gradients of u, v, w, T: J/2 sum_k S^k_m (phi_+ - phi_-)
    const float4 a0 = pc[o + 1], b0 = pc[o - 1], a1 = pc[o + RR], b1 = pc[o - RR];
    const float4 a2 = make_float4(pp5[0], pp5[1], pp5[2], pp5[3]), b2 = make_float4(pm5[0], pm5[1], pm5[2], pm5[3]);
    const float hJ = 0.5f * Jn;
    float g[4][3];
#if VR_PACKED_FACES
    {  // the same sums on the variable pairs (u, v) and (w, T), packed FP32x2
      const float2 m1 = make_float2(-1.f, -1.f), h2 = make_float2(hJ, hJ);
      const float2 d0[2] = {__ffma2_rn(make_float2(b0.x, b0.y), m1, make_float2(a0.x, a0.y)),
                            __ffma2_rn(make_float2(b0.z, b0.w), m1, make_float2(a0.z, a0.w))};
      const float2 d1[2] = {__ffma2_rn(make_float2(b1.x, b1.y), m1, make_float2(a1.x, a1.y)),
                            __ffma2_rn(make_float2(b1.z, b1.w), m1, make_float2(a1.z, a1.w))};
      const float2 d2[2] = {__ffma2_rn(make_float2(b2.x, b2.y), m1, make_float2(a2.x, a2.y)),
                            __ffma2_rn(make_float2(b2.z, b2.w), m1, make_float2(a2.z, a2.w))};
#pragma unroll
      for (int pq = 0; pq < 2; ++pq)
#pragma unroll
        for (int m = 0; m < 3; ++m) {
          float2 t = __fmul2_rn(make_float2(S[m], S[m]), d0[pq]);
          t = __ffma2_rn(make_float2(S[3 + m], S[3 + m]), d1[pq], t);
          t = __ffma2_rn(make_float2(S[6 + m], S[6 + m]), d2[pq], t);
          t = __fmul2_rn(h2, t);
          g[2 * pq][m] = t.x;
          g[2 * pq + 1][m] = t.y;
        }
    }
#else
    const float d0[4] = {a0.x - b0.x, a0.y - b0.y, a0.z - b0.z, a0.w - b0.w};
    const float d1[4] = {a1.x - b1.x, a1.y - b1.y, a1.z - b1.z, a1.w - b1.w};
    const float d2[4] = {a2.x - b2.x, a2.y - b2.y, a2.z - b2.z, a2.w - b2.w};
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int m = 0; m < 3; ++m) g[q][m] = hJ * (S[m] * d0[q] + S[3 + m] * d1[q] + S[6 + m] * d2[q]);
#endif
    const float mu = Fn<float>::div(mu_inf * T * Fn<float>::sqrt_(T) * c.s1p1, T + c.s1);  // Sutherland
    float mu_t = 0.f;
    // Smagorinsky or Vreman, Delta = J^(-1/3); an unfused product, so that
    // mu + mu_t rounds alike in the constant-flag and runtime-flag builds
    if (ModelFlags<MD>::sgs(c)) mu_t = Fn<float>::mul_rn(rho, eddy_nu<float, ModelFlags<MD>::eddy>(c, g, Jn));
    const float mue = mu + mu_t;
    const float kap = c.cp * (mu * c.inv_pr + mu_t * c.inv_prt);
    const float div3 = (g[0][0] + g[1][1] + g[2][2]) * (2.f / 3.f);
    const float t01 = mue * (g[0][1] + g[1][0]), t02 = mue * (g[0][2] + g[2][0]), t12 = mue * (g[1][2] + g[2][1]);
    Fv[0][0] = mue * (2.f * g[0][0] - div3); Fv[0][1] = t01; Fv[0][2] = t02;
    Fv[1][0] = t01; Fv[1][1] = mue * (2.f * g[1][1] - div3); Fv[1][2] = t12;
    Fv[2][0] = t02; Fv[2][1] = t12; Fv[2][2] = mue * (2.f * g[2][2] - div3);
#pragma unroll
    for (int m = 0; m < 3; ++m) Fv[m][3] = u * Fv[m][0] + v * Fv[m][1] + w * Fv[m][2] + kap * g[3][m];
  }

  float lam[3], U[3];
  const float cson = Fn<float>::sqrt_(T);
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    U[k] = S[3 * k] * u + S[3 * k + 1] * v + S[3 * k + 2] * w;
    const float sn = Fn<float>::sqrt_(S[3 * k] * S[3 * k] + S[3 * k + 1] * S[3 * k + 1] + S[3 * k + 2] * S[3 * k + 2]);
    lam[k] = fabsf(U[k]) + cson * sn;
  }
  float sq[3] = {0.f, 0.f, 0.f};
  if (ModelFlags<MD>::sig_half(c)) {
#pragma unroll
    for (int k = 0; k < 3; ++k) sq[k] = Fn<float>::sqrt_(lam[k]);
  }
  const float m1 = rho * u, m2 = rho * v, m3 = rho * w;
#pragma unroll
  for (int k = K0; k < K1; ++k) {
    const float Sx = S[3 * k], Sy = S[3 * k + 1], Sz = S[3 * k + 2];
    float Fk[4];
#if VR_PACKED_FACES
#pragma unroll
    for (int q = 0; q < 4; q += 2) {
      float2 t = __fmul2_rn(make_float2(Sx, Sx), make_float2(Fv[0][q], Fv[0][q + 1]));
      t = __ffma2_rn(make_float2(Sy, Sy), make_float2(Fv[1][q], Fv[1][q + 1]), t);
      t = __ffma2_rn(make_float2(Sz, Sz), make_float2(Fv[2][q], Fv[2][q + 1]), t);
      Fk[q] = t.x;
      Fk[q + 1] = t.y;
    }
#else
#pragma unroll
    for (int q = 0; q < 4; ++q) Fk[q] = Sx * Fv[0][q] + Sy * Fv[1][q] + Sz * Fv[2][q];
#endif
    // E^k = [rho U, rho u U + S_x p, rho v U + S_y p, rho w U + S_z p, (e + p) U]
    G[k][0] = rho * U[k];
    G[k][1] = m1 * U[k] + Sx * p - Fk[0];
    G[k][2] = m2 * U[k] + Sy * p - Fk[1];
    G[k][3] = m3 * U[k] + Sz * p - Fk[2];
    G[k][4] = (e + p) * U[k] - Fk[3];
    const int a = (k + 1) % 3, b = (k + 2) % 3;
    if (ModelFlags<MD>::sig_half(c))  // lambda (1 + (la/l)^1/2 + (lb/l)^1/2) = lambda + sqrt(lambda) (sqrt(la) + sqrt(lb))
      lt[k] = lam[k] + sq[k] * (sq[a] + sq[b]);
    else
      lt[k] = lam[k] > 0.f ? lam[k] * (1.f + Fn<float>::powp(Fn<float>::div(lam[a], lam[k]), c.sigma) +
                                       Fn<float>::powp(Fn<float>::div(lam[b], lam[k]), c.sigma))
                           : 0.f;  // zero face metric (a centreline): the limit for sigma < 1
    float pm, pp;
    if (k == 0) { pm = PP[sC + o - 1]; pp = PP[sC + o + 1]; }
    else if (k == 1) { pm = PP[sC + o - RR]; pp = PP[sC + o + RR]; }
    else { pm = pm5[4]; pp = pp5[4]; }
    nu[k] = Fn<float>::div(fabsf(pp - 2.f * p + pm), pp + 2.f * p + pm);
  }
}

// twice the dissipative face flux between nodes a and b of a line m, a, b, p:
// 2h = Ga + Gb - 2 lam [e2 (qb - qa) - e4 (qp - 3 qb + 3 qa - qm)],
// 2 lam = lt_a + lt_b, e2 = k2 max(nu_a, nu_b), e4 = max(0, k4 - e2); the
// update takes half the time step instead (powers of two: the same rounding,
// four operations fewer per face)
__device__ __forceinline__ void face_v(const KConst<float>& c, float2 La, float2 Lb, const float Ga[5],
                                       const float Gb[5], const float qm[5], const float qa[5], const float qb[5],
                                       const float qp[5], float h[5]) {
  const float lam = La.x + Lb.x;
  const float e2 = c.k2 * fmaxf(La.y, Lb.y);
  const float e4 = fmaxf(0.f, c.k4 - e2);
  const float l2 = lam * e2, l4 = lam * e4;
#if VR_PACKED_FACES
  // 2h = (Ga + Gb) - l2 d1 + l4 d3 on component pairs (0, 1) and (2, 3)
  // with packed FP32x2 operations (each lane rounds as its scalar
  // counterpart), component 4 in scalar form
  const float2 m1 = make_float2(-1.f, -1.f), m3 = make_float2(-3.f, -3.f);
  const float2 ml2 = make_float2(-l2, -l2), pl4 = make_float2(l4, l4);
#pragma unroll
  for (int v = 0; v < 4; v += 2) {
    const float2 a = make_float2(qa[v], qa[v + 1]), b = make_float2(qb[v], qb[v + 1]);
    const float2 m = make_float2(qm[v], qm[v + 1]), p = make_float2(qp[v], qp[v + 1]);
    const float2 d1 = __ffma2_rn(a, m1, b);                       // qb - qa
    const float2 d3 = __ffma2_rn(d1, m3, __ffma2_rn(m, m1, p));  // (qp - qm) - 3 d1
    const float2 g = __fadd2_rn(make_float2(Ga[v], Ga[v + 1]), make_float2(Gb[v], Gb[v + 1]));
    const float2 r = __ffma2_rn(pl4, d3, __ffma2_rn(ml2, d1, g));
    h[v] = r.x;
    h[v + 1] = r.y;
  }
  {
    const float d1 = qb[4] - qa[4];
    const float d3 = (qp[4] - qm[4]) - 3.f * d1;
    h[4] = fmaf(l4, d3, fmaf(-l2, d1, Ga[4] + Gb[4]));
  }
#else
#pragma unroll
  for (int v = 0; v < 5; ++v) {
    const float d1 = qb[v] - qa[v];
    const float d3 = (qp[v] - qm[v]) - 3.f * d1;
    h[v] = (Ga[v] + Gb[v]) - (l2 * d1 - l4 * d3);
  }
#endif
}

struct Smem {
  float* raw;
  float4* QV;
  float* QE;
  float4* PV;
  float* PP;
  float* met;
  float4 *Gi4, *Gj4, *Hi4, *Hj4;
  float *Gi1, *Gj1, *Hi1, *Hj1;
  float2 *Li, *Lj;
  uint64_t* bar;
  __device__ explicit Smem(unsigned char* s) {
    using namespace vr;
    raw = reinterpret_cast<float*>(s + O_RAW);
    QV = reinterpret_cast<float4*>(s + O_QV);
    QE = reinterpret_cast<float*>(s + O_QE);
    PV = reinterpret_cast<float4*>(s + O_PV);
    PP = reinterpret_cast<float*>(s + O_PP);
    met = reinterpret_cast<float*>(s + O_MET);
    Gi4 = reinterpret_cast<float4*>(s + O_GI4);
    Gi1 = reinterpret_cast<float*>(s + O_GI1);
    Gj4 = reinterpret_cast<float4*>(s + O_GJ4);
    Gj1 = reinterpret_cast<float*>(s + O_GJ1);
    Li = reinterpret_cast<float2*>(s + O_LI);
    Lj = reinterpret_cast<float2*>(s + O_LJ);
    Hi4 = reinterpret_cast<float4*>(s + O_HI4);
    Hi1 = reinterpret_cast<float*>(s + O_HI1);
    Hj4 = reinterpret_cast<float4*>(s + O_HJ4);
    Hj1 = reinterpret_cast<float*>(s + O_HJ1);
    bar = reinterpret_cast<uint64_t*>(s + O_BAR);
  }
};

// Node role of thread tid (warps hold one role each): 0 tile node, 2 j-halo
// node, 1 i-halo node.
__device__ __forceinline__ int role_of(int tid) {
  return tid < vr::NTILE ? 0 : (tid < vr::NTILE + vr::NJH ? 2 : 1);
}

// One work item: tile (bx, by), k-chunk bz of grid X, stage st, for the
// threads of node role ROLE (each role runs its own instantiation of the
// plane march, without branches on the role; all roles pass the same
// sequence of block barriers).  The CTA's
// mbarriers are (re)initialised at the start of every item, so the parity of
// every wait follows from the plane index.  On a bounded-wait timeout the
// item records where it gave up, lets its copies in flight land and returns
// false.
// S64: the state between time steps is FP64 (X.Q0d at the updated nodes): the
// update adds the FP32 increment to it in FP64, stages 1-4 round their output
// to FP32 (it feeds only the FP32 flux evaluation), and stage 5 writes both
// the FP64 state and its FP32 copy (the next step's flux input).
// c: the flow constants (X.k, or those a batch's grids share), mu_inf apart.
template <int MD, int ROLE, bool S64>
__device__ __forceinline__ bool item_v(const StageCtx<float, float>& X, const KConst<float>& c, const StageSel& st,
                                       int bx, int by, int bz, unsigned char* smem, bool first) {
  using namespace vr;
  Smem sm(smem);
  const Layout& L = X.L;
  const float mu_inf = X.k.mu_inf;
  const int tid = threadIdx.x;
  const int i0 = bx * TI, j0 = by * TJ;
  const int t0 = L.lo[2] + bz * X.kc;
  const int t1 = min(t0 + X.kc, L.hi[2] + 1);
  const uint32_t xtx = st.stall ? kStallBytes : 0u;
  const long long wlim = st.stall ? kStallLimit : kWaitLimit;

  // node role of this thread, a constant of the instantiation: 0 tile node,
  // 2 j-halo node (rows -1, TJ), 1 i-halo node (columns -1, TI)
  constexpr int role = ROLE;
  int nx, ny;
  if constexpr (ROLE == 0) {
    if (ROWS4) {  // warp w: rows (w & 3) + 8 (w >> 2) and 4 below it
      const int w = tid >> 5, l = tid & 31;
      nx = l & 15;
      ny = (w & 3) + 8 * (w >> 2) + 4 * (l >> 4);
    } else {
      nx = tid % TI;
      ny = tid / TI;
    }
  } else if constexpr (ROLE == 2) {
    const int h = tid - NTILE;
    nx = h % TI;
    ny = (h / TI) ? TJ : -1;
  } else {
    const int h = tid - NTILE - NJH;
    if (ROWS4) {  // both halo columns of four rows per quarter-warp: 2-way, not 4-way, bank conflicts
      ny = h >> 1;
      nx = (h & 1) ? TI : -1;
    } else {
      ny = h % TJ;
      nx = (h / TJ) ? TI : -1;
    }
  }
  const int gi = i0 + nx, gj = j0 + ny;
  const bool own = role == 0 && gi >= L.lo[0] && gi <= L.hi[0] && gj >= L.lo[1] && gj <= L.hi[1];

  // Set by a thread whose wait gave up: in phase 1 / in phase 2 of an
  // iteration.  Every thread reads the word in the other phase, when nobody
  // writes it, and leaves at that phase's end: all threads agree without a
  // reduction in the block barriers (two barriers with a reduction per plane
  // cost 1.1% on 256x192x192).
  volatile int* const gave_up = reinterpret_cast<volatile int*>(smem + O_TMEM + 8);
  // (re)initialise the barriers; every copy of the previous item has been
  // waited for, and every thread is past its last wait
  __syncthreads();
  if (tid == 0) {
    gave_up[0] = gave_up[1] = 0;
    for (int b = 0; b < NBAR; ++b) {
      if (!first) mbar_inval(&sm.bar[b]);
      mbar_init(&sm.bar[b], 1);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // generic-proxy writes to the buffers the prologue stages into, then the barrier
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  __syncthreads();
  // up to here parameters and shared memory only
  if (first) wait_for_previous();

  // thread 0's record of its copies: bit b of pend = barrier b has had one,
  // bit b of ppar = the parity of the last one's phase
  uint32_t pend = 0, ppar = 0;
  // bookkeeping of a copy thread 0 is about to issue on barrier b
  auto begin_copy = [&](int b, uint32_t parity, uint32_t bytes) {
    pend |= 1u << b;
    ppar = (ppar & ~(1u << b)) | (parity << b);
    fence_async_shared();
    mbar_expect_tx(&sm.bar[b], bytes + xtx);
  };
  bool ok = true;  // thread 0 issues no copy after a wait of its own has given up
  auto issue_raw = [&](int p, int b, float* dst, uint32_t parity) {
    if (ROLE == 0 && tid == 0 && ok) {
      begin_copy(b, parity, RAW_TX);
      tma_load_4d(dst, &X.tmQ[st.qin], &sm.bar[b], i0, j0, p + NG, 0);
    }
  };
  // the raw buffer takes planes t0+1, t0+2, ...; the two metric buffers
  // planes t0-1, t0, t0+1, ... in turn
  auto raw_parity = [&](int p) { return (uint32_t)((p - t0 - 1) & 1); };
  auto met_sel = [&](int p) { return (p - t0 + 1) & 1; };
  auto met_parity = [&](int p) { return (uint32_t)(((p - t0 + 1) >> 1) & 1); };
  auto met_buf = [&](int p) { return reinterpret_cast<float*>(smem + O_MET + met_sel(p) * MET_B); };
  auto issue_met = [&](int p) {
    if (ROLE == 0 && tid == 0 && ok) {
      const int b = B_MET + met_sel(p);
      begin_copy(b, met_parity(p), MET_TX);
      tma_load_4d(met_buf(p), &X.tmMv, &sm.bar[b], i0, j0 + 1, p + NG, 0);
    }
  };
  int phase = 0;
  auto wait = [&](int b, uint32_t parity, int p) {
    if (wait_v(&sm.bar[b], parity, wlim)) return;
    ok = false;
    gave_up[phase] = 1;
    if (ROLE == 0 && tid == 0 && atomicCAS(X.err, 0, 1) == 0) {
      int* info = X.err + 1;
      info[0] = b; info[1] = (int)parity; info[2] = p; info[3] = bx; info[4] = by; info[5] = bz; info[6] = st.qin;
    }
  };

  // this thread's node in a ring plane, and its tensor-memory columns
  const int oo = (ny + 2) * RR + nx + 2;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
  const uint32_t tm = __shfl_sync(0xffffffffu, *reinterpret_cast<volatile uint32_t*>(smem + O_TMEM), 0) +
                      ((uint32_t)(warp & 3) << 21) + (uint32_t)((warp >> 2) * T_COLS);

  // Convert a staged plane (planar, in src) into the records of conserved
  // slot sq and primitive slot sp: every thread its own node, whose record
  // also goes to its tensor-memory record rec; halo threads the next node
  // outwards too, and four of them the corners of the one-node halo (the
  // outer corners are not read).
  const int oraw = (ny + 2) * RW + nx + 2;
  auto convert = [&](const float* src, int sq, int sp, int rec) {
    int e = oraw, o = oo;
    constexpr int NC = ROLE == 0 ? 1 : (ROLE == 2 ? 2 : 3);
    bool on = true;
#pragma unroll
    for (int b = 0; b < NC; ++b) {
      float r[10];
      if (on) {
#pragma unroll
        for (int v = 0; v < 5; ++v) r[5 + v] = src[v * PL + e];
        const float ri = Fn<float>::rcp(r[5]);
#pragma unroll
        for (int m = 0; m < 3; ++m) r[m] = r[6 + m] * ri;
        r[4] = c.gm1 * (r[9] - 0.5f * r[5] * (r[0] * r[0] + r[1] * r[1] + r[2] * r[2]));
        r[3] = c.gamma * r[4] * ri;
        st5(sm.QV + sq, sm.QE + sq, o, r + 5);
        st5(sm.PV + sp, sm.PP + sp, o, r);
      }
      if (b == 0) {
        __syncwarp();
        tm_st10(tm + rec, r);
      }
      if (ROLE == 2) {
        const int d = ny < 0 ? -1 : 1;
        e += d * RW;
        o += d * RR;
      }
      if (ROLE == 1) {
        const int h = tid - NTILE - NJH;
        if (b == 0) {
          const int d = nx < 0 ? -1 : 1;
          e += d;
          o += d;
        } else {
          on = h < 4;
          const int cx = (h & 1) ? TI + 2 : 1, cy = (h & 2) ? TJ + 2 : 1;
          e = cy * RW + cx;
          o = cy * RR + cx;
        }
      }
    }
  };

  const float hadt = 0.5f * (float)(st.alpha * X.sc->dt);  // half: the residual is formed of twice the face fluxes
  const long long npad = L.npad;
  float* const Qo = X.Q[st.qout];
  // Q^(0) of the plane being updated: for the first stage it is the stage
  // input, which the own column's records hold; otherwise TMA stages it one
  // plane ahead (tile rows, 36 columns from the aligned column i0-2)
  const bool q0_own = S64 || st.qin == 0;
  const float* q0buf = reinterpret_cast<const float*>(smem + O_Q0);
  auto issue_q0 = [&](int p) {
    if (ROLE == 0 && tid == 0 && !q0_own && ok) {
      begin_copy(B_Q0, (uint32_t)((p - t0) & 1), Q0_TX);
      tma_load_4d(smem + O_Q0, &X.tmQ0u, &sm.bar[B_Q0], i0, j0 + 2, p + NG, 0);
    }
  };
  long long n_t0 = own ? L.at(gi, gj, t0) : 0;  // this thread's node in plane t0
  float* scr[3] = {reinterpret_cast<float*>(smem + O_SCR), reinterpret_cast<float*>(smem + O_SCR + RAW_B),
                   reinterpret_cast<float*>(smem + O_SCR + 2 * RAW_B)};

  // ---- prologue: planes t0-2 .. t0+1 and the metrics of t0-1, t0 staged at
  // once; planes t0-1, t0 converted, the own column's records of t0-2 and
  // t0-1 to tensor memory
  issue_raw(t0 - 2, 1, scr[0], 0);
  issue_raw(t0 - 1, 2, scr[1], 0);
  issue_raw(t0, 3, scr[2], 0);
  issue_met(t0 - 1);
  issue_raw(t0 + 1, B_RAW, sm.raw, 0);
  issue_met(t0);
#pragma unroll 1
  for (int q = 0; q < 3; ++q) {  // primitive slots 1, 0, 1: plane t0's records replace t0-2's, which no other thread reads
    wait(1 + q, 0, t0 - 2 + q);
    convert(scr[0] + q * (RAW_B / 4), q * RPL, ((q + 1) & 1) * RPL, q * T_REC);
  }
  __syncwarp();
  tm_wait_st();
  if (__syncthreads_or(!ok)) goto fail;

  {
    // the node's own face data, from the node pass to the face pass
    float Gi[5], Gj[5];
    float2 Li, Lj;
    const bool do_i = role == 0 || (role == 1 && nx == TI);
    const bool do_j = role == 0 || (role == 2 && ny == TJ);

    // ---- march in k: iteration t writes plane t (from t0 on; the two before
    // it only build up the k march).  Phase 1: node pass of plane t+1, k face
    // t + 1/2, i/j residual of plane t (faces from phase 2 of the previous
    // iteration) and the update of plane t.  Phase 2: i/j faces of plane t+1
    // and the conversion of plane t+3.  r0, r1, r2: conserved ring slots of
    // planes t, t+1, t+2 (t+3 takes t's slot); k0: tensor-memory record of
    // plane t (of four in turn).
    int r0 = 0, r1 = RPL, r2 = 2 * RPL, k0 = 0;
#pragma unroll 1
    for (int t = t0 - 2; t < t1; ++t) {
      const bool live = t + 1 >= t0 && t + 1 < t1;  // plane t+1 is updated: its faces are needed
      const int sp1 = ((t - t0) & 1) * RPL;  // primitive slot of plane t+1
      const int k1 = (k0 + 1) & 3, k2 = (k0 + 2) & 3, k3 = (k0 + 3) & 3;
      float qb[5];  // own conserved record of plane t+1
      float G3n[5], lt3n = 0.f, nu3n = 0.f, Jn = 0.f;
      const int left2 = gave_up[1];  // of the previous iteration's phase 2
      phase = 0;
      wait(B_MET + met_sel(t + 1), met_parity(t + 1), t + 1);
      __syncwarp();
      {
        float pb[5], pt[5], pn[5];
        tm_ld5(tm + k0 * T_REC, pb);
        tm_ld5(tm + k1 * T_REC, pt);
        tm_ld5(tm + k1 * T_REC + 5, qb);
        tm_ld5(tm + k2 * T_REC, pn);
        tm_wait_ld();
        tie(pb);
        tie(pt);
        tie(qb);
        tie(pn);
        const float* met = met_buf(t + 1);
        float G[3][5], lt[3], nu[3];
        if constexpr (ROLE == 0) {
          node_v<0, MD>(sm.PV, sm.PP, met, sp1, pb, pt, pn, qb[0], qb[4], nx, ny, c, mu_inf, G, lt, nu, Jn);
#pragma unroll
          for (int v = 0; v < 5; ++v) {
            Gi[v] = G[0][v];
            Gj[v] = G[1][v];
            G3n[v] = G[2][v];
          }
          lt3n = lt[2];
          nu3n = nu[2];
        } else if (live) {
          node_v<ROLE, MD>(sm.PV, sm.PP, met, sp1, pb, pt, pn, qb[0], qb[4], nx, ny, c, mu_inf, G, lt, nu, Jn);
#pragma unroll
          for (int v = 0; v < 5; ++v) {
            if (ROLE == 1) Gi[v] = G[0][v];
            else Gj[v] = G[1][v];
          }
        }
        if (ROLE == 0 || live) {
          if (ROLE != 2) {
            Li = make_float2(lt[0], nu[0]);
            st5(sm.Gi4, sm.Gi1, ny * GIW + nx + 1, Gi);
            sm.Li[ny * GIW + nx + 1] = Li;
          }
          if (ROLE != 1) {
            Lj = make_float2(lt[1], nu[1]);
            st5j(sm.Gj4, sm.Gj1, ny + 1, nx, Gj);
            sm.Lj[(ny + 1) * TI + nx] = Lj;
          }
        }
      }
      if (!q0_own && t >= t0) wait(B_Q0, (uint32_t)((t - t0) & 1), t);
      if constexpr (ROLE == 0) {
        float mv[13], hl[10], qc[5], qd[5], qp[5], hk[5];
        __syncwarp();
        tm_ld13(tm + T_MARCH, mv);
        tm_ld5(tm + k3 * T_REC + 5, qc);  // plane t-1
        tm_ld5(tm + k0 * T_REC + 5, qd);
        tm_ld5(tm + k2 * T_REC + 5, qp);
        tm_wait_ld();
        tie(mv);
        tie(qc);
        tie(qd);
        tie(qp);
        tm_ld10(tm + T_FACE, hl);
        float q0w[10];  // the FP64 values' words
        if constexpr (S64) tm_ld10(tm + T_Q0D, q0w);
        face_v(c, make_float2(mv[10], mv[11]), make_float2(lt3n, nu3n), mv, G3n, qc, qd, qb, qp, hk);
        {
          float nv[13];
#pragma unroll
          for (int v = 0; v < 5; ++v) {
            nv[v] = G3n[v];
            nv[5 + v] = hk[v];
          }
          nv[10] = lt3n;
          nv[11] = nu3n;
          nv[12] = Jn;
          tm_st13(tm + T_MARCH, nv);
        }
        // i/j residual from the four face fluxes around the node: its own low
        // ones from tensor memory, the high ones of its neighbours' threads
        float hi[5], hj[5];
        ld5(sm.Hi4, sm.Hi1, ny * HIW + nx + 1, hi);
        ld5j(sm.Hj4, sm.Hj1, ny + 1, nx, hj);
        tm_wait_ld();
        tie(hl);
        if constexpr (S64) tie(q0w);
        if (own && t >= t0) {
          float q0[5];
          if constexpr (S64) {  // the increment alone
#pragma unroll
            for (int v = 0; v < 5; ++v) q0[v] = 0.f;
          } else if (q0_own) {
#pragma unroll
            for (int v = 0; v < 5; ++v) q0[v] = qd[v];
          } else {
#pragma unroll
            for (int v = 0; v < 5; ++v) q0[v] = q0buf[v * UPL + ny * RW + nx + 2];
          }
          float* const dst = Qo + n_t0 + (long long)(t - t0) * L.plane;
          const float aj = -(hadt * mv[12]);
          float qn[5];
          const float2 m1 = make_float2(-1.f, -1.f), aj2 = make_float2(aj, aj);
#pragma unroll
          for (int v = 0; v < 4; v += 2) {  // packed pairs, each lane rounding as its scalar counterpart
            const float2 di = __ffma2_rn(make_float2(hl[v], hl[v + 1]), m1, make_float2(hi[v], hi[v + 1]));
            const float2 dj = __ffma2_rn(make_float2(hl[5 + v], hl[6 + v]), m1, make_float2(hj[v], hj[v + 1]));
            const float2 dk = __ffma2_rn(make_float2(mv[5 + v], mv[6 + v]), m1, make_float2(hk[v], hk[v + 1]));
            const float2 r = __ffma2_rn(aj2, __fadd2_rn(__fadd2_rn(di, dj), dk), make_float2(q0[v], q0[v + 1]));
            qn[v] = r.x;
            qn[v + 1] = r.y;
          }
          qn[4] = fmaf(aj, ((hi[4] - hl[4]) + (hj[4] - hl[9])) + (hk[4] - mv[9]), q0[4]);
          if constexpr (S64) {
            double* const dst64 = X.Q0d + n_t0 + (long long)(t - t0) * L.plane;
            double qd[5];
            widen5(qn, qd);
#pragma unroll
            for (int v = 0; v < 5; ++v)
              qd[v] += __hiloint2double(__float_as_int(q0w[2 * v + 1]), __float_as_int(q0w[2 * v]));
#pragma unroll
            for (int v = 0; v < 5; ++v) {
              dst[v * npad] = (float)qd[v];
              if (st.qout == 0) dst64[v * npad] = qd[v];
            }
          } else {
#pragma unroll
            for (int v = 0; v < 5; ++v) dst[v * npad] = qn[v];
          }
        }
      }
      __syncwarp();
      tm_wait_st();
      __syncthreads();
      if (left2) goto fail;
      const int left1 = gave_up[0];
      phase = 1;
      if (t + 3 <= t1) issue_met(t + 3);
      // face fluxes (twice) of plane t+1 on the low side of this thread's
      // node: i face between nx-1 and nx (tile nodes and the i-halo column
      // TI), j face between ny-1 and ny (tile nodes and the j-halo row TJ).
      // A tile node keeps its two faces in tensor memory for its residual.
      if (live) {
        issue_q0(t + 1);
        // the FP64 state of plane t+1, through tensor memory to its update: the
        // faces hide the loads' latency
        double q0d[S64 ? 5 : 1];
        if constexpr (S64 && ROLE == 0) {
          const double* src = X.Q0d + n_t0 + (long long)(t + 1 - t0) * L.plane;
#pragma unroll
          for (int v = 0; v < 5; ++v) q0d[v] = own ? src[v * npad] : 0.0;
        }
        const float4* qv = sm.QV + r1;
        const float* qe = sm.QE + r1;
        float qo[5], hij[10];
        __syncwarp();
        tm_ld5(tm + k1 * T_REC + 5, qo);
        tm_wait_ld();
        tie(qo);
        if (do_i) {
          float Ga[5], qm[5], qa[5], qp[5];
          ld5(sm.Gi4, sm.Gi1, ny * GIW + nx, Ga);
          ld5(qv, qe, oo - 2, qm);
          ld5(qv, qe, oo - 1, qa);
          ld5(qv, qe, oo + 1, qp);
          face_v(c, sm.Li[ny * GIW + nx], Li, Ga, Gi, qm, qa, qo, qp, hij);
          st5(sm.Hi4, sm.Hi1, ny * HIW + nx, hij);
        }
        if (do_j) {
          float Ga[5], qm[5], qa[5], qp[5];
          ld5j(sm.Gj4, sm.Gj1, ny, nx, Ga);
          ld5(qv, qe, oo - 2 * RR, qm);
          ld5(qv, qe, oo - RR, qa);
          ld5(qv, qe, oo + RR, qp);
          face_v(c, sm.Lj[ny * TI + nx], Lj, Ga, Gj, qm, qa, qo, qp, hij + 5);
          st5j(sm.Hj4, sm.Hj1, ny, nx, hij + 5);
        }
        if constexpr (ROLE == 0) {
          tm_st10(tm + T_FACE, hij);
          if constexpr (S64) {
            float q0w[10];
#pragma unroll
            for (int v = 0; v < 5; ++v) {
              q0w[2 * v] = __int_as_float(__double2loint(q0d[v]));
              q0w[2 * v + 1] = __int_as_float(__double2hiint(q0d[v]));
            }
            tm_st10(tm + T_Q0D, q0w);
          }
        }
      }
      if (t + 3 <= t1 + 1) {
        wait(B_RAW, raw_parity(t + 3), t + 3);
        convert(sm.raw, r0, sp1, k3 * T_REC);
        __syncwarp();
        tm_wait_st();
      }
      __syncthreads();
      if (left1) goto fail;
      if (t + 4 <= t1 + 1) issue_raw(t + 4, B_RAW, sm.raw, raw_parity(t + 4));
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
    for (int b = 0; b < NBAR; ++b)
      if (pend & (1u << b)) {
        if (xtx) mbar_complete_tx(&sm.bar[b], xtx);
        mbar_wait_bounded(&sm.bar[b], (ppar >> b) & 1u);
      }
  }
  __syncthreads();
  return false;
}

template <int MD, bool S64>
__global__ void __launch_bounds__(vr::NT, vr::MINB)
    k_stage_v(const __grid_constant__ StageCtx<float, float> X, const StageSel st) {
  extern __shared__ __align__(128) unsigned char smem[];
  // with the barriers' set-up, before the previous kernel's results are needed:
  // 69x47x46 90.3 to 88.2 us per step, 256x192x192 1.697 to 1.686 ms
  if (threadIdx.x == 0) {
    prefetch_map(&X.tmQ[st.qin]);
    prefetch_map(&X.tmMv);
    prefetch_map(&X.tmQ0u);
  }
  tm_alloc(smem);
  switch (role_of(threadIdx.x)) {
    case 0: item_v<MD, 0, S64>(X, X.k, st, blockIdx.x, blockIdx.y, blockIdx.z, smem, true); break;
    case 2: item_v<MD, 2, S64>(X, X.k, st, blockIdx.x, blockIdx.y, blockIdx.z, smem, true); break;
    default: item_v<MD, 1, S64>(X, X.k, st, blockIdx.x, blockIdx.y, blockIdx.z, smem, true); break;
  }
  tm_free(smem);
}

// SHARED: the grids agree in all flow constants but mu_inf; the constants then
// come as a kernel parameter, whose values need no registers (from the
// contexts they do, and the kernel spills).
template <int MD, bool S64, bool SHARED>
__global__ void __launch_bounds__(vr::NT, vr::MINB)
    k_stage_v_batch(const StageCtx<float, float>* __restrict__ ctx, const __grid_constant__ KConst<float> common,
                    const int4* __restrict__ items, int nitems, unsigned int* queue, const StageSel st) {
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ int next;
  bool first = true;
  tm_alloc(smem);
  for (;;) {
    if (threadIdx.x == 0) next = (int)atomicAdd(queue, 1u);
    __syncthreads();
    const int it = next;
    __syncthreads();
    if (it >= nitems) break;
    const int4 w = items[it];
    const KConst<float>& c = SHARED ? common : ctx[w.x].k;
    bool ok;
    switch (role_of(threadIdx.x)) {
      case 0: ok = item_v<MD, 0, S64>(ctx[w.x], c, st, w.y, w.z, w.w, smem, first); break;
      case 2: ok = item_v<MD, 2, S64>(ctx[w.x], c, st, w.y, w.z, w.w, smem, first); break;
      default: ok = item_v<MD, 1, S64>(ctx[w.x], c, st, w.y, w.z, w.w, smem, first); break;
    }
    if (!ok) break;
    first = false;
  }
  tm_free(smem);
}

template <int MD, bool S64>
cudaError_t configure_model() {
  const cudaFuncAttribute at = cudaFuncAttributeMaxDynamicSharedMemorySize;
  cudaError_t e = cudaFuncSetAttribute(k_stage_v<MD, S64>, at, (int)vr::BYTES);
  if (e != cudaSuccess) return e;
  if ((e = cudaFuncSetAttribute(k_stage_v_batch<MD, S64, false>, at, (int)vr::BYTES)) != cudaSuccess) return e;
  if (MD != kModelSmagorinsky || S64) return e;
  return cudaFuncSetAttribute(k_stage_v_batch<kModelSmagorinsky, false, true>, at, (int)vr::BYTES);
}

template <int MD, bool S64>
cudaError_t launch(const StageCtx<float, float>& X, const StageSel& st, cudaStream_t s) {
  const Layout& L = X.L;
  const int nz = L.hi[2] - L.lo[2] + 1;
  dim3 grid((L.hi[0] + vr::TI) / vr::TI, (L.hi[1] + vr::TJ) / vr::TJ, (nz + X.kc - 1) / X.kc);
  count_launches(1);
  return launch_dep(k_stage_v<MD, S64>, grid, vr::NT, vr::BYTES, s, X, st);
}

template <int MD, bool S64, bool SHARED = false>
cudaError_t launch_batch(const void* ctx, const int4* items, int nitems, unsigned int* queue, const StageSel& st,
                         cudaStream_t s, const KConst<float>* common = nullptr) {
  cudaError_t e = cudaMemsetAsync(queue, 0, sizeof(unsigned int), s);
  if (e != cudaSuccess) return e;
  const int slots = device_sm_count() * vr::MINB;
  const int ctas = nitems < slots ? nitems : slots;
  k_stage_v_batch<MD, S64, SHARED><<<ctas, vr::NT, vr::BYTES, s>>>((const StageCtx<float, float>*)ctx,
                                                                   common ? *common : KConst<float>{}, items, nitems,
                                                                   queue, st);
  count_launches(1);
  return cudaGetLastError();
}

}  // namespace

cudaError_t VR_FN(stage_v_configure)() {
  cudaError_t e;
#if VR_TI == 16 && VR_TJ == 16
  if ((e = configure_model<kModelRuntime, true>()) != cudaSuccess) return e;
  if ((e = configure_model<kModelSmagorinsky, true>()) != cudaSuccess) return e;
#endif
  if ((e = configure_model<kModelRuntime, false>()) != cudaSuccess) return e;
  if ((e = configure_model<kModelSmagorinsky, false>()) != cudaSuccess) return e;
  if ((e = configure_model<kModelVreman, false>()) != cudaSuccess) return e;
  return configure_model<kModelEuler, false>();
}

cudaError_t VR_FN(launch_stage_v)(const StageCtx<float, float>& X, const StageSel& st, cudaStream_t s) {
  switch (flow_model(X.k)) {
    case kModelSmagorinsky: return launch<kModelSmagorinsky, false>(X, st, s);
    case kModelVreman: return launch<kModelVreman, false>(X, st, s);
    case kModelEuler: return launch<kModelEuler, false>(X, st, s);
    default: return launch<kModelRuntime, false>(X, st, s);
  }
}

// model: the flow model every grid of the batch shares (kModelRuntime when
// they differ); common: the flow constants they share but for mu_inf (else
// null)
cudaError_t VR_FN(launch_stage_v_batch)(const void* ctx, const int4* items, int nitems, unsigned int* queue,
                                        const StageSel& st, int model, const KConst<float>* common, cudaStream_t s) {
  switch (model) {
    case kModelSmagorinsky:
      if (common) return launch_batch<kModelSmagorinsky, false, true>(ctx, items, nitems, queue, st, s, common);
      return launch_batch<kModelSmagorinsky, false>(ctx, items, nitems, queue, st, s);
    case kModelVreman: return launch_batch<kModelVreman, false>(ctx, items, nitems, queue, st, s);
    case kModelEuler: return launch_batch<kModelEuler, false>(ctx, items, nitems, queue, st, s);
    default: return launch_batch<kModelRuntime, false>(ctx, items, nitems, queue, st, s);
  }
}

#if VR_TI == 16 && VR_TJ == 16
// JZ_P32_S64 grids: one tile shape, and constant flags for the Smagorinsky
// model of the configurations only
cudaError_t launch_stage_v_s64(const StageCtx<float, float>& X, const StageSel& st, cudaStream_t s) {
  if (flow_model(X.k) == kModelSmagorinsky) return launch<kModelSmagorinsky, true>(X, st, s);
  return launch<kModelRuntime, true>(X, st, s);
}

cudaError_t launch_stage_v_batch_s64(const void* ctx, const int4* items, int nitems, unsigned int* queue,
                                     const StageSel& st, int model, cudaStream_t s) {
  if (model == kModelSmagorinsky) return launch_batch<kModelSmagorinsky, true>(ctx, items, nitems, queue, st, s);
  return launch_batch<kModelRuntime, true>(ctx, items, nitems, queue, st, s);
}
#endif

}  // namespace jz
