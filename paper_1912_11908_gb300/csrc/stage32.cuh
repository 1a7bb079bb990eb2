// Per-tile device code of the FP32-bulk stage kernels, shared by the
// single-case kernels (flow32.cu) and the block-table kernels of the
// request loop (batch32.cu), which live in separate modules.
//
// FP32-bulk flow kernels.
//
// Stage values, reconstruction and fluxes run in FP32 on perturbations from
// the free stream, dU = (rho - rho_inf, rho u - rho_inf u_inf,
// rho v - rho_inf v_inf, W'), W' = (rho E - rho_inf E_inf) - H_inf (rho -
// rho_inf).  Primitives are (rho', u, v, p') with p' = p - p_inf and
// T' = T - T_inf formed without ever adding p_inf or H_inf to an FP32 value,
// so O(M^2) pressure and temperature fluctuations keep their FP32 precision
// at any free-stream Mach number.  The state U^n is held in FP64 as the same
// perturbation dU and accumulated in FP64 at the last stage of every step:
// dU^{n+1} = dU^n + (double)[2/3 ((dU^(2) - dU^n) + dt L)], where the bracket
// is an O(dt) increment formed in FP32 (the FP32 mirror of dU^n is rounded
// from the FP64 state after every step, so FP32 rounding never accumulates in
// U^n).
#pragma once

#include <cuda.h>  // CUtensorMap

#include "f32x2.cuh"
#include "dual_update.cuh"  // FP64 point-implicit update of the dual-time pseudo stages
#include "ibm_internal.cuh"

namespace ibm {

// perturbation conserved -> (rho', u, v, p', T').  One rounding for every place that converts a cell: this scalar form
// takes the operations of the form for two cells below one by one, uncontracted, so that a cell has the same primitives in
// an interior tile, a tile at the domain's edge and the reconstruction of a neighbour tile's node, and a face between two
// tiles one flux.  The velocities are the momenta over the rounded density, so that density times velocity returns the
// momentum where 1 + rho' keeps few digits of rho'.  (u_inf + u' rounds differently, with no form closer to 64 bits
// throughout: forces after a dual-time step at M = 0.001, mean over 16 fields, 2048 x 1024 4e-8 here and 6e-8 so, 257 x 131
// 1.5e-7 and 2.1e-7, 768 x 384 8e-8 and 4e-8.)
__device__ __forceinline__ void pert_prim(const PertConsts &c, float dr, float dmx, float dmy, float W, float &u,
                                          float &v, float &pp, float &Tp) {
  const float ir = __fdividef(1.f, __fadd_rn(1.f, dr));
  const float du = __fmul_rn(__fmaf_rn(-c.ux, dr, dmx), ir), dv = __fmul_rn(__fmaf_rn(-c.uy, dr, dmy), ir);
  u = __fmul_rn(__fadd_rn(c.ux, dmx), ir);
  v = __fmul_rn(__fadd_rn(c.uy, dmy), ir);
  const float dq = __fmaf_rn(du, __fadd_rn(c.ux, u), __fmul_rn(dv, __fadd_rn(c.uy, v)));  // |u|^2 - |u_inf|^2
  const float ke2 = __fmaf_rn(dr, __fmaf_rn(u, u, __fmul_rn(v, v)), dq);  // rho |u|^2 - rho_inf |u_inf|^2
  pp = __fmul_rn(c.g1, __fmaf_rn(-0.5f, ke2, __fmaf_rn(c.Hinf, dr, W)));
  Tp = __fmul_rn(__fmul_rn(__fmaf_rn(-c.R, dr, pp), ir), __fdividef(1.f, c.R));
}

// the same for two cells
__device__ __forceinline__ void pert_prim2(const PertConsts &c, f2 dr, f2 dmx, f2 dmy, f2 W, f2 &u, f2 &v, f2 &pp,
                                           f2 &Tp) {
  const f2 ir = rcp2(1.f + dr);
  const f2 du = fma2(-c.ux, dr, dmx) * ir, dv = fma2(-c.uy, dr, dmy) * ir;
  u = (c.ux + dmx) * ir;
  v = (c.uy + dmy) * ir;
  const f2 dq = fma2(du, c.ux + u, dv * (c.uy + v));
  const f2 ke2 = fma2(dr, fma2(u, u, v * v), dq);
  pp = c.g1 * fma2(-0.5f, ke2, fma2(c.Hinf, dr, W));
  Tp = (fma2(-c.R, dr, pp) * ir) * both(__fdividef(1.f, c.R));
}

// (p', u, v, T') -> perturbation conserved
__device__ __forceinline__ void prim_pert(const PertConsts &c, float pp, float u, float v, float Tp, float &dr,
                                          float &dmx, float &dmy, float &W) {
  dr = (pp - c.R * Tp) / (c.R * (1.f + Tp));
  dmx = dr * u + (u - c.ux);
  dmy = dr * v + (v - c.uy);
  const float dq = (u - c.ux) * (u + c.ux) + (v - c.uy) * (v + c.uy);
  const float ke = 0.5f * (dr * (u * u + v * v) + dq);
  W = pp / c.g1 + ke - c.Hinf * dr;
}

// LDFSS(0) in perturbation form (Mr^2 = 1).  States (rho', un, ut, p');
// un_inf / ut_inf the free-stream components along the face normal and
// tangent.  Momentum flux drops the constant p_inf n (its divergence is
// zero); D_L + D_R - 1 is formed in factored form for two subsonic sides so
// p_inf (D_L + D_R - 1) keeps its precision.
//
// PRE (dual time, Sec. 2): the low-Mach numerical sound speed
// c' = 1/2 sqrt((1 - Mr^2)^2 un^2 + 4 Mr^2 c^2), Mr^2 = (Ur/c)^2 with
// Ur = min(c, max(|V|, U_ref, nu/dn)) from face averages (idn = 1/dn),
// scales the mass-flux (dissipation) part; the pressure split takes the
// physical face Mach numbers and its departure from the face mean (the
// rho c du dissipation) is scaled by c'/c, as in the FP64 path.
//
// Two faces at a time in packed arithmetic (f32x2.cuh); the reciprocals, square roots, extrema and selects are scalar.
template <bool PRE = false>
__device__ __forceinline__ void ldfss_pert2(const PertConsts &c, f2 drL, f2 unL, f2 utL, f2 ppL, f2 drR, f2 unR,
                                            f2 utR, f2 ppR, float un_inf, float ut_inf, f2 F[4], float idn = 0.f) {
  const f2 rL = 1.f + drL, rR = 1.f + drR;
  const f2 irL = rcp2(rL), irR = rcp2(rR);
  const float gR = c.gamma * c.R;
  const f2 cL = sqrt2(fma2(c.gamma, ppL, both(gR)) * irL), cR = sqrt2(fma2(c.gamma, ppR, both(gR)) * irR);
  const f2 kL = fma2(unL - both(un_inf), un_inf + unL, (utL - both(ut_inf)) * (ut_inf + utL));
  const f2 kR = fma2(unR - both(un_inf), un_inf + unR, (utR - both(ut_inf)) * (ut_inf + utR));
  const f2 HL = fma2(c.gg, fma2(-c.R, drL, ppL) * irL, 0.5f * kL);
  const f2 HR = fma2(c.gg, fma2(-c.R, drR, ppR) * irR, 0.5f * kR);
  const f2 cb = 0.5f * (cL + cR);
  f2 cs = cb, mr2 = both(1.f);
  if (PRE) {
    const f2 ub = 0.5f * (unL + unR), vb = 0.5f * (utL + utR);
    const f2 Vm = sqrt2(fma2(ub, ub, vb * vb)), nu = (c.mu * idn) * rcp2(0.5f * (rL + rR));
    const f2 Ur = min2(max2(max2(Vm, both(1.f)), nu), cb);
    const f2 q = Ur * rcp2(cb);
    mr2 = min2(q * q, both(1.f));
    const f2 om = both(1.f) - mr2, w = om * ub;
    cs = 0.5f * sqrt2(fma2(w, w, (4.f * mr2) * (cb * cb)));
  }
  const f2 ics = rcp2(cs), ML = unL * ics, MR = unR * ics;
  // the split functions' subsonic / supersonic branches as selects: alpha = 1 (0) for M >= 0 (< 0) on the
  // left, the reverse on the right; beta = -1 subsonic, 0 supersonic
  const bool sLx = fabsf(ML.x) < 1.f, sLy = fabsf(ML.y) < 1.f, sRx = fabsf(MR.x) < 1.f, sRy = fabsf(MR.y) < 1.f;
  const f2 hL = fma2(0.5f, ML, both(0.5f)), hR = fma2(0.5f, MR, both(-0.5f));
  const f2 MpL = hL * hL, MmR = hR * hR;  // M+ and -M-
  const f2 CVL = {sLx ? MpL.x : fmaxf(ML.x, 0.f), sLy ? MpL.y : fmaxf(ML.y, 0.f)};
  const f2 CVR = {sRx ? -MmR.x : fminf(MR.x, 0.f), sRy ? -MmR.y : fminf(MR.y, 0.f)};
  const f2 mm = fma2(MR, MR, ML * ML);
  const f2 sq = fma2(0.5f, sqrt2(0.5f * mm), both(-0.5f)), sq2 = sq * sq;
  const f2 Mh = {sLx && sRx ? sq2.x : 0.f, sLy && sRy ? sq2.y : 0.f};
  const f2 dp = ppL - ppR, ic2 = ics * ics;
  // -(dp + |dp|) / 2 and -(|dp| - dp) / 2
  const f2 dpL = {fminf(-dp.x, 0.f), fminf(-dp.y, 0.f)}, dpR = {fminf(dp.x, 0.f), fminf(dp.y, 0.f)};
  const f2 Cp = CVL - Mh * fma2(dpL, ic2 * irL, both(1.f));
  const f2 Cm = fma2(Mh, fma2(dpR, ic2 * irR, both(1.f)), CVR);
  const f2 mL = rL * (cs * Cp), mR = rR * (cs * Cm);
  // p_inf (D_L + D_R - 1) + D_L p'_L + D_R p'_R; with low-Mach scaling (pressure split with the physical face Mach
  // numbers) the departure from the face mean 1/2 (p'_L + p'_R) is scaled by c'/c
  f2 ph;
  bool low_x = false, low_y = false;
  if (PRE) low_x = mr2.x < 1.f, low_y = mr2.y < 1.f;
  {
    f2 m1 = ML, m2 = MR, kLs = hL, kRs = hR, q3 = mm, im = ics;
    bool pLx = sLx, pLy = sLy, pRx = sRx, pRy = sRy;
    f2 icb = both(1.f);
    if (PRE) {
      icb = rcp2(cb);
      im = f2{low_x ? icb.x : ics.x, low_y ? icb.y : ics.y};
      m1 = unL * im;
      m2 = unR * im;
      pLx = fabsf(m1.x) < 1.f, pLy = fabsf(m1.y) < 1.f, pRx = fabsf(m2.x) < 1.f, pRy = fabsf(m2.y) < 1.f;
      kLs = fma2(0.5f, m1, both(0.5f));
      kRs = fma2(0.5f, m2, both(-0.5f));
      q3 = fma2(m2, m2, m1 * m1);
    }
    const f2 PpL = (PRE ? kLs * kLs : MpL) * (both(2.f) - m1), PmR = (PRE ? kRs * kRs : MmR) * (2.f + m2);
    // outside |M| < 1: 1 or 0 by the sign of M
    const f2 DL = {pLx ? PpL.x : __saturatef(m1.x), pLy ? PpL.y : __saturatef(m1.y)};
    const f2 DR = {pRx ? PmR.x : __saturatef(-m2.x), pRy ? PmR.y : __saturatef(-m2.y)};
    // (M_R - M_L from the velocities' difference: p_inf / 4 of its rounding reaches the pressure)
    const f2 cub = (0.25f * ((unR - unL) * im)) * (-3.f + fma2(m2, m1, q3)), sup = -1.f + (DL + DR);
    const f2 Dm1 = {pLx && pRx ? cub.x : sup.x, pLy && pRy ? cub.y : sup.y};
    if (PRE) {
      const f2 dep = fma2(c.R, Dm1, fma2(-0.5f + DL, ppL, (-0.5f + DR) * ppR)), mean = 0.5f * (ppL + ppR);
      const f2 sc = cs * icb;
      ph = fma2(f2{low_x ? sc.x : 1.f, low_y ? sc.y : 1.f}, dep, mean);
    } else {
      ph = fma2(c.R, Dm1, fma2(DL, ppL, DR * ppR));
    }
  }
  F[0] = mL + mR;
  F[1] = fma2(mL, unL, fma2(mR, unR, ph));
  F[2] = fma2(mL, utL, mR * utR);
  F[3] = fma2(mL, HL, mR * HR);
}

// ---------------------------------------------------------------------------
// Fused residual + stage update in FP32 perturbation form, same tiling as
// the FP64 kernel.  Stage 3 accumulates U^{n+1} in FP64 and refreshes the
// FP32 mirror of U^{n+1}.
// ---------------------------------------------------------------------------
// A block is 128 threads on a 16 x 16 tile, every thread with one reconstruction item, two or three flux items of two
// faces and two cells.  The stage was bound by issue slots (86% busy, 1303 thread instructions per cell at
// 3072 x 1536); packed arithmetic took it to about 840.  256 threads with half of them idle in the reconstruction left
// too few warps (3072 x 1536, four steps: 3.31 ms; scalar 3.03 ms; 128 threads, seven blocks per SM 2.95 ms).  With the
// faces' values free of bank conflicts, the update's operands read ahead of its barrier and stores, and the lists in
// the face storage (eight blocks of 27.5 KB per SM) it is 2.56 ms: issue slots 71% busy, FP32 pipe 57%, the rest the
// phases' barriers.
constexpr int NTH = 128;
// A wide block is 288 threads on the same tile: one pair of cells, half a reconstruction item, one pair of faces (there
// are 272) and one cell each, for a chain less than half as long, three blocks per SM at 72 registers.  It serves grids
// of few tiles (ibm__stage_wide, ibm__dual_wide).
constexpr int WIDE = 288, WIDE_BLOCKS = 3;
// Blocks of 128 threads of the block-table kernels per SM: 16 requests 11.3 ms, with seven (72 registers) 11.6, with six
// (80) 11.4; explicit tables of few tiles take six (ibm__batch_blocks)
constexpr int BATCH_BLOCKS = 8, BATCH_FEW = 6;
constexpr int TX = STAGE_TILE, TY = STAGE_TILE, HX = TX + 2 * NG, HY = TY + 2 * NG;
// Shared memory is laid out for pairs: a thread reconstructs two adjacent rows (x direction) or columns (y direction)
// and forms the fluxes of their two faces with packed arithmetic.  The face values of a direction are [variable][face
// along the line][line], the two lines of a pair adjacent (8-byte accesses), the eight pairs of a face permuted by the
// face's number (face_slot): reads and writes of a face's pairs, of two faces, and of one line along the faces (the
// stage update) all fall in different banks.  VP is the pitch of the cell planes: with 498, the reads of
// 8 row pairs x 2 halves x 2 variables fall in 32 banks.
constexpr int FP = TX, NF1 = (TX + 1) * FP, NFD = 4 * NF1;  // one variable's, one direction's and side's face values
constexpr int VP = 498;
static_assert(TX == TY && VP >= HY * HX && VP % 2 == 0 && HX % 2 == 0, "pairs are 8-byte aligned");
constexpr int RB_MAX = 192;  // IB / ghost nodes a body tile's loaded region may hold

// Shared memory of one tile.  face holds, in turn: the TMA box of the tile's
// stage input, the stencils of the region's IB / ghost nodes (body tiles),
// the WENO face states, the face fluxes; each use ends behind a barrier
// before the next begins.
struct TileSmem {
  alignas(128) float face[4 * NFD];  // x left, x right, y left, y right
  alignas(8) float q[5][VP];         // rho', u, v, p', T' of the loaded region, HY x HX each
  unsigned long long mbar;
  unsigned int mbar_phase;  // persistent kernel: parity of the barrier's next phase (barrier initialised once)
  // float offset of line l (a pair's first if even) of face f of a variable
  static __device__ __forceinline__ int face_slot(int f, int l) { return f * FP + (l ^ (f & 14)); }
  // body tiles: cell and stencil of the listed nodes, in the face storage behind the TMA box and the stencils; IB nodes
  // from slot 0 up, ghost nodes from the last slot down
  __device__ __forceinline__ int *rbm() { return reinterpret_cast<int *>(face) + RB_MAX * (int)sizeof(RStencil32) / 4; }
  __device__ __forceinline__ int *rbe() { return rbm() + RB_MAX; }
  float wm[7];    // wall velocity and acceleration at the stage time; 1 if Eq. 7 applies (else 0); the rotation
                  // rate and its rate of change of a pitching body (else 0)
  float lred[WIDE / 32];  // per-warp maxima of the CFL reduction
  int nrb[2];     // listed IB and ghost nodes (body tiles)
};
static_assert(RB_MAX * (sizeof(RStencil32) + 2 * sizeof(int)) <= sizeof(float) * 4 * NFD, "node stencils fit the face storage");

// ---------------------------------------------------------------------------
// TMA staging of a tile (Blackwell bulk tensor copy, inline PTX).  The FP32
// arrays are 3-D tensors (padded column, padded row, variable plane); the
// loaded region of an interior tile is the box of TMA_W x HY x 4 floats at
// padded (i0, j0, 0) -- i0 is a multiple of the tile width, so the copy
// starts on a 64-byte boundary.  One elected thread arms an mbarrier with the
// box's byte count and issues the copy; the block waits on the barrier.
// ---------------------------------------------------------------------------
constexpr int TMA_W = (HX + 3) / 4 * 4;  // box width: HX rounded up to a multiple of 16 bytes
constexpr unsigned TMA_BYTES = 4u * HY * TMA_W * sizeof(float);
// a tile's copy completes within microseconds; a wait gives up after about a second of %globaltimer (the
// iteration count is only a backstop: the time a try_wait suspends is implementation-defined)
constexpr unsigned long long TMA_WAIT_NS = 1ull << 30;
constexpr unsigned TMA_WAIT_BACKSTOP = 1u << 28;

__device__ __forceinline__ unsigned smem_u32(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void tma_init(unsigned long long *mbar) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(mbar)) : "memory");
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

// arm the (initialised) barrier with the box's byte count and issue the copy
__device__ __forceinline__ void tma_load(float *dst, const CUtensorMap *map, int x, int y, unsigned long long *mbar) {
  const unsigned m = smem_u32(mbar);
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(m), "r"(TMA_BYTES) : "memory");
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];" ::
          "r"(smem_u32(dst)),
      "l"((unsigned long long)map), "r"(x), "r"(y), "r"(0), "r"(m)
      : "memory");
}

__device__ __forceinline__ unsigned long long globaltimer_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// wait for the completion of the barrier's phase with the given parity; false if it has not completed within
// TMA_WAIT_NS
__device__ __forceinline__ bool tma_wait(unsigned long long *mbar, unsigned parity) {
  const unsigned m = smem_u32(mbar);
  unsigned long long t0 = 0;
  for (unsigned it = 0; it < TMA_WAIT_BACKSTOP; it++) {
    unsigned ok;
    asm volatile(
        "{ .reg .pred p; mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }"
        : "=r"(ok)
        : "r"(m), "r"(parity)
        : "memory");
    if (ok) return true;
    if ((it & 63) == 0) {
      const unsigned long long t = globaltimer_ns();
      if (it == 0) t0 = t;
      else if (t - t0 > TMA_WAIT_NS) return false;
    }
  }
  return false;
}

// spectral radius of the CFL rule for one cell of the FP32 mirror
__device__ __forceinline__ float cfl_lambda(const Consts &k, const PertConsts &c, const float m[4]) {
  float u, v, pp, Tp;
  pert_prim(c, m[0], m[1], m[2], m[3], u, v, pp, Tp);
  const float r = __fadd_rn(1.f, m[0]);  // as pert_prim has it: one reciprocal
  const float cs = sqrtf(c.gamma * (c.R + pp) / r);
  return (fabsf(u) + cs) * c.idx + (fabsf(v) + cs) * c.idy + c.vis / r;
}

// block maximum of lam (all threads call), then the grid-wide maximum and
// dt through the last-block pattern
template <int NT>
__device__ __forceinline__ void cfl_block_max(const Consts &k, float lam, float *red, DevState *ds,
                                              unsigned int nblocks, bool defer) {
  for (int off = 16; off > 0; off >>= 1) lam = fmaxf(lam, __shfl_xor_sync(0xffffffffu, lam, off));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = lam;
  __syncthreads();
  if (threadIdx.x == 0) {
    float m = red[0];
    for (int w = 1; w < NT / 32; w++) m = fmaxf(m, red[w]);
    atomicMax(&ds->lmax_bits, (unsigned long long)__double_as_longlong((double)m));
    finish_cfl(k, ds, nblocks, defer);
  }
}

// cells the flux update advances: fluid cells, and IB nodes when the ghost layers alone impose the wall
__device__ __forceinline__ bool advanced(const Consts &k, uint8_t t) { return t == FLUID || (k.ib_advance && t == IB); }

// load of a value that other blocks of the same launch may have written (CG:
// through L2, never the non-coherent read-only path)
template <bool CG, class T>
__device__ __forceinline__ T ld_stage(const T *p) {
  if (CG) return __ldcg(p);
  return *p;
}

// ---------------------------------------------------------------------------
// IB / ghost reconstruction (Sec. 4.4-4.6, Eq. 4-8; Sec. 5) evaluated while a
// tile is loaded.  Values are primitives (p', u, v, T').  A ghost node's
// image point may use IB nodes, which are rebuilt from their own stencils
// (their corners are fluid): a body tile rebuilds all IB nodes of its loaded
// region, then all ghost nodes, reading corners from shared memory and only
// corners outside the region from the stage input.
// ---------------------------------------------------------------------------
template <bool CG = false>
__device__ __forceinline__ void raw_prim(const PertConsts &c, const float *U, long long id, long long P,
                                         float q[4]) {
  float u, v, pp, Tp;
  pert_prim(c, ld_stage<CG>(U + id), ld_stage<CG>(U + id + P), ld_stage<CG>(U + id + 2 * P),
            ld_stage<CG>(U + id + 3 * P), u, v, pp, Tp);
  q[0] = pp;
  q[1] = u;
  q[2] = v;
  q[3] = Tp;
}

__device__ __forceinline__ void wall_bc(const PertConsts &c, const RStencil32 &s, const float qp[4], const float *wm,
                                        float q[4]) {
  // wm = (Vx, Vy, Ax, Ay, supersonic, omega, domega/dt) at the stage time: the wall's motion at P' is the
  // body's translation plus, for a pitching body, omega x r and domega/dt x r - omega^2 r with r = P' - pivot
  // (zero terms otherwise).  Neumann pressure dp/dn = rho G (Eq. 5-6), G = -n.a plus the centripetal
  // u_t^2 kappa of Eq. 7 (u_t tangential to the wall, relative to it, at the probe); with rho = p / (R T) and
  // T fixed along the normal (Eq. 8) it integrates to p = p_probe exp(-dxi G / (R T)), here in perturbation
  // form p' = p'_probe + (R + p'_probe) expm1(...) so that p' keeps its digits
  const float om = wm[5], al = wm[6];
  const float Vx = wm[0] - om * s.ry, Vy = wm[1] + om * s.rx;
  const float Ax = wm[2] - al * s.ry - om * om * s.rx, Ay = wm[3] + al * s.rx - om * om * s.ry;
  float G = -(s.nx * Ax + s.ny * Ay);
  if (wm[4] != 0.f) {
    const float ut = -(qp[1] - Vx) * s.ny + (qp[2] - Vy) * s.nx;
    G = G + ut * ut * s.curv;
  }
  // (static body: G = 0 and p'_node = p'_probe exactly, without the exponential)
  q[0] = G != 0.f ? qp[0] + (c.R + qp[0]) * expm1f(-s.dxi * G / (c.R * (1.f + qp[3]))) : qp[0];
  q[1] = Vx + (qp[1] - Vx) * s.ratio;
  q[2] = Vy + (qp[2] - Vy) * s.ratio;
  q[3] = qp[3];
}

// The quadratic form (Sec. 4.5, Sec. 5; IBM_INTERP_QUADRATIC) of wall_bc: quadratics in the distance along the
// normal through the wall condition and the probes' values qp (first) and qb (second) -- the Lagrange weights
// for the Dirichlet velocity, zero wall slope for T', wall slope rho G for p' with the first probe's density --
// in perturbation form (differences of perturbations are differences of the variables)
__device__ __forceinline__ void wall_bc_quad(const PertConsts &c, const RStencil32 &s, const RStencilQ &t,
                                             const float qp[4], const float qb[4], const float *wm, float q[4]) {
  const float om = wm[5], al = wm[6];
  const float Vx = wm[0] - om * s.ry, Vy = wm[1] + om * s.rx;
  const float Ax = wm[2] - al * s.ry - om * om * s.rx, Ay = wm[3] + al * s.rx - om * om * s.ry;
  float G = -(s.nx * Ax + s.ny * Ay);
  if (wm[4] != 0.f) {
    const float ut = -(qp[1] - Vx) * s.ny + (qp[2] - Vy) * s.nx;
    G = G + ut * ut * s.curv;
  }
  const float b = (c.R + qp[0]) / (c.R * (1.f + qp[3])) * G;
  q[0] = qp[0] + (qb[0] - qp[0]) * t.m + b * t.dq;
  q[1] = Vx + (qp[1] - Vx) * t.L1 + (qb[1] - Vx) * t.L2;
  q[2] = Vy + (qp[2] - Vy) * t.L1 + (qb[2] - Vy) * t.L2;
  q[3] = qp[3] + (qb[3] - qp[3]) * t.m;
}

// An IB node outside a tile's loaded region, rebuilt from its own stencil (QUAD: and its second probe)
template <bool CG, bool QUAD = false>
static __device__ __noinline__ void rebuild_ib(const Consts &k, const PertConsts &c, const float *U,
                                               const RStencil32 &s, const RStencilQ *t, const float *wm,
                                               float q[4]) {
  float qp[4] = {0.f, 0.f, 0.f, 0.f};
  float raw[4][4];  // the corners' loads in flight together (bits 0-3 of the mask: valid corners; bit 4: IB node)
#pragma unroll
  for (int b = 0; b < 4; b++)
#pragma unroll
    for (int v = 0; v < 4; v++)
      raw[b][v] = s.mask >> b & 1 ? ld_stage<CG>(U + s.corner + (b & 1) + (b >> 1) * k.pitch + v * k.plane) : 0.f;
#pragma unroll
  for (int b = 0; b < 4; b++) {
    if (!(s.mask >> b & 1)) continue;
    float cq[4];
    pert_prim(c, raw[b][0], raw[b][1], raw[b][2], raw[b][3], cq[1], cq[2], cq[0], cq[3]);
    for (int v = 0; v < 4; v++) qp[v] += s.w[b] * cq[v];
  }
  if (QUAD && t->mask) {
    float qb[4] = {0.f, 0.f, 0.f, 0.f};
    for (int b = 0; b < 4; b++) {
      if (!(t->mask >> b & 1)) continue;
      float cq[4];
      raw_prim<CG>(c, U, t->corner + (b & 1) + (b >> 1) * k.pitch, k.plane, cq);
      for (int v = 0; v < 4; v++) qb[v] += t->w[b] * cq[v];
    }
    wall_bc_quad(c, s, *t, qp, qb, wm, q);
  } else {
    wall_bc(c, s, qp, wm, q);
  }
}

// ---------------------------------------------------------------------------
// Fused residual + stage update in FP32 perturbation form.  One 16x16 tile
// per block.  (1) Load tile + 3-cell halo: domain halos by index mapping, IB
// and ghost nodes rebuilt on the fly, conversion to (rho', u, v, p', T') in
// shared memory.  (2) WENO5 per cell and direction: the three smoothness
// indicators of a cell's five-point window serve both the left state of its
// right face and the right state of its left face.  (3) LDFSS + central
// viscous flux per face.  (4) Flux divergence and SSP-RK3 stage update;
// stage 3 accumulates U^{n+1} in FP64.
// ---------------------------------------------------------------------------
// blk: the block's index within this case's launch (plain: tile index; body:
// slot in the body-tile list).  Every thread of the block calls it.
// DUAL: a pseudo stage of dual time -- preconditioned faces, wall motion at
// t + dt_phys, FP64 point-implicit update (dp; D holds the sub-iteration's
// start, Out receives the FP32 mirror of the new iterate).
// TMA: the kernel may stage interior tiles with a tensor copy (tmap: tensor
// map of In; NULL loads every tile with per-thread loads).
// PERSIST: the tile's stage inside the persistent step kernel -- blk is the
// tile itself; In, D and the stage arrays may have been written by other
// blocks of the same launch (coherent loads); stage times come from t and dt,
// which stay fixed during the launch; the step's end (t, step count) and the
// next dt are left to the kernel.
// sm: the block's shared memory.
// TVD: the second-order TVD reconstruction in place of WENO5 (Sec. 2), compiled into its own kernels so that
// the WENO5 kernels carry no branch for it.
template <int STAGE, bool BODY, bool DUAL = false, bool TMA = false, bool PERSIST = false, bool TVD = false,
          bool QUAD = false, int NT = NTH>
__device__ __forceinline__ void stage_tile(const Consts &k, const PertConsts &c, float *Mn,
                                           const float *__restrict__ In, float *Out, double *D,
                                           const uint8_t *__restrict__ tag,
                                           const int *__restrict__ sid, const RStencil32 *__restrict__ rs,
                                           const uint8_t *__restrict__ tile_body, const int *__restrict__ body_tiles,
                                           DevState *ds, bool fuse_cfl, unsigned int ncfl, int blk, TileSmem &sm,
                                           const DualPtrs &dp = DualPtrs{}, const CUtensorMap *tmap = nullptr,
                                           const RStencilQ *__restrict__ rsq = nullptr) {
  static_assert(NT == NTH || NT == WIDE, "threads of a block");
  constexpr int CROWS = NT / TX, CELLS = (TY + CROWS - 1) / CROWS;  // rows between a thread's cells, cells it updates
  static_assert(!TMA || 4 * HY * TMA_W <= RB_MAX * (int)sizeof(RStencil32) / 4, "TMA box ahead of the listed nodes");
  float *s_face = sm.face;
  unsigned long long &s_mbar = sm.mbar;
  auto sq = [&sm](int v, int b, int a) -> float & { return sm.q[v][b * HX + a]; };
  float(*s_raw)[HY][TMA_W] = reinterpret_cast<float(*)[HY][TMA_W]>(s_face);  // TMA box
  float *wm = sm.wm;
  float *lred = sm.lred;
  const int ntx = (k.nx + TX - 1) / TX;
  // every block reads dt before any block can finish the fused CFL reduction
  const double dtd = ds->dt;
  const float dt = ds->dtf;
  int tile;
  if (PERSIST) {
    tile = blk;
  } else if (BODY) {
    tile = blk < ds->nbody_tiles ? body_tiles[blk] : -1;
  } else {
    tile = blk;
    if (!DUAL && blk == 0 && threadIdx.x == 0) {
      if (STAGE == 1) {  // stage times for the body kernels of stages 2 and 3
        ds->tst[0] = ds->t + dtd;
        ds->tst[1] = ds->t + 0.5 * dtd;
      } else if (STAGE == 3) {  // end of the step; the body kernel of stage 3 reads tst, not t
        ds->t = ds->t + dtd;
        ds->steps += 1;
      }
    }
  }
  // plain launch: a listed tile is left to its body block; its tags are on their way before the answer is known
  const bool listed = !PERSIST && !BODY && tile_body[blk];
  if (BODY && tile < 0) {
    if (STAGE == 3 && fuse_cfl && threadIdx.x == 0) finish_cfl(k, ds, ncfl, PERSIST);
    return;
  }
  const int i0 = (tile % ntx) * TX, j0 = (tile / ntx) * TY;
  const int tx = threadIdx.x % TX, ty0 = threadIdx.x / TX;  // the thread's cells: rows ty0, ty0 + CROWS, ...
  uint8_t tags[CELLS];
  bool work = false;
#pragma unroll
  for (int h = 0; h < CELLS; h++) {
    const int ci = i0 + tx, cj = j0 + ty0 + h * CROWS;
    const bool in = (NT == NTH || ty0 < TY) && ci < k.nx && cj < k.ny;  // (wide: threads beyond the tile's cells)
    tags[h] = in ? tag[cj * k.nx + ci] : (uint8_t)SOLID;
    // stages 1 and 3 also keep the IB / ghost nodes of U^n current; stage 2 only needs the cells it advances
    work |= STAGE == 2 ? advanced(k, tags[h]) : tags[h] != SOLID;
  }
  // interior tile (the loaded region needs no domain mapping): one tensor copy stages it,
  // issued before the tags are read
  const bool interior = i0 >= NG && j0 >= NG && i0 + TX + NG <= k.nx && j0 + TY + NG <= k.ny;
  const bool tma = TMA && tmap != nullptr && interior;
  if (listed) {
    if (STAGE == 3 && fuse_cfl && threadIdx.x == 0) finish_cfl(k, ds, ncfl, PERSIST);
    return;
  }
  if (TMA && tma && threadIdx.x == 0) {
    if (PERSIST) {
      // the box may hold values other blocks of this launch wrote: order the tensor copy after them
      asm volatile("fence.proxy.async.global;" ::: "memory");
    } else {
      tma_init(&s_mbar);
    }
    tma_load(s_face, tmap, i0, j0, &s_mbar);
  }
  if (!__syncthreads_or(work)) {
    if (TMA && tma && threadIdx.x == 0) {  // the copy on its way still writes the box
      if (!tma_wait(&s_mbar, PERSIST ? sm.mbar_phase : 0u)) atomicOr(&ds->err, ERR_TIMEOUT);
      if (PERSIST) sm.mbar_phase ^= 1u;
    }
    if (STAGE == 3 && fuse_cfl && threadIdx.x == 0) finish_cfl(k, ds, ncfl, PERSIST);
    return;
  }
  // L2 prefetch of the operands the stage update reads at the end of the tile (the mirror of U^n; the stage
  // input; the FP64 master at stage 3): one line per tile row and plane, issued before the tile's arithmetic
  // so that those reads find L2 rather than DRAM after the L2 has turned over
  if (!DUAL && threadIdx.x < 4 * TY) {
    const int r = threadIdx.x % TY, v = threadIdx.x / TY;
    if (j0 + r < k.ny) {
      const long long o = cidx(k, i0, j0 + r) + v * k.plane;
      asm volatile("prefetch.global.L2 [%0];" ::"l"(Mn + o));
      if (STAGE >= 2) asm volatile("prefetch.global.L2 [%0];" ::"l"(In + o));
      if (STAGE == 3) {
        asm volatile("prefetch.global.L2 [%0];" ::"l"(D + o));
        asm volatile("prefetch.global.L2 [%0];" ::"l"(D + o + 8));
      }
    }
  }
  if (BODY && threadIdx.x == 0) {
    double X[2], V[2], Acc[2];
    const double ts = DUAL ? ds->t + k.dt_phys
                           : (PERSIST ? stage_time(ds, STAGE) : (STAGE == 1 ? ds->t : ds->tst[STAGE - 2]));
    body_motion(k, ds, ts, X, V, Acc);
    wm[0] = (float)V[0];
    wm[1] = (float)V[1];
    wm[2] = (float)Acc[0];
    wm[3] = (float)Acc[1];
    wm[4] = supersonic_motion(k, V) ? 1.f : 0.f;
    double th = 0.0, om = 0.0, al = 0.0;
    if (k.motion.kind == IBM_MOTION_PITCH) pitch_at(k.motion, ts, &th, &om, &al);
    wm[5] = (float)om;
    wm[6] = (float)al;
  }
  // body tiles: the listed nodes of the thread's cells, on their way while the copy is
  int esid[(HX * HY / 2 + NT - 1) / NT][2];
  if (BODY && interior) {
#pragma unroll
    for (int r = 0; r < (HX * HY / 2 + NT - 1) / NT; r++) {
      const int m = min((int)threadIdx.x + r * NT, HX * HY / 2 - 1), b = m / (HX / 2), a = 2 * (m - b * (HX / 2));
      const int *ps = sid + (j0 - NG + b) * k.nx + i0 - NG + a;
      esid[r][0] = ps[0];
      esid[r][1] = ps[1];
    }
  }
  __syncthreads();
  if (TMA && tma) {
    const unsigned parity = PERSIST ? sm.mbar_phase : 0u;
    if (__syncthreads_or(!tma_wait(&s_mbar, parity))) {
      // the copy has not completed and may still write the box: wait for it once more (bounded), then leave
      // the tile without touching shared memory or outputs.  The step's state is invalid; the error flag makes
      // the next synchronising call report it.
      if (threadIdx.x == 0) {
        atomicOr(&ds->err, ERR_TIMEOUT);
        tma_wait(&s_mbar, parity);
        if (STAGE == 3 && fuse_cfl) finish_cfl(k, ds, ncfl, PERSIST);
      }
      return;
    }
  }

  const long long P = k.plane;
  // body tiles: every IB / ghost node of the loaded region, with its stencil staged in shared memory (in the
  // face storage, after the TMA box has been consumed)
  int *s_nrb = sm.nrb;
  int *s_rbm = sm.rbm(), *s_rbe = sm.rbe();
  RStencil32 *s_rs = reinterpret_cast<RStencil32 *>(s_face);
  if (BODY && threadIdx.x < 2) s_nrb[threadIdx.x] = 0;
  const int nib_all = BODY ? ds->offset[1] : 0;  // the case's list holds its IB nodes first
  if (BODY) __syncthreads();
  // a listed node of the loaded region (body tiles), by class: each pass of the rebuild then takes its own nodes only
  auto list_node = [&](int m, int e) {
    if (e < 0) return;
    const int ghost = e >= nib_all, n = atomicAdd(&s_nrb[ghost], 1);
    if (n < RB_MAX) {
      const int slot = ghost ? RB_MAX - 1 - n : n;
      s_rbm[slot] = m;
      s_rbe[slot] = e;
    }
  };
  if (interior) {  // no domain mapping: two cells at a time, from the tensor copy's box or from memory
    constexpr int NC = (HX * HY / 2 + NT - 1) / NT;
#pragma unroll
    for (int r = 0; r < NC; r++) {
      const int m = threadIdx.x + r * NT, b = m / (HX / 2), a = 2 * (m - b * (HX / 2));
      if (m >= HX * HY / 2) break;
      f2 w[4], u, v, pp, Tp;
      if (TMA && tma) {
        for (int q = 0; q < 4; q++) w[q] = ld2(&s_raw[q][b][a]);
      } else {
        const float *p = In + cidx(k, i0 - NG + a, j0 - NG + b);  // an even column of the padded row
        for (int q = 0; q < 4; q++) {
          const float2 t = ld_stage<PERSIST>(reinterpret_cast<const float2 *>(p + q * P));
          w[q] = f2{t.x, t.y};
        }
      }
      pert_prim2(c, w[0], w[1], w[2], w[3], u, v, pp, Tp);
      float *o = &sm.q[0][b * HX + a];
      st2(o, w[0]);
      st2(o + VP, u);
      st2(o + 2 * VP, v);
      st2(o + 3 * VP, pp);
      st2(o + 4 * VP, Tp);
      if (BODY) {
        list_node(b * HX + a, esid[r][0]);
        list_node(b * HX + a + 1, esid[r][1]);
      }
    }
  } else {
    // every load of the thread's cells before the first use
    constexpr int NC = (HX * HY + NT - 1) / NT;
    float w[NC][4];
    int e[NC];
#pragma unroll
    for (int r = 0; r < NC; r++) {
      const int m = threadIdx.x + r * NT;
      int gi = i0 - NG + m % HX, gj = j0 - NG + m / HX;
      const bool in = m < HX * HY && halo_map(k, gi, gj);
      const float *p = In + cidx(k, gi, gj);
      e[r] = BODY && in ? sid[gj * k.nx + gi] : -1;
#pragma unroll
      for (int q = 0; q < 4; q++) w[r][q] = in ? ld_stage<PERSIST>(p + q * P) : 0.f;  // free stream: zero perturbation
    }
    static_assert(NC % 2 == 0, "converted two at a time");
#pragma unroll
    for (int r = 0; r < NC; r += 2) {
      f2 u, v, pp, Tp;
      pert_prim2(c, f2{w[r][0], w[r + 1][0]}, f2{w[r][1], w[r + 1][1]}, f2{w[r][2], w[r + 1][2]},
                 f2{w[r][3], w[r + 1][3]}, u, v, pp, Tp);
#pragma unroll
      for (int s = 0; s < 2; s++) {
        const int m = threadIdx.x + (r + s) * NT;
        if (m >= HX * HY) break;
        float *o = &sm.q[0][m];
        o[0] = w[r + s][0];
        o[VP] = s ? u.y : u.x;
        o[2 * VP] = s ? v.y : v.x;
        o[3 * VP] = s ? pp.y : pp.x;
        o[4 * VP] = s ? Tp.y : Tp.x;
        if (BODY) list_node(m, e[r + s]);
      }
    }
  }
  __syncthreads();
  // every thread has waited on this phase: the next tile's copy completes the other parity
  if (PERSIST && TMA && tma && threadIdx.x == 0) sm.mbar_phase ^= 1u;
  if (BODY) {
    const int nib = min(s_nrb[0], RB_MAX), ngh = min(s_nrb[1], RB_MAX - nib);
    for (int r = threadIdx.x; r < nib + ngh; r += NT) {
      const int slot = r < nib ? r : RB_MAX - 1 - (r - nib);
      s_rs[slot] = rs[s_rbe[slot]];
    }
    __syncthreads();
    // rebuild the listed nodes in place: IB nodes, barrier, ghost nodes (whose image points may use IB
    // nodes); corners inside the loaded region come from shared memory
    // four lanes per node, one stencil corner each, so that corners outside the loaded region (chains of
    // dependent global loads) overlap; the node's first lane sums the corners in stencil order
    for (int pass = k.ib_advance ? 1 : 0; pass < 2; pass++) {  // IB nodes (pass 0) unless advanced
      const int np = pass == 0 ? nib : ngh;
      for (int t0 = 0; t0 < 4 * np; t0 += NT) {  // block-uniform: every lane takes part in the shuffles
        const int t = (t0 + (int)threadIdx.x) >> 2, cq = threadIdx.x & 3, r = pass == 0 ? t : RB_MAX - 1 - t;
        const bool listed_node = t < np;
        bool node = false;
        float v4[4] = {0.f, 0.f, 0.f, 0.f};
        if (listed_node) {
          const RStencil32 &st = s_rs[r];
          node = (st.mask & 15) != 0;
          if (node && (st.mask >> cq & 1)) {
            const int cn = st.ccell + (cq & 1) + (cq >> 1) * k.nx;
            const int la = cn % k.nx - (i0 - NG), lb = cn / k.nx - (j0 - NG);
            if (la >= 0 && la < HX && lb >= 0 && lb < HY) {
              v4[0] = sq(3, lb, la);
              v4[1] = sq(1, lb, la);
              v4[2] = sq(2, lb, la);
              v4[3] = sq(4, lb, la);
            } else {
              // corner outside the loaded region: fluid value, or an IB node rebuilt from its own stencil
              const int e2 = pass == 1 ? sid[cn] : -1;
              if (!k.ib_advance && e2 >= 0 && (rs[e2].mask & 15))
                rebuild_ib<PERSIST, QUAD>(k, c, In, rs[e2], QUAD ? rsq + e2 : nullptr, wm, v4);
              else raw_prim<PERSIST>(c, In, st.corner + (cq & 1) + (cq >> 1) * k.pitch, P, v4);
            }
          }
        }
        // quadratic form: the same lane also takes its corner of the second probe's square
        const RStencilQ *tq = nullptr;
        float v4b[4] = {0.f, 0.f, 0.f, 0.f};
        if (QUAD && node) {
          tq = rsq + s_rbe[r];
          if (tq->mask >> cq & 1) {
            const int cn = tq->ccell + (cq & 1) + (cq >> 1) * k.nx;
            const int la = cn % k.nx - (i0 - NG), lb = cn / k.nx - (j0 - NG);
            if (la >= 0 && la < HX && lb >= 0 && lb < HY) {
              v4b[0] = sq(3, lb, la);
              v4b[1] = sq(1, lb, la);
              v4b[2] = sq(2, lb, la);
              v4b[3] = sq(4, lb, la);
            } else {
              const int e2 = pass == 1 ? sid[cn] : -1;
              if (!k.ib_advance && e2 >= 0 && (rs[e2].mask & 15))
                rebuild_ib<PERSIST, QUAD>(k, c, In, rs[e2], rsq + e2, wm, v4b);
              else raw_prim<PERSIST>(c, In, tq->corner + (cq & 1) + (cq >> 1) * k.pitch, P, v4b);
            }
          }
        }
        const int lane0 = (int)(threadIdx.x & 31) & ~3;
        float qp[4] = {0.f, 0.f, 0.f, 0.f};
        const unsigned int mask = listed_node ? (unsigned int)s_rs[r].mask : 0u;
        for (int j = 0; j < 4; j++) {
          const float wj = listed_node ? s_rs[r].w[j] : 0.f;
          for (int v = 0; v < 4; v++) {
            const float x = __shfl_sync(0xffffffffu, v4[v], lane0 + j);
            if (mask >> j & 1) qp[v] += wj * x;
          }
        }
        float qb[4] = {0.f, 0.f, 0.f, 0.f};
        if (QUAD) {
          const unsigned int maskb = tq ? (unsigned int)tq->mask : 0u;
          for (int j = 0; j < 4; j++) {
            const float wj = tq ? tq->w[j] : 0.f;
            for (int v = 0; v < 4; v++) {
              const float x = __shfl_sync(0xffffffffu, v4b[v], lane0 + j);
              if (maskb >> j & 1) qb[v] += wj * x;
            }
          }
        }
        if (!node || cq != 0) continue;
        const RStencil32 &st = s_rs[r];
        const int m = s_rbm[r], a = m % HX, b = m / HX;
        float q[4];
        if (QUAD && tq->mask) wall_bc_quad(c, st, *tq, qp, qb, wm, q);
        else wall_bc(c, st, qp, wm, q);
        sq(0, b, a) = (q[0] - c.R * q[3]) / (c.R * (1.f + q[3]));
        sq(1, b, a) = q[1];
        sq(2, b, a) = q[2];
        sq(3, b, a) = q[0];
        sq(4, b, a) = q[3];
        const bool own = a >= NG && a < NG + TX && b >= NG && b < NG + TY;
        if (own && STAGE == 1) {  // U^n on this node for output and for a node that turns fluid
          float d0, d1, d2, d3;
          prim_pert(c, q[0], q[1], q[2], q[3], d0, d1, d2, d3);
          D[st.cell] = d0;
          D[st.cell + P] = d1;
          D[st.cell + 2 * P] = d2;
          D[st.cell + 3 * P] = d3;
        }
      }
      __syncthreads();
    }
    if (threadIdx.x == 0 && s_nrb[0] + s_nrb[1] > RB_MAX) atomicOr(&ds->err, ERR_CAPACITY);
  }
  // WENO5 (Sec. 2) along lines: an item is one variable of a pair of adjacent interior tile rows (x) or columns (y)
  // and one of its two halves -- nine consecutive window centres, local 2..10 or 11..19, the cells whose faces the
  // tile needs.  The smoothness indicators are written with the second differences d2 and first differences g of the
  // line, beta_0 = 13/12 d2(c-1)^2 + 1/4 (d2(c-1) + 2 g(c-1))^2, beta_1 = 13/12 d2(c)^2 + 1/4 (g(c-1) + g(c))^2,
  // beta_2 = 13/12 d2(c+1)^2 + 1/4 (d2(c+1) - 2 g(c))^2 with g(j) = f(j+1) - f(j), so that each centre loads one
  // value and forms one new squared second difference, shared by three windows.  The three candidate
  // polynomials and the nonlinear weights of a window give the left state at its right face and, mirrored, the
  // right state at its left face.
  // Every operation of the window is one packed instruction for both lines (40 and 4 reciprocals for 4 face states),
  // and the results are stored as pairs.
  static_assert(TX == 16 && TY == 16, "items: 2 directions x 4 variables x 2 halves x 8 line pairs");
  // Wide blocks break each half in two (five and four centres), for a chain of half the length.
  constexpr int WN = NT == NTH ? 9 : 5;
  if (NT == NTH || threadIdx.x < 256) {
    const int lp = threadIdx.x & 7, half = threadIdx.x >> 3 & 1, v = threadIdx.x >> 4 & 3, part = threadIdx.x >> 7;
    const bool xdir = (threadIdx.x & 64) == 0;
    const int ls = xdir ? 1 : HX, ps = xdir ? HX : 1;  // strides along the line and between the pair's lines
    const int w0 = 9 * half + 5 * part;                // the item's first window, centred at local w0 + 2
    const float *lp0 = &sm.q[v][xdir ? (NG + 2 * lp) * HX : NG + 2 * lp] + w0 * ls, *lp1 = lp0 + ps;
    // window w gives the left state of face w (between local cells w + 2 and w + 3) and the right state of face w - 1,
    // at face_slot(w, 2 lp), formed from the slot's bits: with two halves w0 is half mod 2
    float *const of = s_face + (xdir ? 0 : 2 * NFD) + v * NF1 + w0 * FP;
    const int slot0 = 2 * lp ^ 8 * half, hp = 2 * half;
    auto store = [&](int i, f2 qL, f2 qR, float *&prev) {
      if constexpr (NT == WIDE) {
        const int w = w0 + i, slot = 2 * lp;
        if (w <= TX) st2(of + i * FP + (slot ^ (w & 14)), qL);
        if (w >= 1) st2(of + (i - 1) * FP + (slot ^ ((w - 1) & 14)) + NFD, qR);
        return;
      }
      float *const p = of + i * FP + (slot0 ^ (i & 1 ? (i & 14) + hp : i & 14));
      if (i < 8 || half == 0) st2(p, qL);
      if (i > 0) st2(prev + NFD, qR);
      else if (half == 1) st2(of - FP + (2 * lp ^ 8) + NFD, qR);  // face 8
      prev = p;
    };
    float *prev = nullptr;
    if (TVD) {
      // the second-order TVD scheme (Sec. 2): MUSCL with the minmod limiter over the same items; differences
      // of perturbations equal differences of the variables, so the limiter sees what it would in absolute form
      f2 f1 = {lp0[ls], lp1[ls]}, f2c = {lp0[2 * ls], lp1[2 * ls]};
      auto minmod = [](float a, float b) {
        float m = 0.f;
        if (a > 0.f && b > 0.f) m = a < b ? a : b;
        else if (a < 0.f && b < 0.f) m = a > b ? a : b;
        return m;
      };
#pragma unroll
      for (int i = 0; i < WN; i++) {
        if (NT == WIDE && i == 4 && part == 1) break;  // the second part (whole warps) has four windows
        const f2 f3 = {lp0[(i + 3) * ls], lp1[(i + 3) * ls]};
        const f2 a = f2c - f1, b = f3 - f2c;
        // minmod(a, b) for the left state at the right face, minmod(-b, -a) = -minmod(a, b) for the right state
        const f2 m = {minmod(a.x, b.x), minmod(a.y, b.y)};
        store(i, fma2(0.5f, m, f2c), fma2(-0.5f, m, f2c), prev);
        f1 = f2c;
        f2c = f3;
      }
    } else {
      // smoothness indicators e_k = eps + beta_k = [eps + 13/12 d2^2] + (b_k / 2)^2; candidates as differences from
      // the centre value, in x = g / 2 and y = d2 / 6: left (2 y_m + x_m, x_0 - y_c, x_0 - y_p), right (mirrored) minus
      // (x_0 - 2 y_p, x_m + y_c, x_m + y_m), with linear weights (1/6, 1, 1/2); the nonlinear weights d_k / e_k^2
      // cleared of their common denominator (s12 for k = 0, s02, s01)
      const f2 eps = both(1e-6f);
      f2 fa = {lp0[0], lp1[0]}, fb = {lp0[ls], lp1[ls]}, fc = {lp0[2 * ls], lp1[2 * ls]}, fd = {lp0[3 * ls], lp1[3 * ls]};
      f2 gm = fc - fb, g0 = fd - fc;
      f2 dm = gm - (fb - fa), dc = g0 - gm;  // second differences centred at c - 1 and c
      f2 am = fma2((13.f / 12.f) * dm, dm, eps), ac = fma2((13.f / 12.f) * dc, dc, eps);
      f2 xm = 0.5f * gm, x0 = 0.5f * g0, ym = (1.f / 6.f) * dm, yc = (1.f / 6.f) * dc;
#pragma unroll
      for (int i = 0; i < WN; i++) {
        if (NT == WIDE && i == 4 && part == 1) break;  // the second part (whole warps) has four windows
        const f2 fe = {lp0[(i + 4) * ls], lp1[(i + 4) * ls]};
        const f2 g1 = fe - fd, dn = g1 - g0;
        const f2 an = fma2((13.f / 12.f) * dn, dn, eps), yp = (1.f / 6.f) * dn;
        const f2 b0 = fma2(0.5f, dm, gm), b1 = xm + x0, b2 = fma2(-0.5f, dn, g0);
        const f2 e0 = fma2(b0, b0, am), e1 = fma2(b1, b1, ac), e2 = fma2(b2, b2, an);
        const f2 e01 = e0 * e1, e12 = e1 * e2, e02 = e0 * e2;
        const f2 s01 = e01 * e01, s12 = e12 * e12, s02 = e02 * e02;
        const f2 a1 = (1.f / 6.f) * s12, a3 = 0.5f * s01, c1 = (1.f / 6.f) * s01, c3 = 0.5f * s12;
        const f2 nL = fma2(a1, fma2(2.f, ym, xm), fma2(s02, x0 - yc, a3 * (x0 - yp)));
        const f2 nR = fma2(c1, fma2(-2.f, yp, x0), fma2(s02, xm + yc, c3 * (xm + ym)));
        const f2 qL = fma2(nL, rcp2((a1 + s02) + a3), fc), qR = fc - nR * rcp2((c1 + s02) + c3);
        store(i, qL, qR, prev);
        fc = fd;
        fd = fe;
        gm = g0;
        g0 = g1;
        dm = dc;
        dc = dn;
        am = ac;
        ac = an;
        xm = x0;
        x0 = 0.5f * g1;
        ym = yc;
        yc = yp;
      }
    }
  }
  __syncthreads();

  const float mu = c.mu, kap = c.kappa, idx = c.idx, idy = c.idy;
  // an item is the faces of two adjacent rows (x direction) or columns (y direction) at one place of the line
  for (int m = threadIdx.x; m < 2 * (TX + 1) * (TX / 2); m += NT) {
    const bool xdir = m < (TX + 1) * (TX / 2);
    const int mm = xdir ? m : m - (TX + 1) * (TX / 2), f = mm >> 3, l = 2 * (mm & 7);
    float *fl = s_face + (xdir ? 0 : 2 * NFD) + sm.face_slot(f, l);  // left states, then the flux; right states NFD further
    const int n = xdir ? 1 : 2, t = 3 - n;  // variables: velocity along the normal and the tangent
    const float *fn = fl + n * NF1, *ft = fl + t * NF1;
    f2 rL = ld2(fl), unL = ld2(fn), utL = ld2(ft), pL = ld2(fl + 3 * NF1);
    f2 rR = ld2(fl + NFD), unR = ld2(fn + NFD), utR = ld2(ft + NFD), pR = ld2(fl + NFD + 3 * NF1);
    // the first cells of the pair's faces; the second cells are ls further, the other line ps
    const int ls = xdir ? 1 : HX, ps = xdir ? HX : 1;
    const float *qa = &sm.q[0][xdir ? (NG + l) * HX + f + 2 : (f + 2) * HX + NG + l];
    const float *qn = qa + n * VP, *qt = qa + t * VP, *qT = qa + 4 * VP;
    if (!(rL.x > -1.f && rL.y > -1.f && rR.x > -1.f && rR.y > -1.f && pL.x > -c.R && pL.y > -c.R && pR.x > -c.R &&
          pR.y > -c.R)) {  // first-order states on the faces where a density or pressure is not positive
      if (!(rL.x > -1.f) || !(pL.x > -c.R) || !(rR.x > -1.f) || !(pR.x > -c.R)) {
        rL.x = qa[0], unL.x = qn[0], utL.x = qt[0], pL.x = qa[3 * VP];
        rR.x = qa[ls], unR.x = qn[ls], utR.x = qt[ls], pR.x = qa[3 * VP + ls];
      }
      if (!(rL.y > -1.f) || !(pL.y > -c.R) || !(rR.y > -1.f) || !(pR.y > -c.R)) {
        rL.y = qa[ps], unL.y = qn[ps], utL.y = qt[ps], pL.y = qa[3 * VP + ps];
        rR.y = qa[ls + ps], unR.y = qn[ls + ps], utR.y = qt[ls + ps], pR.y = qa[3 * VP + ls + ps];
      }
    }
    const float idn = xdir ? idx : idy, idt = xdir ? idy : idx;
    f2 F[4];  // mass, momentum along the normal and the tangent, energy
    ldfss_pert2<DUAL>(c, rL, unL, utL, pL, rR, unR, utR, pR, xdir ? c.ux : c.uy, xdir ? c.uy : c.ux, F, idn);
    // viscous part from the cells before and after the face, lines (before, first) and (second, after) of the pair:
    // differences along the normal, sums, and differences across the lines of the two cells' sums
    f2 dn[2], av[2], dt2[2];
#pragma unroll
    for (int w = 0; w < 2; w++) {
      const float *q = w ? qt : qn;
      f2 lo0, hi0, lo1, hi1;
      if (xdir) {
        lo0 = f2{q[-HX], q[0]}, hi0 = f2{q[HX], q[2 * HX]};
        lo1 = f2{q[1 - HX], q[1]}, hi1 = f2{q[1 + HX], q[1 + 2 * HX]};
      } else {
        lo0 = ld2(q - 1), hi0 = ld2(q + 1), lo1 = ld2(q + HX - 1), hi1 = ld2(q + HX + 1);
      }
      const f2 lo = lo0 + lo1, hi = hi0 + hi1;
      dt2[w] = hi - lo;
      av[w] = f2{lo.y, hi.x};
      dn[w] = f2{lo1.y, hi1.x} - f2{lo0.y, hi0.x};
    }
    const f2 Tn = f2{qT[ls], qT[ls + ps]} - f2{qT[0], qT[ps]};
    const f2 tnn = fma2((4.f / 3.f) * mu * idn, dn[0], ((-1.f / 6.f) * mu * idt) * dt2[1]);
    const f2 tnt = fma2(0.25f * mu * idt, dt2[0], (mu * idn) * dn[1]);
    const f2 work = 0.5f * fma2(av[0], tnn, av[1] * tnt);
    st2(fl, F[0]);
    st2(fl + n * NF1, F[1] - tnn);
    st2(fl + t * NF1, F[2] - tnt);
    st2(fl + 3 * NF1, F[3] - fma2(kap * idn, Tn, work));
  }
  // the update's operands: read ahead of the barrier and of the stores (which may alias them), all in flight together
  float um[CELLS][4], ui[CELLS][4];
  double ud[CELLS][4];
  if constexpr (!DUAL) {
#pragma unroll
    for (int h = 0; h < CELLS; h++) {
      const bool adv = advanced(k, tags[h]);
      const long long id = cidx(k, i0 + tx, j0 + ty0 + h * CROWS);
#pragma unroll
      for (int v = 0; v < 4; v++) {
        if (adv) um[h][v] = Mn[id + v * P];
        if (STAGE >= 2 && adv) ui[h][v] = ld_stage<PERSIST>(In + id + v * P);
        if (STAGE == 3 && (adv || (BODY && tags[h] != SOLID))) ud[h][v] = ld_stage<PERSIST>(D + id + v * P);
      }
    }
  }
  __syncthreads();

  float lam = 0.f;
#pragma unroll(DUAL ? 1 : CELLS)
  for (int h = 0; h < CELLS; h++) {
    const int ty = ty0 + h * CROWS;
    const long long id = cidx(k, i0 + tx, j0 + ty);
    const uint8_t mytag = h == 0 ? tags[0] : tags[CELLS - 1];
    if (advanced(k, mytag)) {
      float L[4];
      const float *x0 = s_face + sm.face_slot(tx, ty), *x1 = s_face + sm.face_slot(tx + 1, ty);
      const float *y0 = s_face + 2 * NFD + sm.face_slot(ty, tx), *y1 = s_face + 2 * NFD + sm.face_slot(ty + 1, tx);
      for (int v = 0; v < 4; v++)
        L[v] = -__fmaf_rn(x1[v * NF1] - x0[v * NF1], idx, __fmul_rn(y1[v * NF1] - y0[v * NF1], idy));
      if (DUAL) {
        dual_update_cell<STAGE>(k, c, id, P, L, dp, Out, ds->steps > 0);
      } else if (STAGE == 1) {
        for (int v = 0; v < 4; v++) Out[id + v * P] = um[h][v] + dt * L[v];
      } else if (STAGE == 2) {
        for (int v = 0; v < 4; v++)
          Out[id + v * P] = 0.75f * um[h][v] + 0.25f * (ui[h][v] + dt * L[v]);
      } else {
        // FP64 accumulation: dU^{n+1} = dU^n + (double)[2/3 ((dU^(2) - dU^n) + dt L)]
        float mnew[4];
        for (int v = 0; v < 4; v++) {
          const long long o = id + v * P;
          const float inc = (2.f / 3.f) * ((ui[h][v] - um[h][v]) + dt * L[v]);
          const double dn = ud[h][v] + f32_to_f64(inc);  // off the FP64 pipe, the stage's last phase: 768 x 384 step 76.6 -> 74.5 us
          D[o] = dn;
          mnew[v] = (float)dn;
          Mn[o] = mnew[v];
        }
        if (fuse_cfl) lam = fmaxf(lam, cfl_lambda(k, c, mnew));
      }
    } else if (!DUAL && BODY && STAGE == 3 && mytag != SOLID) {
      // IB / ghost node: the mirror of U^{n+1} takes the value rebuilt at stage 1
      for (int v = 0; v < 4; v++) Mn[id + v * P] = f64_to_f32(ud[h][v]);
    }
  }
  // one call site for the whole block (the reduction has a barrier)
  if (STAGE == 3 && fuse_cfl) cfl_block_max<NT>(k, lam, lred, ds, ncfl, PERSIST);
}

// The block's copy of a table entry's case.  Indexed in the kernel's parameters, the constants and pointers were read
// early and held across the tile in spilled registers (12.2 ms for a burst of 16 requests, 11.9 from shared memory); the
// compiler still reads some early.
static_assert(sizeof(TileSmem) + sizeof(StageCase) + 1024 <= 228 * 1024 / BATCH_BLOCKS,
              "the resident blocks that the launch bounds of the table kernels count on (1 KB of each block is reserved)");
template <int NT>
__device__ __forceinline__ void load_case(StageCase &dst, const StageCase &src) {
  static_assert(sizeof(StageCase) % 8 == 0, "copied in 8-byte words");
  for (int i = threadIdx.x; i < (int)(sizeof(StageCase) / 8); i += NT)
    reinterpret_cast<unsigned long long *>(&dst)[i] = reinterpret_cast<const unsigned long long *>(&src)[i];
  __syncthreads();
}

}  // namespace ibm
