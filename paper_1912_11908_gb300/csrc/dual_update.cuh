// Dual-time pseudo-stage update of one fluid cell in FP32-bulk form (FP64
// arithmetic), included by stage32.cuh ahead of the per-tile code.
#pragma once

#include "fp64_math.cuh"
#include "ibm_internal.cuh"

namespace ibm {

// ---------------------------------------------------------------------------
// Dual time in FP32-bulk form (Sec. 2).  The residual of a pseudo stage is the
// FP32 perturbation residual above (preconditioned LDFSS faces); the
// point-implicit update of each fluid cell runs in FP64:
//   [T Gamma / dtau + a T dW/dQ] dQ = -(R' + BDF'),   a = 3/(2 dt) or 1/dt,
// in perturbation variables W' = T W (T subtracts H_inf times the mass row
// from the energy row), so the energy rows of the Weiss-Smith matrices carry
// H - H_inf instead of H and never cancel against H_inf; R' = -L is the FP32
// residual, BDF' is formed from the FP64 iterate and the time levels' part
// fixed for the physical step (formed once per step), the 4x4
// system is solved in FP64 through its structure (solve_precond; the
// reciprocal of its FP32 pseudo-time step coefficient in FP32),
// Q' = (p', u, v, T') is updated and combined with the sub-iteration's start
// as SSP-RK3 stage, and the new iterate is stored in FP64 with its FP32
// mirror.
// ---------------------------------------------------------------------------
struct DualPtrs {
  const double *In64;  // FP64 iterate the stage starts from (perturbation)
  double *Out64;       // FP64 iterate it produces
  const double *G;     // the physical step's constant part of the BDF term: (W^{n-1} - 4 W^n) / (2 dt), or
                       // -W^n / dt on the first step (perturbation)
  double *Q0;          // (p', u', v', T') of the sub-iteration's start: written by stage 1, read by 2 and 3
};

// IEEE 754 binary32 <-> binary64 conversions done on the integer bits, off the
// FP64 pipe (which bounds the pseudo stage).  f32_to_f64 is exact for every
// normal and zero value (the FP32 arithmetic here flushes subnormals to
// zero); f64_to_f32 rounds to nearest, ties to even, for results in the
// normal FP32 range and leaves anything else to the hardware conversion.
__device__ __forceinline__ double f32_to_f64(float f) {
  const unsigned int b = __float_as_uint(f), e = (b >> 23) & 0xffu;
  if (e == 0xffu) return (double)f;  // infinity or NaN
  const unsigned int hi = (b & 0x80000000u) | (e ? ((e + 896u) << 20) | ((b & 0x7fffffu) >> 3) : 0u);
  return __hiloint2double((int)hi, (int)(e ? b << 29 : 0u));
}
__device__ __forceinline__ float f64_to_f32(double d) {
  const unsigned int hi = (unsigned int)__double2hiint(d), lo = (unsigned int)__double2loint(d);
  const unsigned int e = (hi >> 20) & 0x7ffu;
  if (e - 897u >= 254u) return (float)d;  // outside the normal FP32 exponent range: hardware conversion
  unsigned int f = (hi & 0x80000000u) | ((e - 896u) << 23) | ((hi & 0xfffffu) << 3) | (lo >> 29);
  const unsigned int rest = lo & 0x1fffffffu;  // the 29 dropped mantissa bits
  f += (rest > 0x10000000u) | ((rest == 0x10000000u) & (f & 1u));
  return __uint_as_float(f);
}

// The update below is bound by the FP64 pipe: reciprocals and the products that no fused multiply-add holds follow
// fp64_math.cuh (integer pipes), and the kinetic terms are written with dq = |u|^2 - |u_inf|^2 alone,
//   rho |u|^2 - |u_inf|^2 = drho |u_inf|^2 + rho dq,
// so that p' = (gamma - 1) [W + (H_inf - |u_inf|^2 / 2) drho - rho dq / 2].  About 48 FP64 instructions per cell and
// pseudo stage (93 before).  2048 x 1024, M = 0.001: 454 -> 283 us per pseudo stage, FP64 pipe 82% busy.
//
// FP64 perturbation conserved -> (p', u', v', T') with u' = u - u_inf; dr = rho - 1, r = rho, ir = 1 / rho
__device__ __forceinline__ void pert_prim64(const Consts &k, const double W[4], double q[4], double &r, double &ir,
                                            double &u, double &v, double &dq) {
  r = 1.0 + W[0];
  ir = rcp64(r);
  q[1] = mul64(fma(-k.uinf[0], W[0], W[1]), ir);
  q[2] = mul64(fma(-k.uinf[1], W[0], W[2]), ir);
  u = k.uinf[0] + q[1];
  v = k.uinf[1] + q[2];
  dq = fma(q[1], u + k.uinf[0], mul64(q[2], v + k.uinf[1]));
  q[0] = fma(-k.g1, half64(mul64(r, dq)), fma(k.g1hq, W[0], mul64(k.g1, W[3])));
  q[3] = mul64(fma(k.iR, q[0], -W[0]), ir);
}

// (p', u', v', T') -> FP64 perturbation conserved
__device__ __forceinline__ void prim_pert64(const Consts &k, const double q[4], double w[4]) {
  const double dr = mul64(fma(k.iR, q[0], -q[3]), rcp64(1.0 + q[3]));
  const double u = k.uinf[0] + q[1], v = k.uinf[1] + q[2];
  const double dq = fma(q[1], u + k.uinf[0], mul64(q[2], v + k.uinf[1]));
  w[0] = dr;
  w[1] = fma(dr, u, q[1]);
  w[2] = fma(dr, v, q[2]);
  w[3] = fma(k.ig1, q[0], fma(-k.hq, dr, half64(mul64(1.0 + dr, dq))));
}

// Exact solution of the point-implicit system in perturbation rows.  With
// s = 1/dtau + a the operator is s times the Weiss-Smith matrix whose first
// column parameter is tau = (theta_G/dtau + a theta_J) / s (the other columns
// are shared by Gamma and dW/dQ), so the momentum rows give du, dv directly
// (after subtracting u, v times the first row) and the first and energy rows
// leave a 2x2 system in dp, dT:
//   tau dp + rho_T dT = S0/s,   -dp + rho cp dT = (S3 - dH S0)/s - rho (u du + v dv).
// is = 1/s, ir = 1/rho.  1/s scales the whole update (a pseudo-time step
// size: it sets the path in pseudo time, not the fixed point, which the FP64
// right-hand side S fixes) and is taken in FP32 like s itself.  The pivot
// tau rho cp + rho_T is inverted in FP64: dp = rho cp dT - X is a small
// difference of two terms of size X, so a relative error in 1/pivot would
// reach dp multiplied by X / dp.
__device__ __forceinline__ void solve_precond(double is, double tau, double r, double ir, double u, double v,
                                              double rT, double cpv, double dH, const double S[4], double dQ[4]) {
  const double irs = mul64(is, ir);
  const double du = mul64(fma(-u, S[0], S[1]), irs);
  const double dv = mul64(fma(-v, S[0], S[2]), irs);
  const double X = fma(-r, fma(u, du, mul64(v, dv)), mul64(fma(-dH, S[0], S[3]), is));
  const double Y = mul64(S[0], is), rc = mul64(r, cpv);
  const double dT = mul64(fma(tau, X, Y), rcp64(fma(tau, rc, rT)));
  dQ[0] = fma(rc, dT, -X);
  dQ[1] = du;
  dQ[2] = dv;
  dQ[3] = dT;
}

// pseudo stage STAGE of one fluid cell (id: state index); L = FP32 residual
template <int STAGE>
__device__ __forceinline__ void dual_update_cell(const Consts &k, const PertConsts &c, long long id, long long P,
                                                 const float L[4], const DualPtrs &dp,
                                                 float *Out32, bool bdf2) {
  const double idt = k.idt_phys;
  const double aw = bdf2 ? 1.5 * idt : idt;  // coefficient of the iterate in the BDF term
  double W[4], S[4], Qk[4], r, ir, u, v, dq;
  for (int q = 0; q < 4; q++) W[q] = dp.In64[id + q * P];
  pert_prim64(k, W, Qk, r, ir, u, v, dq);
  // -(R' + BDF') with R' = -L and the BDF term aw W + G: BDF2 (3 W - 4 W^n + W^{n-1}) / (2 dt), BDF1 (W - W^n) / dt
  for (int q = 0; q < 4; q++) S[q] = fma(-aw, W[q], f32_to_f64(L[q]) - dp.G[id + q * P]);
  // pseudo-time coefficients (local dtau, preconditioning parameter) in FP32: they set the pseudo-time path,
  // not the fixed point R' + BDF' = 0.  (Sums of products written out as fused multiply-adds here and in the divergence, so
  // that blocks of either width give a case the same bits.)
  const float rf = f64_to_f32(r), irf = 1.f / rf, uf = f64_to_f32(u), vf = f64_to_f32(v);
  const float Tf = 1.f + f64_to_f32(Qk[3]), iTf = 1.f / Tf;
  const float csf = sqrtf(c.gamma * (c.R + f64_to_f32(Qk[0])) * irf), icsf = 1.f / csf;
  const float Vm = sqrtf(__fmaf_rn(uf, uf, __fmul_rn(vf, vf)));
  float Ur = fmaxf(fmaxf(Vm, 1.f), c.mu * irf / c.dmin);
  Ur = fminf(Ur, csf);
  const float ui = __fmul_rn(Ur, icsf), mr2 = __fmul_rn(ui, ui);
  const float up = __fmul_rn(__fmul_rn(0.5f, Vm), 1.f + mr2);
  const float om = __fsub_rn(1.f, mr2), ov = __fmul_rn(om, Vm), ur = __fmul_rn(2.f, Ur);
  const float cp_ = __fmul_rn(0.5f, sqrtf(__fmaf_rn(ov, ov, __fmul_rn(ur, ur))));
  const float lam = __fmaf_rn(__fadd_rn(up, cp_), c.idx + c.idy, __fmul_rn(c.vis, irf));
  const float idtau = lam / c.cfl_tau;
  const float af = bdf2 ? __fmul_rn(1.5f, c.idt_phys) : c.idt_phys;
  const float thG = __fadd_rn(1.f / __fmul_rn(Ur, Ur), iTf / c.cp), thJ = iTf / c.R;
  const float sf = __fadd_rn(idtau, af);
  const float tau = __fmaf_rn(thG, idtau, __fmul_rn(af, thJ)) / sf;
  const double dH = fma(k.cp, Qk[3], half64(dq));
  double dQ[4];
  solve_precond(f32_to_f64(1.f / sf), f32_to_f64(tau), r, ir, u, v, -f32_to_f64(rf * iTf), k.cp, dH, S, dQ);
  double Q0[4], Qn[4], Wo[4];
  if (STAGE == 1) {  // the stage starts from the sub-iteration's start: keep its primitives for stages 2 and 3
    for (int q = 0; q < 4; q++) dp.Q0[id + q * P] = Qk[q];
  } else {
    for (int q = 0; q < 4; q++) Q0[q] = dp.Q0[id + q * P];
  }
  for (int q = 0; q < 4; q++) {
    const double e = Qk[q] + dQ[q];
    Qn[q] = STAGE == 1 ? e : (STAGE == 2 ? fma(0.75, Q0[q], half64(half64(e))) : fma(1.0 / 3.0, Q0[q], mul64(2.0 / 3.0, e)));
  }
  prim_pert64(k, Qn, Wo);
  for (int q = 0; q < 4; q++) {
    dp.Out64[id + q * P] = Wo[q];
    Out32[id + q * P] = f64_to_f32(Wo[q]);
  }
}

}  // namespace ibm
