// FP64 flow kernels: time step, IB / ghost reconstruction and the fused
// residual + SSP-RK3 stage update (domain halos are applied while the stage
// kernel loads its tile).
//
// State layout: structure of arrays, four conserved planes (rho, rho u,
// rho v, rho E), each (ny + 6) rows of `pitch` doubles; cell (i, j) of the
// interior sits at (j + 3) * pitch + (i + 3).  Rows are padded to a multiple
// of 32 elements so every row starts 256-byte aligned.
#include <algorithm>

#include "fp64_math.cuh"
#include "ibm_internal.cuh"

namespace ibm {

// ---------------------------------------------------------------------------
// Time step from the CFL rule over fluid cells:
//   dt = CFL / max[(|u|+c)/dx + (|v|+c)/dy + 2 gamma mu/(Pr rho)(1/dx^2+1/dy^2)].
// Positive doubles order like their bit patterns, so the maximum is an
// integer atomicMax (order-independent, exact); the last block to finish
// turns it into dt.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_dt(Consts k, const double *__restrict__ A,
                                            const uint8_t *__restrict__ tag, DevState *ds) {
  const int ncell = k.nx * k.ny;
  double lmax = 0.0;
  const double idx = 1.0 / k.dx, idy = 1.0 / k.dy;
  const double vis = (2.0 * k.gamma * k.mu / k.prandtl) * fma(idx, idx, idy * idy);
  for (int n = blockIdx.x * blockDim.x + threadIdx.x; n < ncell; n += gridDim.x * blockDim.x) {
    if (tag[n] != FLUID && !(k.ib_advance && tag[n] == IB)) continue;
    long long id = cidx(k, n % k.nx, n / k.nx);
    const double r = A[id], ir = rcp64(r), u = A[id + k.plane] * ir, v = A[id + 2 * k.plane] * ir;
    const double p = (k.gamma - 1.0) * fma(-0.5 * r, fma(u, u, v * v), A[id + 3 * k.plane]);
    const double c = sqrt64(k.gamma * p * ir);
    double lam = fma(fabs(u) + c, idx, fma(fabs(v) + c, idy, vis * ir));
    if (not_finite(lam)) {
      // a state beyond the range of fp64_math.cuh, whose results are NaN there and would drop out of the maximum: the
      // bound in the hardware's arithmetic, so that a cell that overflowed drives dt to zero
      const double ui = A[id + k.plane] / r, vi = A[id + 2 * k.plane] / r;
      const double ci = sqrt(k.gamma * ((k.gamma - 1.0) * (A[id + 3 * k.plane] - 0.5 * r * (ui * ui + vi * vi))) / r);
      lam = (fabs(ui) + ci) / k.dx + (fabs(vi) + ci) / k.dy + vis / r;
    }
    lmax = fmax(lmax, lam);
  }
  for (int off = 16; off > 0; off >>= 1) lmax = fmax(lmax, __shfl_xor_sync(0xffffffffu, lmax, off));
  __shared__ double wm[8];
  if ((threadIdx.x & 31) == 0) wm[threadIdx.x >> 5] = lmax;
  __syncthreads();
  if (threadIdx.x == 0) {
    double m = wm[0];
    for (int w = 1; w < 8; w++) m = fmax(m, wm[w]);
    atomicMax(&ds->lmax_bits, (unsigned long long)__double_as_longlong(m));
    finish_cfl(k, ds, gridDim.x * gridDim.y);
  }
}

int sm_count() {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) {
    cudaGetLastError();
    return 152;
  }
  return sms;
}
extern "C" int ibm__sm_count() { return sm_count(); }

void launch_dt(const Consts &k, const double *A, const uint8_t *tag, DevState *ds, cudaStream_t s, int *nlaunch) {
  if (k.dt_fixed > 0.0) return;  // ds->dt was set at creation
  int ncell = k.nx * k.ny;
  int blocks = min((ncell + 255) / 256, 152 * 8);
  k_dt<<<blocks, 256, 0, s>>>(k, A, tag, ds);
  *nlaunch += 1;
}

// ---------------------------------------------------------------------------
// Sec. 4.4-4.6, Sec. 5: rebuild IB nodes (pass 0) or ghost nodes (pass 1)
// from their stencils.  Primitives p, u, v, T are interpolated at the probe
// / image point; velocity is Dirichlet (Eq. 4), linear along the normal
// through the wall velocity at P'; pressure is Neumann with
// dp/dn = -rho n.a_wall (Eq. 5-6), plus, for a body moving faster than the
// free-stream sound speed, the centripetal term rho u_t^2 kappa of the normal
// momentum balance (Eq. 7, in the sign convention of Eq. 6; u_t is the
// velocity tangential to the wall relative to it at the probe, kappa the
// signed curvature at P'); temperature is adiabatic (Eq. 8), which makes the
// pressure condition a linear ODE in p along the normal, integrated exactly.
// One thread per list entry; in place on the stage array.
// ---------------------------------------------------------------------------
// A state written by the caller ([4][ny][nx] absolute conserved, contiguous, already on the device) into the
// case's padded layout: FP64 as given, or -- FP32-bulk, M != null -- as the perturbation from the free stream
// (dU = U - U_inf, the energy row less H_inf d rho) with its FP32 mirror.  One thread per cell.
__global__ void k_set_state(Consts k, const double *__restrict__ U, double *__restrict__ A, float *__restrict__ M) {
  const long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long ncell = (long long)k.nx * k.ny;
  if (n >= ncell) return;
  const long long id = cidx(k, (int)(n % k.nx), (int)(n / k.nx)), P = k.plane;
  double u0 = U[n], u1 = U[n + ncell], u2 = U[n + 2 * ncell], u3 = U[n + 3 * ncell];
  if (M) {
    const double d = u0 - 1.0;
    u0 = d;
    u1 = u1 - k.Uinf[1];
    u2 = u2 - k.Uinf[2];
    u3 = (u3 - k.Uinf[3]) - k.Hinf * d;
    M[id] = (float)u0;
    M[id + P] = (float)u1;
    M[id + 2 * P] = (float)u2;
    M[id + 3 * P] = (float)u3;
  }
  A[id] = u0;
  A[id + P] = u1;
  A[id + 2 * P] = u2;
  A[id + 3 * P] = u3;
}

void launch_set_state(const Consts &k, const double *U, double *A, float *M, cudaStream_t s) {
  const long long ncell = (long long)k.nx * k.ny;
  k_set_state<<<(unsigned)((ncell + 255) / 256), 256, 0, s>>>(k, U, A, M);
}

// (p, u, v, T) interpolated at a probe from the valid corners of its square
__device__ __forceinline__ void probe_f64(const Consts &k, const double *U, int i0, int j0, int mask,
                                          const double w[4], double qp[4]) {
  for (int q = 0; q < 4; q++) qp[q] = 0.0;
  for (int q = 0; q < 4; q++) {
    if (!(mask >> q & 1)) continue;
    long long id = cidx(k, i0 + (q & 1), j0 + (q >> 1));
    const double r = U[id], ir = rcp64(r), u = U[id + k.plane] * ir, v = U[id + 2 * k.plane] * ir;
    const double p = (k.gamma - 1.0) * fma(-0.5 * r, fma(u, u, v * v), U[id + 3 * k.plane]);
    qp[0] += w[q] * p;
    qp[1] += w[q] * u;
    qp[2] += w[q] * v;
    qp[3] += w[q] * (p * ir * k.iR);
  }
}

__device__ __forceinline__ void recon_one_f64(const Consts &k, double *U, const ibm_stencil &s, const double Vb[2],
                                              const double Ab[2], bool sup, double t) {
  if (s.mask == 0) return;
  double V[2], Acc[2];
  wall_kin(k, t, s.bx, s.by, Vb, Ab, V, Acc);  // the wall's motion at P'
  double qp[4];
  probe_f64(k, U, s.i0, s.j0, s.mask, s.w, qp);
  // dp/dn = rho G (Eq. 5-7)
  double G = -(s.nx * Acc[0] + s.ny * Acc[1]);
  if (sup) {
    const double ut = -(qp[1] - V[0]) * s.ny + (qp[2] - V[1]) * s.nx;
    G = G + ut * ut * s.curv;
  }
  double p, u, v, T;
  if (k.quad && s.maskb != 0) {
    // quadratic form (Sec. 4.5, Sec. 5): quadratics in the distance s along the normal through the wall
    // condition (s = 0) and the probes at s1, s2, evaluated at the node s_n -- Lagrange for the Dirichlet
    // velocity, a + b s + c s^2 with the wall slope b given for T (0) and p (rho G, the first probe's density)
    double qb[4];
    probe_f64(k, U, s.i0b, s.j0b, s.maskb, s.wb, qb);
    const double s1 = s.xi_probe, s2 = s.xi_probe2, sn = s.xi_node;
    const double L1 = sn * (sn - s2) / (s1 * (s1 - s2)), L2 = sn * (sn - s1) / (s2 * (s2 - s1));
    const double m = (sn * sn - s1 * s1) / (s2 * s2 - s1 * s1);
    const double b = qp[0] / (k.R * qp[3]) * G;
    u = V[0] + (qp[1] - V[0]) * L1 + (qb[1] - V[0]) * L2;
    v = V[1] + (qp[2] - V[1]) * L1 + (qb[2] - V[1]) * L2;
    T = qp[3] + (qb[3] - qp[3]) * m;
    p = qp[0] + (qb[0] - qp[0]) * m + b * ((sn - s1) - (s2 - s1) * m);
  } else {
    // linear form: rho = p / (R T) and T fixed along the normal (Eq. 8), integrated exactly from the probe to
    // the node, p = p_probe exp(-(xi_p - xi_n) G / (R T)), positive however coarse the grid
    // (G = 0, a wall without normal acceleration: p = p_probe, without the exponential)
    const double ratio = s.xi_node * rcp64(s.xi_probe);
    p = G != 0.0 ? qp[0] * exp(-(s.xi_probe - s.xi_node) * G * (k.iR * rcp64(qp[3]))) : qp[0];
    u = V[0] + (qp[1] - V[0]) * ratio;
    v = V[1] + (qp[2] - V[1]) * ratio;
    T = qp[3];
  }
  const double r = p * (k.iR * rcp64(T));
  const long long id = cidx(k, s.cell % k.nx, s.cell / k.nx);
  U[id] = r;
  U[id + k.plane] = r * u;
  U[id + 2 * k.plane] = r * v;
  U[id + 3 * k.plane] = fma(p, k.ig1, 0.5 * r * fma(u, u, v * v));
}

// one cluster of RC blocks: all IB nodes, a cluster barrier, then all ghost nodes.  A few hundred nodes of FP64 work
// hold one SM's FP64 pipe for most of the launch (two lanes per clock); eight SMs share it, and the barrier in place of
// a second launch keeps the pair of passes at one launch per stage.  Per stage, its launch included: 257 x 131 dual time about
// 20 -> 10 us, 768 x 384 wedge about 100 -> 15 us.
constexpr int RC = 8, RT = 128;
__global__ void __cluster_dims__(RC, 1, 1) __launch_bounds__(RT)
    k_recon1_f64(Consts k, double *U, const ibm_stencil *__restrict__ st, int cap, const DevState *__restrict__ ds,
                 int stage) {
  double X[2], V[2], Acc[2];
  const double ts = stage_time(ds, stage);
  body_motion(k, ds, ts, X, V, Acc);
  const bool sup = supersonic_motion(k, V);
  const int nib = min(ds->offset[1], cap), tot = min(ds->offset[4], cap);
  // consecutive warps of nodes on different blocks
  const int first = ((threadIdx.x >> 5) * RC + blockIdx.x) * 32 + (threadIdx.x & 31);
  if (!k.ib_advance)  // IB nodes rebuilt (else advanced by the flux update)
    for (int e = first; e < nib; e += RC * RT) recon_one_f64(k, U, st[e], V, Acc, sup, ts);
  __threadfence();
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
  for (int e = nib + first; e < tot; e += RC * RT) recon_one_f64(k, U, st[e], V, Acc, sup, ts);
}

// many blocks, one pass (0: IB nodes, 1: ghost nodes) per launch
__global__ void __launch_bounds__(128) k_recon_f64(Consts k, double *U, const ibm_stencil *__restrict__ st,
                                                   int cap, const DevState *__restrict__ ds, int stage, int pass) {
  const int lo = pass == 0 ? 0 : ds->offset[1];
  const int hi = min(pass == 0 ? ds->offset[1] : ds->offset[4], cap);
  const int e = lo + blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= hi) return;
  double X[2], V[2], Acc[2];
  const double ts = stage_time(ds, stage);
  body_motion(k, ds, ts, X, V, Acc);
  recon_one_f64(k, U, st[e], V, Acc, supersonic_motion(k, V), ts);
}

void launch_recon_f64(const Consts &k, double *U, const ibm_stencil *st, int cap, const DevState *ds, int stage,
                      cudaStream_t s, int *nlaunch) {
  if (cap <= 0) return;
  if (cap <= RECON_ONE_BLOCK_MAX) {
    k_recon1_f64<<<RC, RT, 0, s>>>(k, U, st, cap, ds, stage);
    *nlaunch += 1;
    return;
  }
  int blocks = (cap + 127) / 128;
  if (!k.ib_advance) {  // IB nodes rebuilt (else advanced by the flux update)
    k_recon_f64<<<blocks, 128, 0, s>>>(k, U, st, cap, ds, stage, 0);
    *nlaunch += 1;
  }
  k_recon_f64<<<blocks, 128, 0, s>>>(k, U, st, cap, ds, stage, 1);
  *nlaunch += 1;
}

// ---------------------------------------------------------------------------
// Fused residual + stage update, FP64.  One TX x TY tile of cells per block,
// one thread per cell: the tile and its 3-cell halo are loaded once and
// converted to primitives in shared memory; WENO5 (or TVD-2) runs along tile
// lines -- an item is one variable of one row or column, or half of one, and
// its consecutive windows share their differences (Weno64); every face then
// takes its LDFSS + central viscous flux, and each fluid cell its flux
// divergence and SSP-RK3 stage
//   stage 1: out = Un + dt L(in)
//   stage 2: out = 3/4 Un + 1/4 (in + dt L(in))
//   stage 3: out = 1/3 Un + 2/3 (in + dt L(in))
// or, in dual time, its point-implicit pseudo stage.  Tiles without a fluid
// cell exit at once.
//
// The kernel is bound by the FP64 pipe (fp64_math.cuh; 85% busy in ncu):
// a window per state with IEEE divisions took about 2,000 FP64 instructions
// per cell and stage, the shared windows and reciprocals about 540, with
// products on the integer pipes 370, with reciprocals and square roots there
// too about 330.  768 x 384 wedge, two steps: 6.90 -> 3.07 -> 2.21 -> 1.56 ms
// (the last with the reconstruction on a cluster).
// ---------------------------------------------------------------------------
struct F64Consts {
  double ih[2], g1, ig1, iR;
  // viscous terms of the x and y faces, h the spacing along the normal and t along the tangent: mu 4/3 / h,
  // mu 2/3 / (4 t), mu / (4 t), mu / h, kappa / h, and (mu / h)^2
  double nn[2], nt[2], ts[2], tv[2], kt[2], munu2[2];
  // dual time: mu / min(dx, dy), 2 gamma mu / Pr (1 / dx^2 + 1 / dy^2), 1 / CFL_tau, 1 / cp
  double nud, dif, icfl, icp;
};

static F64Consts f64_consts(const Consts &k) {
  F64Consts c;
  c.ih[0] = 1.0 / k.dx;
  c.ih[1] = 1.0 / k.dy;
  c.g1 = k.gamma - 1.0;
  c.ig1 = k.ig1;
  c.iR = k.iR;
  for (int d = 0; d < 2; d++) {
    const double in = c.ih[d], it = c.ih[1 - d];
    c.nn[d] = k.mu * (4.0 / 3.0) * in;
    c.nt[d] = k.mu * (2.0 / 3.0) * 0.25 * it;
    c.ts[d] = k.mu * 0.25 * it;
    c.tv[d] = k.mu * in;
    c.kt[d] = k.kappa * in;
    c.munu2[d] = (k.mu * in) * (k.mu * in);
  }
  c.nud = k.mu / k.dmin;
  c.dif = (2.0 * k.gamma * k.mu / k.prandtl) * (c.ih[0] * c.ih[0] + c.ih[1] * c.ih[1]);
  c.icfl = k.cfl_tau > 0.0 ? 1.0 / k.cfl_tau : 0.0;
  c.icp = 1.0 / k.cp;
  return c;
}

template <int TX, int TY>
struct Tile64 {
  double sq[4][TY + 2 * NG][TX + 2 * NG];  // rho, u, v, p
  double sT[TY + 2 * NG][TX + 2 * NG];
  double Lx[4][TY][TX + 1], Rx[4][TY][TX + 1];  // x-face states; Lx then the x flux
  double Ly[4][TY + 1][TX], Ry[4][TY + 1][TX];  // y-face states; Ly then the y flux
};

// n windows of a line, the first centred at lp[0] (stride ls): a window's left state to L[i], its right state to
// R[i] for i < nl and i >= 1 of the line's windows i0 + 0 .. n - 1 (stride os).  The loop stays rolled: unrolled, the
// integer multiplications overflow the instruction cache.
__device__ __forceinline__ void line64(const double *lp, int ls, int n, double *L, double *R, int os, int i0, int nl,
                                       bool tvd) {
  double f3 = lp[ls];
  if (tvd) {
    // Sec. 2, the second-order TVD scheme: MUSCL with the minmod limiter
    double f1 = lp[-ls], f2 = lp[0];
#pragma unroll 1
    for (int i = 0; i < n; i++) {
      f3 = lp[(i + 1) * ls];
      const double a = f2 - f1, b = f3 - f2;
      double m = 0.0;
      if (a > 0.0 && b > 0.0) m = a < b ? a : b;
      else if (a < 0.0 && b < 0.0) m = a > b ? a : b;
      if (i0 + i < nl) L[(i0 + i) * os] = fma(0.5, m, f2);
      if (i0 + i >= 1) R[(i0 + i - 1) * os] = fma(-0.5, m, f2);
      f1 = f2;
      f2 = f3;
    }
    return;
  }
  Weno64 w;
  w.start(lp[-2 * ls], lp[-ls], lp[0], f3);
#pragma unroll 1
  for (int i = 0; i < n; i++) {
    const double f4 = lp[(i + 2) * ls];
    double qL, qR;
    w.next(f3, f4, qL, qR);
    if (i0 + i < nl) L[(i0 + i) * os] = qL;
    if (i0 + i >= 1) R[(i0 + i - 1) * os] = qR;
    f3 = f4;
  }
}

// Dual time (Sec. 2): pseudo-time stage of the point-implicit preconditioned update
//   [Gamma/dtau + a dW/dQ] dQ = -(R + BDF(W)),  a = 3/(2 dt) (BDF2) or 1/dt (first step),
// combined with the sub-iteration's start Q0 (held in A) as SSP-RK3 stage STAGE.  Gamma and dW/dQ are Weiss-Smith
// matrices that differ in their first column's parameter only (1/Ur^2 + 1/(T cp) and 1/(R T)), so the sum is s times
// such a matrix, s = 1/dtau + a, and its rows less multiples of the first solve in closed form: the momentum rows give
// du, dv, the energy row r cp dT - dp = Y, and the first row dT.  Rv: flux divergence.
template <int STAGE>
__device__ __forceinline__ void dual_cell64(const Consts &k, const F64Consts &c, const double *A, const double *In,
                                            double *Out, const double *__restrict__ Wn, const double *__restrict__ Wm,
                                            long long id, const double Rv[4], bool bdf2) {
  const long long P = k.plane;
  double W[4], S[4];
  for (int v = 0; v < 4; v++) W[v] = In[id + v * P];
  const double r = W[0], ir = rcp64(r), u = mul64(W[1], ir), v = mul64(W[2], ir), V2 = fma(u, u, mul64(v, v));
  const double pr = mul64(c.g1, fma(-half64(r), V2, W[3])), T = mul64(mul64(pr, ir), c.iR);
  const double aw = bdf2 ? 1.5 * k.idt_phys : k.idt_phys;
  for (int q = 0; q < 4; q++) {
    const long long o = id + q * P;
    const double t = bdf2 ? fma(0.5, Wm[o], fma(1.5, W[q], mul64(-2.0, Wn[o]))) : W[q] - Wn[o];
    S[q] = fma(-k.idt_phys, t, -Rv[q]);
  }
  // pseudo-time step of the preconditioned eigenvalues, reference velocity by squares
  const double c2 = mul64(mul64(k.gamma, pr), ir), vis = mul64(c.nud, ir);
  const double ur2 = fmin(fmax(fmax(V2, 1.0), mul64(vis, vis)), c2), ic2 = rcp64(c2);
  const double mr2 = mul64(ur2, ic2), t = half64(1.0 - mr2), Vm = sqrt64(V2), cq = sqrt64(fma(mul64(t, t), V2, ur2));
  const double lam = fma(fma(half64(Vm), 1.0 + mr2, cq), c.ih[0] + c.ih[1], mul64(c.dif, ir));
  const double idtau = mul64(lam, c.icfl), s = idtau + aw;
  const double iT = rcp64(T), rT = mul64(-r, iT);
  const double th = fma(idtau, fma(iT, c.icp, rcp64(ur2)), mul64(mul64(aw, c.iR), iT));
  const double is = rcp64(s), isr = mul64(is, ir), H = fma(k.cp, T, half64(V2));
  const double du = mul64(fma(-u, S[0], S[1]), isr), dv = mul64(fma(-v, S[0], S[2]), isr);
  const double rcp_ = mul64(r, k.cp);
  const double Y = fma(fma(-H, S[0], S[3]), is, mul64(-r, fma(u, du, mul64(v, dv))));
  const double dT = mul64(fma(th, Y, S[0]), rcp64(fma(th, rcp_, mul64(s, rT))));
  const double dQ[4] = {fma(rcp_, dT, -Y), du, dv, dT}, Qk[4] = {pr, u, v, T};
  double Qn[4];
  if (STAGE == 1) {
    for (int q = 0; q < 4; q++) Qn[q] = Qk[q] + dQ[q];
  } else {
    const double r0 = A[id], ir0 = rcp64(r0), u0 = mul64(A[id + P], ir0), v0 = mul64(A[id + 2 * P], ir0);
    const double p0 = mul64(c.g1, fma(-half64(r0), fma(u0, u0, mul64(v0, v0)), A[id + 3 * P]));
    const double Q0[4] = {p0, u0, v0, mul64(mul64(p0, ir0), c.iR)};
    for (int q = 0; q < 4; q++) {
      const double e = Qk[q] + dQ[q];
      Qn[q] = STAGE == 2 ? fma(0.75, Q0[q], half64(half64(e))) : fma(1.0 / 3.0, Q0[q], mul64(2.0 / 3.0, e));
    }
  }
  const double rn = mul64(mul64(Qn[0], c.iR), rcp64(Qn[3]));
  Out[id] = rn;
  Out[id + P] = mul64(rn, Qn[1]);
  Out[id + 2 * P] = mul64(rn, Qn[2]);
  Out[id + 3 * P] = fma(Qn[0], c.ig1, mul64(half64(rn), fma(Qn[1], Qn[1], mul64(Qn[2], Qn[2]))));
}

template <int STAGE, bool DUAL, int TX, int TY>
__global__ void __launch_bounds__(TX *TY) k_stage_f64(Consts k, F64Consts c, const double *Un,
                                                      const double *__restrict__ In, double *Out,
                                                      const double *__restrict__ Wn, const double *__restrict__ Wm,
                                                      const uint8_t *__restrict__ tag, DevState *ds) {
  constexpr int HX = TX + 2 * NG, HY = TY + 2 * NG, NT = TX * TY;
  extern __shared__ __align__(16) unsigned char smem64[];
  Tile64<TX, TY> &sm = *reinterpret_cast<Tile64<TX, TY> *>(smem64);
  auto &sq = sm.sq;
  auto &sT = sm.sT;
  const int i0 = blockIdx.x * TX, j0 = blockIdx.y * TY;
  const int tx = threadIdx.x % TX, ty = threadIdx.x / TX;
  const int ci = i0 + tx, cj = j0 + ty;
  const bool inside = ci < k.nx && cj < k.ny;
  // cells the flux update advances: fluid cells, and IB nodes when the ghost layers alone impose the wall
  const bool fluid = inside && (tag[cj * k.nx + ci] == FLUID || (k.ib_advance && tag[cj * k.nx + ci] == IB));
  const double dt = DUAL ? 0.0 : ds->dt;
  if (!DUAL && STAGE == 3 && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) {
    // end of the step (no other kernel of this stage reads t)
    ds->t = ds->t + dt;
    ds->steps += 1;
  }
  if (!__syncthreads_or(fluid)) return;

  const long long P = k.plane;
  for (int m = threadIdx.x; m < HX * HY; m += NT) {
    const int a = m % HX, b = m / HX;
    int gi = i0 - NG + a, gj = j0 - NG + b;
    double U0, U1, U2, U3;
    if (halo_map(k, gi, gj)) {
      const long long id = cidx(k, gi, gj);
      U0 = In[id];
      U1 = In[id + P];
      U2 = In[id + 2 * P];
      U3 = In[id + 3 * P];
    } else {
      U0 = k.Uinf[0];
      U1 = k.Uinf[1];
      U2 = k.Uinf[2];
      U3 = k.Uinf[3];
    }
    const double ir = rcp64(U0);
    const double u = mul64(U1, ir), v = mul64(U2, ir);
    const double p = mul64(c.g1, fma(-half64(U0), fma(u, u, mul64(v, v)), U3));
    sq[0][b][a] = U0;
    sq[1][b][a] = u;
    sq[2][b][a] = v;
    sq[3][b][a] = p;
    sT[b][a] = mul64(mul64(p, ir), c.iR);
  }
  __syncthreads();

  // face states along lines: TX (TY) + 2 windows per row (column), in two halves of nine or one of ten; one code
  // path for both directions
  constexpr int NX = TX == 16 ? 9 : 10, HFX = TX == 16 ? 2 : 1, NY = TY == 16 ? 9 : 10, HFY = TY == 16 ? 2 : 1;
  static_assert(4 * TY * HFX + 4 * TX * HFY == NT, "one item per thread");
  {
    const bool xd = threadIdx.x < 4 * TY * HFX;
    const int u = xd ? threadIdx.x : threadIdx.x - 4 * TY * HFX;
    const int half = xd ? u % HFX : u / TX % HFY, line = xd ? u / HFX % TY : u % TX,
              v = xd ? u / (HFX * TY) : u / (TX * HFY);
    const int i0w = half * (xd ? NX : NY);
    line64(xd ? &sq[v][NG + line][2 + i0w] : &sq[v][2 + i0w][NG + line], xd ? 1 : HX, xd ? NX : NY,
           xd ? &sm.Lx[v][line][0] : &sm.Ly[v][0][line], xd ? &sm.Rx[v][line][0] : &sm.Ry[v][0][line], xd ? 1 : TX, i0w,
           (xd ? TX : TY) + 1, k.tvd2);
  }
  __syncthreads();

  // face fluxes: inviscid (first order where a reconstructed density or pressure is not positive) less viscous; d the
  // direction, un / ut the velocity components along the normal and the tangent, sn / st the strides
  for (int m = threadIdx.x; m < (TX + 1) * TY + TX * (TY + 1); m += NT) {
    const int d = m < (TX + 1) * TY ? 0 : 1, mm = d ? m - (TX + 1) * TY : m;
    const int f = d ? mm / TX : mm % (TX + 1), line = d ? mm % TX : mm / (TX + 1);
    const int at = d ? (f + 2) * HX + line + NG : (line + NG) * HX + f + 2, sn = d ? HX : 1, st = d ? 1 : HX;
    const double *q0 = &sq[0][0][0] + at, *qn = q0 + (1 + d) * HX * HY, *qt = q0 + (2 - d) * HX * HY,
                 *q3 = q0 + 3 * HX * HY, *T = &sT[0][0] + at;
    double *o = (d ? &sm.Ly[0][0][0] : &sm.Lx[0][0][0]) + mm;
    const double *r = (d ? &sm.Ry[0][0][0] : &sm.Rx[0][0][0]) + mm;
    const int vs = d ? (TY + 1) * TX : TY * (TX + 1);  // values per variable
    double rL = o[0], uL = o[(1 + d) * vs], vL = o[(2 - d) * vs], pL = o[3 * vs];
    double rR = r[0], uR = r[(1 + d) * vs], vR = r[(2 - d) * vs], pR = r[3 * vs];
    if (!positive(rL) || !positive(pL) || !positive(rR) || !positive(pR)) {
      rL = q0[0];
      uL = qn[0];
      vL = qt[0];
      pL = q3[0];
      rR = q0[sn];
      uR = qn[sn];
      vR = qt[sn];
      pR = q3[sn];
    }
    double F[4];
    ldfss64<DUAL, 1>(rL, uL, &vL, pL, rR, uR, &vR, pR, k.gamma, c.ig1, c.munu2[d], F);
    const double u0 = qn[0], u1 = qn[sn], v0 = qt[0], v1 = qt[sn];
    const double us = (qn[st] - qn[-st]) + (qn[sn + st] - qn[sn - st]);
    const double ws = (qt[st] - qt[-st]) + (qt[sn + st] - qt[sn - st]);
    const double tn = fma(c.nn[d], u1 - u0, -mul64(c.nt[d], ws)), tt = fma(c.ts[d], us, mul64(c.tv[d], v1 - v0));
    const double w = fma(u0 + u1, tn, mul64(v0 + v1, tt));
    o[0] = F[0];
    o[(1 + d) * vs] = F[1] - tn;
    o[(2 - d) * vs] = F[2] - tt;
    o[3 * vs] = fma(-c.kt[d], T[sn] - T[0], fma(-0.5, w, F[3]));
  }
  __syncthreads();
  if (!fluid) return;
  const long long id = cidx(k, ci, cj);
  double Rv[4];
  for (int v = 0; v < 4; v++)
    Rv[v] = fma(sm.Lx[v][ty][tx + 1] - sm.Lx[v][ty][tx], c.ih[0],
                mul64(sm.Ly[v][ty + 1][tx] - sm.Ly[v][ty][tx], c.ih[1]));
  if (DUAL) {
    dual_cell64<STAGE>(k, c, Un, In, Out, Wn, Wm, id, Rv, ds->steps > 0);
    return;
  }
  for (int v = 0; v < 4; v++) {
    const long long o = id + v * P;
    if (STAGE == 1) Out[o] = fma(-dt, Rv[v], Un[o]);
    else if (STAGE == 2) Out[o] = fma(0.75, Un[o], half64(half64(fma(-dt, Rv[v], In[o]))));
    else Out[o] = fma(1.0 / 3.0, Un[o], mul64(2.0 / 3.0, fma(-dt, Rv[v], In[o])));
  }
}

template <int STAGE, bool DUAL, int TX, int TY>
static void launch_tile_f64(const Consts &k, const double *Un, const double *In, double *Out, const double *Wn,
                            const double *Wm, const uint8_t *tag, DevState *ds, cudaStream_t s) {
  constexpr int bytes = (int)sizeof(Tile64<TX, TY>);
  if (bytes > 48 * 1024)
    cudaFuncSetAttribute(k_stage_f64<STAGE, DUAL, TX, TY>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  k_stage_f64<STAGE, DUAL, TX, TY><<<dim3((k.nx + TX - 1) / TX, (k.ny + TY - 1) / TY), TX * TY, bytes, s>>>(
      k, f64_consts(k), Un, In, Out, Wn, Wm, tag, ds);
}

// Tile shape by the work of the fullest SM: an SM's time is its tiles' FP64 instructions (halo cells, windows and
// faces included: 1, 0.53 and 0.30 of the 16 x 16 tile), and the tiles are dealt evenly, so a grid of few tiles takes
// the shape whose last round is fullest -- 257 x 131 cells are 153 tiles of 16 x 16 on 152 SMs, 289 of 16 x 8: a
// dual-time pseudo stage there went from 374 us (16 x 16, the arithmetic before) to 55.  Rows of tiles run along
// gridDim.y, so a grid taller than 65,535 rows of eight cells keeps the 16 x 16 tile.  Returns 0: 16 x 16, 1: 16 x 8,
// 2: 8 x 8.
extern "C" int ibm__tile_shape_f64(int nx, int ny, int sms) {
  if ((ny + 7) / 8 > 65535) return 0;
  const auto cost = [&](int tx, int ty, double work) {
    const long long tiles = (long long)((nx + tx - 1) / tx) * ((ny + ty - 1) / ty);
    return (double)((tiles + sms - 1) / sms) * work;
  };
  const double c0 = cost(16, 16, 1.0), c1 = cost(16, 8, 0.53), c2 = cost(8, 8, 0.30);
  return c0 <= c1 && c0 <= c2 ? 0 : c1 <= c2 ? 1 : 2;
}

template <bool DUAL>
static void launch_tiles_f64(const Consts &k, int stage, const double *Un, const double *In, double *Out,
                             const double *Wn, const double *Wm, const uint8_t *tag, DevState *ds, cudaStream_t s) {
  const int shape = ibm__tile_shape_f64(k.nx, k.ny, sm_count());
#define IBM_F64(S)                                                                                    \
  (shape == 0   ? launch_tile_f64<S, DUAL, 16, 16>(k, Un, In, Out, Wn, Wm, tag, ds, s)                \
   : shape == 1 ? launch_tile_f64<S, DUAL, 16, 8>(k, Un, In, Out, Wn, Wm, tag, ds, s)                 \
                : launch_tile_f64<S, DUAL, 8, 8>(k, Un, In, Out, Wn, Wm, tag, ds, s))
  if (stage == 1) IBM_F64(1);
  else if (stage == 2) IBM_F64(2);
  else IBM_F64(3);
#undef IBM_F64
}

void launch_dual_f64(const Consts &k, int stage, const double *A, const double *In, double *Out, const double *Wn,
                     const double *Wm, const uint8_t *tag, DevState *ds, cudaStream_t s) {
  launch_tiles_f64<true>(k, stage, A, In, Out, Wn, Wm, tag, ds, s);
}

__global__ void k_dual_end(Consts k, DevState *ds) {
  ds->t = ds->t + k.dt_phys;
  ds->steps += 1;
}

void launch_dual_end(const Consts &k, DevState *ds, cudaStream_t s) { k_dual_end<<<1, 1, 0, s>>>(k, ds); }

void launch_stage_f64(const Consts &k, int stage, const double *Un, const double *In, double *Out,
                      const uint8_t *tag, DevState *ds, cudaStream_t s) {
  launch_tiles_f64<false>(k, stage, Un, In, Out, nullptr, nullptr, tag, ds, s);
}

__global__ void k_fp64_arithmetic(int op, const double *__restrict__ a, const double *__restrict__ b,
                                  double *__restrict__ out, size_t n) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const double x = a[i];
    out[i] = op == IBM_FP64_MUL     ? mul64(x, b[i])
             : op == IBM_FP64_HALF  ? half64(x)
             : op == IBM_FP64_RCP   ? rcp64(x)
             : op == IBM_FP64_RSQRT ? rsqrt64(x)
                                    : sqrt64(x);
  }
}

cudaError_t launch_fp64_arithmetic(int op, const double *a, const double *b, double *out, size_t n) {
  k_fp64_arithmetic<<<(unsigned)std::min<size_t>((n + 255) / 256, 1024), 256>>>(op, a, b, out, n);
  return cudaGetLastError();
}

}  // namespace ibm
