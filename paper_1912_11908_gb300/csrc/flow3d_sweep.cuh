// 3-D residual by directional sweeps, FP64 and FP32-bulk (included by flow3d.cu).
//
// A sweep forms the face fluxes of one direction -- WENO5 states, LDFSS(0), central viscous flux (Sec. 2) -- and adds
// their difference to the cells' flux divergence: y first, then z, then x with the stage update (its warps need no
// block barrier, so the update's operands load while others compute).  No face flux goes to memory, and a WENO window
// is formed once per cell and direction: it gives the left state of the cell's upper face and the right state of its
// lower face from shared differences.
// Lanes run along x in every sweep (coalesced); the neighbouring window's state and the neighbouring face's flux come
//   x: by shuffles -- a warp's 32 windows give 31 faces and 30 cells;
//   y, z: through shared memory -- a block's rows of windows give one face less and two cells less.
// One thread per face with both windows of every face, and flux arrays in memory, took 1.5x the instructions and 35
// array passes per stage; a thread marching along y or z with the windows sliding through registers took fewest
// instructions but waits on memory with too few warps (192 x 96 x 96, FP32-bulk, per sweep: 65 us by faces, 129 us
// marching, 52 here).  FP32-bulk is bound by issue slots (74-80% busy) and, in the x sweep, by the update's operands;
// FP64 by the FP64 pipe.  A step: FP32-bulk 192 x 96 x 96 0.95 -> 0.75 ms, FP64 96 x 48 x 48 3.92 -> 1.46 ms (1.38 with
// the reciprocals on the integer pipes).
#pragma once

#include "fp64_math.cuh"

namespace {

using ibm::ldfss64;
using ibm::positive;
using ibm::Weno64;

__device__ __forceinline__ float mulx(float a, float b) { return a * b; }
__device__ __forceinline__ double mulx(double a, double b) { return mul64(a, b); }

// The FP32 form of Weno64 (fp64_math.cuh): the nonlinear weights through reciprocals of the indicators (in range for
// indicators up to 1e19), one quotient per state.
struct Weno32 {
  float f, g, d0, d1, e0, e1;
  __device__ __forceinline__ void start(float f0, float f1, float f2, float f3) {
    const float ga = f1 - f0, gb = f2 - f1, gc = f3 - f2;
    f = f2;
    g = gb;
    d0 = gb - ga;
    d1 = gc - gb;
    e0 = fmaf((13.0f / 12.0f) * d0, d0, 1e-6f);
    e1 = fmaf((13.0f / 12.0f) * d1, d1, 1e-6f);
  }
  __device__ __forceinline__ void next(float f3, float f4, float &qL, float &qR) {
    const float g0 = f3 - f, d2 = (f4 - f3) - g0, e2 = fmaf((13.0f / 12.0f) * d2, d2, 1e-6f);
    const float b0 = fmaf(0.5f, d0, g), b1 = fmaf(0.5f, d1, g), b2 = fmaf(0.5f, d2, -g0);
    const float i0 = __fdividef(1.0f, fmaf(b0, b0, e0)), i1 = __fdividef(1.0f, fmaf(b1, b1, e1)),
                i2 = __fdividef(1.0f, fmaf(b2, b2, e2));
    const float w0 = i0 * i0, w1 = i1 * i1, w2 = i2 * i2;
    const float l0 = fmaf(1.0f / 3.0f, d0, 0.5f * g), l1 = fmaf(3.0f, g0, -d1), l2 = fmaf(0.5f, g0, -b2);
    const float NL = fmaf(w0, l0, fmaf(w1, l1, w2 * l2)), DL = fmaf(6.0f, w1, fmaf(3.0f, w2, w0));
    const float r0 = fmaf(1.0f / 3.0f, d2, -0.5f * g0), r1 = fmaf(-3.0f, g, -d1), r2 = fmaf(-0.5f, g, -b0);
    const float NR = fmaf(w2, r0, fmaf(w1, r1, w0 * r2)), DR = fmaf(6.0f, w1, fmaf(3.0f, w0, w2));
    qL = f + __fdividef(NL, DL);
    qR = f + __fdividef(NR, DR);
    f = f3;
    g = g0;
    d0 = d1;
    d1 = d2;
    e0 = e1;
    e1 = e2;
  }
};

template <class T>
struct Window;
template <>
struct Window<float> : Weno32 {};
template <>
struct Window<double> : Weno64 {};

// parameters of a sweep: FP64 absolute variables, or FP32 perturbations (P32)
struct P64 {
  double gamma, ig1, mu, ih[3];
  double vn[3], vt[3], kq[3];  // mu / h, mu / (4 h), kappa / h per axis
};

template <class T>
struct Real;
template <>
struct Real<float> {
  using Par = P32;
  using Q = F6f;
  using L = F5f;
};
template <>
struct Real<double> {
  using Par = P64;
  using Q = F6;
  using L = F5;
};

// first-order states where a reconstructed density or pressure is not positive
__device__ __forceinline__ bool states_ok(const P64 &, const double qL[5], const double qR[5]) {
  return positive(qL[0]) && positive(qL[4]) && positive(qR[0]) && positive(qR[4]);
}
__device__ __forceinline__ bool states_ok(const P32 &c, const float qL[5], const float qR[5]) {
  return 1.0f + qL[0] > 0.0f && c.pinf + qL[4] > 0.0f && 1.0f + qR[0] > 0.0f && c.pinf + qR[4] > 0.0f;
}

// LDFSS(0) (Mr = 1) across a face normal to axis DIR; F in the order of the conserved variables
template <int DIR>
__device__ __forceinline__ void inviscid(const P64 &c, const double qL[5], const double qR[5], double F[5]) {
  constexpr int t1 = DIR == 0 ? 1 : 0, t2 = DIR == 2 ? 1 : 2;
  const double uL[2] = {qL[1 + t1], qL[1 + t2]}, uR[2] = {qR[1 + t1], qR[1 + t2]};
  double f[5];
  ldfss64<false, 2>(qL[0], qL[1 + DIR], uL, qL[4], qR[0], qR[1 + DIR], uR, qR[4], c.gamma, c.ig1, 0.0, f);
  F[0] = f[0];
  F[1 + DIR] = f[1];
  F[1 + t1] = f[2];
  F[1 + t2] = f[3];
  F[4] = f[4];
}
// on perturbation states q' = (rho', u', v', w', p'): F = mass, momentum less p_inf n, rho u H'
template <int DIR>
__device__ __forceinline__ void inviscid(const P32 &c, const float qL[5], const float qR[5], float F[5]) {
  const float rL = 1.0f + qL[0], rR = 1.0f + qR[0];
  const float irL = __fdividef(1.0f, rL), irR = __fdividef(1.0f, rR);
  const float c2L = c.gamma * (c.pinf + qL[4]) * irL, c2R = c.gamma * (c.pinf + qR[4]) * irR;
  const float cL = c2L * rsqrtf(c2L), cR = c2R * rsqrtf(c2R);  // sound speeds (approximate square roots)
  float uL[3], uR[3];
  // H' = gamma/(gamma-1) (p / rho - p_inf) + (|u|^2 - |U_inf|^2) / 2
  float kL = 0.0f, kR = 0.0f;
#pragma unroll
  for (int a = 0; a < 3; a++) {
    uL[a] = c.u0[a] + qL[1 + a];
    uR[a] = c.u0[a] + qR[1 + a];
    kL = fmaf(qL[1 + a], c.u0[a] + uL[a], kL);
    kR = fmaf(qR[1 + a], c.u0[a] + uR[a], kR);
  }
  const float HL = fmaf(0.5f, kL, c.gg * fmaf(-c.pinf, qL[0], qL[4]) * irL);
  const float HR = fmaf(0.5f, kR, c.gg * fmaf(-c.pinf, qR[0], qR[4]) * irR);
  const float unL = uL[DIR], unR = uR[DIR];
  const float cs = 0.5f * (cL + cR), ics = __fdividef(1.0f, cs);
  const float ML = unL * ics, MR = unR * ics;
  const bool subL = fabsf(ML) < 1.0f, subR = fabsf(MR) < 1.0f;
  const float aL = 0.5f * ML + 0.5f, aR = 0.5f * MR - 0.5f;
  const float MpL = aL * aL, MmR = -aR * aR;
  const float CL = subL ? MpL : fmaxf(ML, 0.0f), CR = subR ? MmR : fminf(MR, 0.0f);
  const float m2 = 0.5f * fmaf(ML, ML, MR * MR);
  const float sq = 0.5f * ((m2 > 0.0f ? m2 * rsqrtf(m2) : 0.0f) - 1.0f);
  const float Mh = subL && subR ? sq * sq : 0.0f;
  const float dp = qL[4] - qR[4], ic2 = ics * ics;
  const float Cp = CL - Mh * (1.0f - fmaxf(dp, 0.0f) * ic2 * irL);
  const float Cm = CR + Mh * (1.0f - fmaxf(-dp, 0.0f) * ic2 * irR);
  const float DL = subL ? MpL * (2.0f - ML) : (ML >= 0.0f ? 1.0f : 0.0f);
  const float DR = subR ? -MmR * (2.0f + MR) : (MR >= 0.0f ? 0.0f : 1.0f);
  // D_L + D_R - 1 factored between two subsonic sides, so that p_inf times it keeps its digits
  const float Dm1 = subL && subR ? 0.25f * (MR - ML) * fmaf(MR, MR, fmaf(MR, ML, fmaf(ML, ML, -3.0f))) : (DL + DR) - 1.0f;
  const float mL = rL * cs * Cp, mR = rR * cs * Cm;
  F[0] = mL + mR;
#pragma unroll
  for (int a = 0; a < 3; a++) F[1 + a] = fmaf(mL, uL[a], mR * uR[a]);
  F[1 + DIR] += fmaf(c.pinf, Dm1, fmaf(DL, qL[4], DR * qR[4]));
  F[4] = fmaf(mL, HL, mR * HR);
}

// the free-stream velocity that perturbations leave out, twice
__device__ __forceinline__ float twice_base(const P32 &c, int a) { return 2.0f * c.u0[a]; }
__device__ __forceinline__ double twice_base(const P64 &, int) { return 0.0; }

// viscous part of the face between cells a and b along DIR: ua, ub the cells' velocities (perturbations), dT their
// temperature difference, D1 / D2 the sums of the two cells' central differences along the tangents t1 < t2
template <int DIR, class T, class Par>
__device__ __forceinline__ void viscous(const Par &c, const T ua[3], const T ub[3], T dT, const T D1[3], const T D2[3],
                                        T F[5]) {
  constexpr int t1 = DIR == 0 ? 1 : 0, t2 = DIR == 2 ? 1 : 2;
  T G[3][3];  // mu d u_c / d x_e
#pragma unroll
  for (int e = 0; e < 3; e++) {
    G[e][DIR] = mulx(ub[e] - ua[e], c.vn[DIR]);
    G[e][t1] = mulx(D1[e], c.vt[t1]);
    G[e][t2] = mulx(D2[e], c.vt[t2]);
  }
  const T div = G[0][0] + G[1][1] + G[2][2];
  T work = T(0);  // twice the work of the stress
#pragma unroll
  for (int e = 0; e < 3; e++) {
    const T tau = e == DIR ? fma(T(2), G[DIR][DIR], mulx(T(-2.0 / 3.0), div)) : G[e][DIR] + G[DIR][e];
    F[1 + e] -= tau;
    work = fma(twice_base(c, e) + ua[e] + ub[e], tau, work);
  }
  F[4] = fma(-c.kq[DIR], dT, fma(T(-0.5), work, F[4]));
}

template <int DIR>
__device__ __forceinline__ long long stride_of(const Grid3 &g) {
  return DIR == 0 ? 1 : DIR == 1 ? (long long)g.W : g.plane;
}

// x sweep: block of 32 lanes along x, BY rows; a warp covers the cells bx * 30 .. + 29 and one window on each side;
// done(cell index, j, k, i, divergence of this direction) for every cell.  Every lane of a warp calls it.
constexpr int XCELLS = 30;
template <class T, class Done>
__device__ __forceinline__ void sweep_x(const Grid3 &g, const typename Real<T>::Par &c, const typename Real<T>::Q &Q,
                                        int j, int k, Done done) {
  const int lane = threadIdx.x;
  const int ci = blockIdx.x * XCELLS - 1 + lane, i = min(ci, g.nx);
  const long long a = cid(g, i, j, k);
  T q[5], qL[5], qR[5], un[3];
#pragma unroll
  for (int v = 0; v < 5; v++) {
    const T *p = Q.v[v] + a;
    Window<T> w;
    const T f3 = p[1];
    q[v] = p[0];
    w.start(p[-2], p[-1], q[v], f3);
    T r;
    w.next(f3, p[2], qL[v], r);
    qR[v] = __shfl_down_sync(0xffffffffu, r, 1);  // the right state of the face between this cell and the next
    if (v >= 1 && v <= 3) un[v - 1] = f3;
  }
  // the fallback's right state: the next cell's values
  if (!states_ok(c, qL, qR)) {
#pragma unroll
    for (int v = 0; v < 5; v++) {
      qL[v] = q[v];
      qR[v] = Q.v[v][a + 1];
    }
  }
  T F[5];
  inviscid<0>(c, qL, qR, F);
  if (c.mu > T(0)) {
    T D1[3], D2[3];
#pragma unroll
    for (int e = 0; e < 3; e++) {
      const T *p = Q.v[1 + e] + a;
      const T y = p[g.W] - p[-g.W], z = p[g.plane] - p[-g.plane];
      D1[e] = y + __shfl_down_sync(0xffffffffu, y, 1);
      D2[e] = z + __shfl_down_sync(0xffffffffu, z, 1);
    }
    viscous<0, T>(c, q + 1, un, Q.v[5][a + 1] - Q.v[5][a], D1, D2, F);
  }
  const bool cell = lane >= 1 && lane <= XCELLS && ci < g.nx;
  T d[5];
#pragma unroll
  for (int v = 0; v < 5; v++) d[v] = mulx(F[v] - __shfl_up_sync(0xffffffffu, F[v], 1), c.ih[0]);
  if (cell) done(a, ci, d);
}

// y and z sweeps: a block of 16 lanes along x (whole sectors; 32 lanes leave two blocks per SM, 60 us for 52) and up to
// SROWS rows along DIR, one window per row; the y sweep writes
// the cells' divergence, the z sweep adds to it.  Every thread of the block calls it.
constexpr int SROWS = 16, SLANES = 16;
constexpr int GRID_YZ_MAX = 65535;  // gridDim.y and gridDim.z
template <class T>
struct SweepSmem {
  T x[11][SROWS][SLANES];  // right states (then fluxes) and the tangential differences of the rows
  // FP32: the rows' values with two rows on either side, each loaded once -- the FP32 sweep's loads are all in flight
  // together, where five loads per window in turn left it waiting on them.  The FP64 sweep is bound
  // by the FP64 pipe either way.
  T q[sizeof(T) == 4 ? 5 : 1][sizeof(T) == 4 ? SROWS + 4 : 1][SLANES];
};
template <int DIR, class T>
__device__ __forceinline__ void sweep_yz(const Grid3 &g, const typename Real<T>::Par &c, const typename Real<T>::Q &Q,
                                         const typename Real<T>::L &Lo, int i, int o, SweepSmem<T> &sm) {
  const int n = DIR == 1 ? g.ny : g.nz, row = threadIdx.y, last = blockDim.y - 1, lane = threadIdx.x;
  const int cc = blockIdx.z * (last - 1) - 1 + row, cl = min(cc, n), ic = min(i, g.nx - 1);
  const long long st = stride_of<DIR>(g), s2 = DIR == 1 ? g.plane : (long long)g.W;
  const long long a = DIR == 1 ? cid(g, ic, cl, o) : cid(g, ic, o, cl);
  constexpr bool staged = sizeof(T) == 4;
  const bool vis = c.mu > T(0), cell = row >= 1 && row < last && cc < n && i < g.nx;
  T q[5], qL[5], un[3], D1[3], D2[3], dT = T(0), sum[5];
  // every load of the sweep before the first barrier
  if (staged) {
    // rows cc - 2 .. cc + 2 of the block (clamped to the last halo row)
    const int c0 = blockIdx.z * (last - 1) - 3;
    for (int r = row; r < last + 5; r += last + 1) {
      const int cr = min(c0 + r, n + 2);
      const long long m = DIR == 1 ? cid(g, ic, cr, o) : cid(g, ic, o, cr);
#pragma unroll
      for (int v = 0; v < 5; v++) sm.q[v][r][lane] = Q.v[v][m];
    }
  }
  if (vis) {
#pragma unroll
    for (int e = 0; e < 3; e++) {
      const T *p = Q.v[1 + e] + a;
      D1[e] = p[1] - p[-1];
      D2[e] = p[s2] - p[-s2];
    }
    dT = Q.v[5][a + st] - Q.v[5][a];
  }
  if (DIR == 2 && cell) {  // the y sweep's sum
#pragma unroll
    for (int v = 0; v < 5; v++) sum[v] = Lo.v[v][a];
  }
  if (staged) __syncthreads();
#pragma unroll
  for (int v = 0; v < 5; v++) {
    T f[5];
#pragma unroll
    for (int t = 0; t < 5; t++) f[t] = staged ? sm.q[staged ? v : 0][staged ? row + t : 0][lane] : Q.v[v][a + (t - 2) * st];
    Window<T> w;
    q[v] = f[2];
    w.start(f[0], f[1], f[2], f[3]);
    T r;
    w.next(f[3], f[4], qL[v], r);
    sm.x[v][row][lane] = r;  // the right state of the face between the row before and this one
    if (v >= 1 && v <= 3) un[v - 1] = f[3];
  }
  if (vis) {
#pragma unroll
    for (int e = 0; e < 3; e++) {
      sm.x[5 + e][row][lane] = D1[e];
      sm.x[8 + e][row][lane] = D2[e];
    }
  }
  __syncthreads();
  T F[5];
  if (row < last) {  // the face between this row's cell and the next
    T qR[5];
#pragma unroll
    for (int v = 0; v < 5; v++) qR[v] = sm.x[v][row + 1][lane];
    if (!states_ok(c, qL, qR)) {
#pragma unroll
      for (int v = 0; v < 5; v++) {
        qL[v] = q[v];
        qR[v] = Q.v[v][a + st];
      }
    }
    inviscid<DIR>(c, qL, qR, F);
    if (vis) {
#pragma unroll
      for (int e = 0; e < 3; e++) {
        D1[e] += sm.x[5 + e][row + 1][lane];
        D2[e] += sm.x[8 + e][row + 1][lane];
      }
      viscous<DIR, T>(c, q + 1, un, dT, D1, D2, F);
    }
  }
  __syncthreads();
  if (row < last) {
#pragma unroll
    for (int v = 0; v < 5; v++) sm.x[v][row][lane] = F[v];
  }
  __syncthreads();
  if (cell) {
#pragma unroll
    for (int v = 0; v < 5; v++) {
      const T d = mulx(F[v] - sm.x[v][row - 1][lane], c.ih[DIR]);
      Lo.v[v][a] = DIR == 1 ? d : sum[v] + d;
    }
  }
}

template <int DIR, class T>
__global__ void __launch_bounds__(SLANES *SROWS) k3_sweep_yz(Grid3 g, typename Real<T>::Par c, typename Real<T>::Q Q,
                                                          typename Real<T>::L Lo, int o0) {
  __shared__ SweepSmem<T> sm;
  sweep_yz<DIR, T>(g, c, Q, Lo, blockIdx.x * SLANES + threadIdx.x, o0 + blockIdx.y, sm);
}

// the y (DIR 1) or z (DIR 2) sweep in blocks of `rows` rows: gridDim.y runs over the cells of the third axis, at most
// 65,535 of them per launch (one launch for any usual grid); returns the launches
template <int DIR, class T>
inline int launch_sweep_yz(const Grid3 &g, const typename Real<T>::Par &c, const typename Real<T>::Q &Q,
                           const typename Real<T>::L &Lo, int rows, cudaStream_t s) {
  const int n = DIR == 1 ? g.ny : g.nz, no = DIR == 1 ? g.nz : g.ny;
  int launches = 0;
  for (int o0 = 0; o0 < no; o0 += GRID_YZ_MAX, launches++)
    k3_sweep_yz<DIR, T><<<dim3((g.nx + SLANES - 1) / SLANES, std::min(no - o0, GRID_YZ_MAX), (n + rows - 3) / (rows - 2)),
                          dim3(SLANES, rows), 0, s>>>(g, c, Q, Lo, o0);
  return launches;
}

// x sweep with the SSP-RK3 stage on the fluid cells: out = Un - dt D, 3/4 Un + 1/4 (in - dt D),
// 1/3 Un + 2/3 (in - dt D), D the flux divergence of the three directions
template <int STAGE>
__global__ void __launch_bounds__(TC) k3_sweep_x(Grid3 g, P64 c, F6 Q, F5 Lo, F5 Un, F5 In, F5 Out,
                                                 const uint8_t *__restrict__ tags, const double *__restrict__ dtp) {
  const int j = blockIdx.y * BY + threadIdx.y, k = blockIdx.z;
  if (j >= g.ny) return;  // whole warps
  const double dt = *dtp;
  sweep_x<double>(g, c, Q, j, k, [&](long long m, int i, const double d[5]) {
    if (tags[((long long)k * g.ny + j) * g.nx + i] != TAG_FLUID) return;
#pragma unroll
    for (int v = 0; v < 5; v++) {
      const double D = Lo.v[v][m] + d[v], un = Un.v[v][m];
      if (STAGE == 1) Out.v[v][m] = fma(-dt, D, un);
      else if (STAGE == 2) Out.v[v][m] = fma(0.75, un, half64(half64(fma(-dt, D, In.v[v][m]))));
      else Out.v[v][m] = fma(1.0 / 3.0, un, mul64(2.0 / 3.0, fma(-dt, D, In.v[v][m])));
    }
  });
}

// FP32-bulk: on perturbations with M the mirror of U^n (the energy row regains H_inf times the mass row);
// stages 1 and 2 out = M - dt D, M + ((In - M) - dt D) / 4; stage 3 accumulates the FP32 increment
// 2/3 ((In - M) - dt D) onto the FP64 master A, whose new value refreshes the mirror
template <int STAGE>
__global__ void __launch_bounds__(TC) k3_sweep_x32(Grid3 g, Phys3 ph, P32 c, F6f Q, F5f Lo, F5f M, F5f In, F5f Out,
                                                   F5 A, const uint8_t *__restrict__ tags,
                                                   const double *__restrict__ dtp) {
  const int j = blockIdx.y * BY + threadIdx.y, k = blockIdx.z;
  if (j >= g.ny) return;  // whole warps
  const float dt = (float)*dtp;
  // the update's operands, read at the end, are on their way to L2 while the sweep computes (one line per plane and
  // warp, two where the warp's cells straddle lines)
  if (threadIdx.x == 1 || threadIdx.x == XCELLS) {
    const long long m = cid(g, min((int)(blockIdx.x * XCELLS - 1 + threadIdx.x), g.nx - 1), j, k);
#pragma unroll
    for (int v = 0; v < 5; v++) {
      asm volatile("prefetch.global.L2 [%0];" ::"l"(Lo.v[v] + m));
      asm volatile("prefetch.global.L2 [%0];" ::"l"(M.v[v] + m));
      if (STAGE >= 2) asm volatile("prefetch.global.L2 [%0];" ::"l"(In.v[v] + m));
      if (STAGE == 3) asm volatile("prefetch.global.L2 [%0];" ::"l"(A.v[v] + m));
    }
  }
  sweep_x<float>(g, c, Q, j, k, [&](long long m, int i, const float d[5]) {
    if (tags[((long long)k * g.ny + j) * g.nx + i] != TAG_FLUID) return;
    float D[5];
#pragma unroll
    for (int v = 0; v < 5; v++) D[v] = Lo.v[v][m] + d[v];
    D[4] = fmaf(c.Hinf, D[0], D[4]);
#pragma unroll
    for (int v = 0; v < 5; v++) {
      const float mv = M.v[v][m];
      if (STAGE == 1) {
        Out.v[v][m] = fmaf(-dt, D[v], mv);
      } else if (STAGE == 2) {
        Out.v[v][m] = fmaf(0.25f, fmaf(-dt, D[v], In.v[v][m] - mv), mv);
      } else {
        const float inc = (2.0f / 3.0f) * fmaf(-dt, D[v], In.v[v][m] - mv);
        const double a = A.v[v][m] + (double)inc;
        A.v[v][m] = a;
        M.v[v][m] = (float)(a - ph.Uinf[v]);
      }
    }
  });
}

// rows of a y or z sweep's blocks over n cells: r rows give r - 2 cells; the fewest rows in all (the longer block on a
// tie)
inline int sweep_rows(int n) {
  int best = SROWS;
  for (int r = SROWS; r >= 8; r--)
    if ((n + r - 3) / (r - 2) * r < (n + best - 3) / (best - 2) * best) best = r;
  return best;
}

}  // namespace
