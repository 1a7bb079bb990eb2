// FP64 arithmetic of the residuals (2-D and 3-D).  GB300 retires two FP64 lanes per SM and clock (1.056 TFLOP/s
// measured, 1/70 of its FP32 rate), so an FP64 residual is bound by the number of FP64 instructions, and everything
// here is written to issue few of them: plain products, reciprocals and square roots on the integer pipes (the
// arguments are densities, pressures, speeds and smoothness weights in the normal range); one reciprocal shared where
// several quotients stand side by side; signs and magnitudes against 1 tested on the integer bits.  With reciprocals and
// square roots corrected on the FP64 pipe instead: 768 x 384 FP64 wedge, two steps, 1.71 ms (1.56 here); 257 x 131 FP64
// dual time 5.80 (5.25, also with the update's products off the pipe); 96 x 48 x 48 FP64 sphere 2.94 (2.76); FP32-bulk
// dual time 2048 x 1024 27.8 (25.6).
#pragma once

namespace ibm {

__device__ __forceinline__ int hi64(double x) { return __double2hiint(x); }

// a * b on the integer pipes.  An FP64 instruction holds its pipe for 16 cycles per warp, 64 issue slots of the SM's
// four schedulers, which an FP64-bound kernel leaves 93% idle; this takes about 40.  The 53-bit
// mantissas are multiplied as 64-bit integers and the whole product is rounded half up: within 1/2 ulp, equal to the
// hardware's but for ties.  (Without the partial product of the low words, 0.501 ulp and 1% less time.)
// Subnormal operands and results are zero; an infinite or NaN operand, or a product beyond the range, gives NaN (or
// infinity where the rounding alone leaves the range).  (No
// branch to the hardware multiplication: the compiler would issue it for every call.)
__device__ __forceinline__ double mul64(double a, double b) {
  const unsigned ah = __double2hiint(a), al = __double2loint(a), bh = __double2hiint(b), bl = __double2loint(b);
  const unsigned ea = ah & 0x7ff00000u, eb = bh & 0x7ff00000u, es = ea + eb;
  const unsigned xh = 0x80000000u | __funnelshift_l(al, ah, 11), xl = al << 11;
  const unsigned yh = 0x80000000u | __funnelshift_l(bl, bh, 11), yl = bl << 11;
  const unsigned long long m1 = (unsigned long long)xl * yh + __umulhi(xl, yl), m2 = (unsigned long long)xh * yl + (unsigned)m1;
  unsigned long long P = (unsigned long long)xh * yh + (m1 >> 32) + (m2 >> 32);  // the upper word, in [2^62, 2^64)
  const bool top = (long long)P < 0;
  if (!top) P += P;
  const unsigned long long q = (P >> 11) + ((unsigned)P >> 10 & 1u);  // the leading one adds 1 to the exponent
  const unsigned sign = (ah ^ bh) & 0x80000000u, et = es + (top ? 0x00100000u : 0u);
  unsigned hi = (unsigned)(q >> 32) + (et - 0x40000000u) + sign, lo = (unsigned)q;
  const bool nan = max(ea, eb) >= 0x7ff00000u || et > 0xbfd00000u;  // operand not finite, or product above the range
  const bool zero = min(ea, eb) == 0u || et < 0x40000000u;          // operand or product subnormal
  if (zero) hi = sign;
  if (nan) hi = 0x7ff80000u;
  if (zero || nan) lo = 0u;
  return __hiloint2double((int)hi, (int)lo);
}

// x / 2 on the integer pipe (exact; subnormal results are zero, infinities and NaN stay)
__device__ __forceinline__ double half64(double x) {
  const unsigned h = __double2hiint(x), e = h & 0x7ff00000u;
  const bool tiny = e < 0x00200000u;
  const unsigned hi = tiny ? h & 0x80000000u : e == 0x7ff00000u ? h : h - 0x00100000u;
  return __hiloint2double((int)hi, tiny ? 0 : __double2loint(x));
}

// 1 / x for normal x, on the integer pipes: third-order correction of an FP32 reciprocal (Householder's method: the new
// error is the old one cubed), about 35 instructions in place of three on the FP64 pipe (192 issue slots).  With m the 53-bit mantissa and Y the FP32
// reciprocal as a 24-bit integer, 2^76 - m Y is the residual e = 1 - D y in units of 2^-76, exact modulo 2^64
// (|e| < 2^-21); y (1 + e + e^2) is formed to 2^-60 and rounded to nearest: within 0.51 ulp (0.507 measured).
// NaN for zero, subnormal, infinite and NaN x; a result below the normal range is zero.
__device__ __forceinline__ double rcp64(double x) {
  const unsigned h = __double2hiint(x), l = __double2loint(x), e20 = h & 0x7ff00000u;
  float y0;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y0) : "f"(__uint_as_float(0x3f000000u | (__funnelshift_l(l, h, 3) & 0x7fffffu))));
  const unsigned Y = __float_as_uint(y0) - 0x3f000000u;  // 2^23 y0
  const long long E = -(long long)((unsigned long long)l * Y + ((unsigned long long)((h & 0xfffffu | 0x100000u) * Y) << 32));
  const int Eh = (int)(E >> 30);
  const long long c = (E + ((long long)Eh * Eh >> 16)) >> 16;  // e + e^2 in units of 2^-60
  const unsigned long long q = (((unsigned long long)Y << 39) + ((long long)Y * c >> 21) + 512u) >> 10;
  unsigned hi = (unsigned)(q >> 32) + (0x7fc00000u - e20) + (h & 0x80000000u), lo = (unsigned)q;
  const bool nan = e20 - 0x00100000u >= 0x7fe00000u, zero = e20 >= 0x7fd00000u;
  if (zero) hi = h & 0x80000000u;
  if (nan) hi = 0x7ff80000u;
  if (zero || nan) lo = 0u;
  return __hiloint2double((int)hi, (int)lo);
}

// 1 / sqrt(x) for normal x > 0, the same way: X = x 4^-k in [1, 4) as a 54-bit integer, the residual 1 - X y^2 from the
// middle 64 bits of its product with Y^2 (|e| < 2^-21, in units of 2^-68), y (1 + e / 2 + 3 e^2 / 8): within 0.51 ulp (0.508 measured).
// NaN for anything else.
__device__ __forceinline__ double rsqrt64(double x) {
  const unsigned h = __double2hiint(x), l = __double2loint(x), odd = (h >> 20) + 1u & 1u;
  float y0;
  asm("rsqrt.approx.ftz.f32 %0, %1;"
      : "=f"(y0)
      : "f"(__uint_as_float((127u + odd << 23) | (__funnelshift_l(l, h, 3) & 0x7fffffu))));
  const unsigned Y = __float_as_uint(y0) - 0x3e800000u;  // 2^24 y0
  const unsigned mh = __funnelshift_l(l, h & 0xfffffu | 0x100000u, odd), ml = l << odd;
  const unsigned long long Y2 = (unsigned long long)Y * Y;
  const unsigned yl = (unsigned)Y2, yh = (unsigned)(Y2 >> 32);
  const long long E = -(long long)(((unsigned long long)ml * yl >> 32) + (unsigned long long)ml * yh +
                                   (unsigned long long)mh * yl + ((unsigned long long)(mh * yh) << 32));
  const int Eh = (int)(E >> 24);
  const long long c = ((E >> 1) + (3 * ((long long)Eh * Eh) >> 23)) >> 8;  // e / 2 + 3 e^2 / 8 in units of 2^-60
  const unsigned long long q = (((unsigned long long)Y << 39) + ((long long)Y * c >> 21) + 512u) >> 10;
  // exponent 1022 - k with k = (biased exponent - 1023 - odd) / 2; q's leading one adds 1
  const unsigned hi = (unsigned)(q >> 32) + (0x3fd00000u + ((0x3ffu + odd) << 19) - ((h & 0x7ff00000u) >> 1));
  const bool ok = h - 0x00100000u < 0x7fe00000u;
  return __hiloint2double(ok ? (int)hi : 0x7ff80000, ok ? (int)(unsigned)q : 0);
}

// sqrt(x) for x >= 0, within 1.53 ulp; 0 for +0 and subnormal x (squares of speeds below 1e-154)
__device__ __forceinline__ double sqrt64(double x) {
  return (unsigned)hi64(x) < 0x00100000u ? 0.0 : mul64(x, rsqrt64(x));
}

// |x| < 1 (exact: the biased exponent is below 1023); false for NaN
__device__ __forceinline__ bool below_one(double x) { return (hi64(x) & 0x7fffffff) < 0x3ff00000; }
// x positive, normal and finite
__device__ __forceinline__ bool positive(double x) { return (unsigned)(hi64(x) - 1) < 0x7fefffffu; }
__device__ __forceinline__ bool negative(double x) { return hi64(x) < 0; }
// x infinite or NaN
__device__ __forceinline__ bool not_finite(double x) { return (hi64(x) & 0x7ff00000) == 0x7ff00000; }

// Sec. 2: fifth-order WENO (Jiang-Shu smoothness indicators, linear weights 1/10, 6/10, 3/10, eps = 1e-6) of one
// five-point window, both of its values: the left state at the centre's right face and, mirrored, the right state at
// its left face.  With first differences g and second differences d of the line, the indicators are
//   eps + beta_k = [eps + 13/12 d^2] + (first-difference term / 2)^2,
// whose bracket three windows share; the candidates are taken relative to the centre's value and the nonlinear
// weights d_k / (eps + beta_k)^2 cleared of their common denominator, so that each value is f + N / D and one
// reciprocal of D_L D_R serves both.  D_L D_R holds eighth powers of an indicator: in range for jumps up to about 1e19
// within a window.  About 37 FP64 instructions for two states.
struct Weno64 {
  double f, g, hg, d0, d1, e0, e1;  // centre value; g = f(c) - f(c-1) and half of it; second differences at c - 1 and
                                    // c; their brackets
  // window centred at f2; the first advance() moves to it
  __device__ __forceinline__ void start(double f0, double f1, double f2, double f3) {
    const double ga = f1 - f0, gb = f2 - f1, gc = f3 - f2;
    f = f2;
    g = gb;
    hg = half64(gb);
    d0 = gb - ga;
    d1 = gc - gb;
    e0 = fma(mul64(13.0 / 12.0, d0), d0, 1e-6);
    e1 = fma(mul64(13.0 / 12.0, d1), d1, 1e-6);
  }
  // the two states of the window at f, f3 and f4 the values one and two beyond it; then moves the window on
  __device__ __forceinline__ void next(double f3, double f4, double &qL, double &qR) {
    const double g0 = f3 - f, hg0 = half64(g0), d2 = (f4 - f3) - g0, e2 = fma(mul64(13.0 / 12.0, d2), d2, 1e-6);
    const double b0 = fma(0.5, d0, g), b1 = fma(0.5, d1, g), b2 = fma(0.5, d2, -g0);
    const double i0 = fma(b0, b0, e0), i1 = fma(b1, b1, e1), i2 = fma(b2, b2, e2);
    const double t0 = mul64(i0, i0), t1 = mul64(i1, i1), t2 = mul64(i2, i2);
    const double s12 = mul64(t1, t2), s02 = mul64(t0, t2), s01 = mul64(t0, t1);
    // left: candidates less f times (1, 6, 3), the linear weights in units of 1/10
    const double l0 = fma(1.0 / 3.0, d0, hg), l1 = fma(3.0, g0, -d1), l2 = hg0 - b2;
    const double NL = fma(s12, l0, fma(s02, l1, mul64(s01, l2))), DL = fma(6.0, s02, fma(3.0, s01, s12));
    const double r0 = fma(1.0 / 3.0, d2, -hg0), r1 = fma(-3.0, g, -d1), r2 = -hg - b0;
    const double NR = fma(s01, r0, fma(s02, r1, mul64(s12, r2))), DR = fma(6.0, s02, fma(3.0, s12, s01));
    const double inv = rcp64(mul64(DL, DR));
    qL = fma(mul64(NL, DR), inv, f);
    qR = fma(mul64(NR, DL), inv, f);
    f = f3;
    g = g0;
    hg = hg0;
    d0 = d1;
    d1 = d2;
    e0 = e1;
    e1 = e2;
  }
};

// Sec. 2, LDFSS(0) with D tangential velocity components: face flux of the states (rho, un, ut..., p), F = (mass,
// normal momentum, tangential momenta..., energy).  PRE: the dual-time low-Mach form -- numerical sound speed
// c' = 1/2 sqrt((1 - Mr^2)^2 un^2 + 4 Mr^2 c^2) of the reference velocity Ur = min(c, max(|V|, U_ref, nu/dn)) (face
// averages; taken by squares), pressure split in the physical Mach numbers with its departure from the face mean
// scaled by c'/c.  munu2 = (mu / dn)^2.
template <bool PRE, int D>
__device__ __forceinline__ void ldfss64(double rL, double unL, const double utL[D], double pL, double rR, double unR,
                                        const double utR[D], double pR, double gamma, double ig1, double munu2,
                                        double F[3 + D]) {
  const double irr = rcp64(mul64(rL, rR)), irL = mul64(irr, rR), irR = mul64(irr, rL);
  const double c2L = mul64(mul64(gamma, pL), irL), c2R = mul64(mul64(gamma, pR), irR);
  const double cL = mul64(c2L, rsqrt64(c2L)), cR = mul64(c2R, rsqrt64(c2R));
  double kL = mul64(unL, unL), kR = mul64(unR, unR);
#pragma unroll
  for (int d = 0; d < D; d++) {
    kL = fma(utL[d], utL[d], kL);
    kR = fma(utR[d], utR[d], kR);
  }
  const double HL = fma(0.5, kL, mul64(c2L, ig1)), HR = fma(0.5, kR, mul64(c2R, ig1));  // gamma/(gamma-1) p/rho = c^2/(gamma-1)
  const double cb = half64(cL + cR), icb = rcp64(cb);
  double cs = cb, ics = icb;
  bool low = false;
  if (PRE) {
    const double ub = half64(unL + unR);
    double v2 = mul64(ub, ub);
#pragma unroll
    for (int d = 0; d < D; d++) {
      const double vb = half64(utL[d] + utR[d]);
      v2 = fma(vb, vb, v2);
    }
    const double rb = half64(rL + rR), rb2 = mul64(rb, rb), cb2 = mul64(cb, cb);
    double ur2 = fmax(v2, 1.0);
    if (munu2 > mul64(ur2, rb2)) ur2 = mul64(munu2, rcp64(rb2));
    if (ur2 < cb2) {
      low = true;
      const double t = mul64(half64(fma(-mul64(ur2, icb), icb, 1.0)), ub);
      const double x = fma(t, t, ur2);
      ics = rsqrt64(x);
      cs = mul64(x, ics);
    }
  }
  const double ML = mul64(unL, ics), MR = mul64(unR, ics);
  const bool subL = below_one(ML), subR = below_one(MR);
  const double aL = half64(ML + 1.0), aR = half64(MR - 1.0);
  const double MpL = mul64(aL, aL), MmR = -mul64(aR, aR);
  const double CL = subL ? MpL : (negative(ML) ? 0.0 : ML), CR = subR ? MmR : (negative(MR) ? MR : 0.0);
  const double sq = half64(sqrt64(half64(fma(ML, ML, mul64(MR, MR)))) - 1.0);
  const double Mh = subL && subR ? mul64(sq, sq) : 0.0;
  // only the side that the pressure falls to is weighted: M_1/2 (1 - |dp| / (rho c'^2))
  const double dp = pL - pR;
  const bool up = negative(dp);
  const double Mw = mul64(Mh, fma(-fabs(dp), mul64(up ? irR : irL, mul64(ics, ics)), 1.0));
  const double Cp = CL - (up ? Mh : Mw), Cm = CR + (up ? Mw : Mh);
  double DL, DR, ph;
  if (PRE && low) {
    const double mL = mul64(unL, icb), mR = mul64(unR, icb), bL = half64(mL + 1.0), bR = half64(mR - 1.0);
    DL = below_one(mL) ? mul64(mul64(bL, bL), 2.0 - mL) : (negative(mL) ? 0.0 : 1.0);
    DR = below_one(mR) ? mul64(mul64(bR, bR), 2.0 + mR) : (negative(mR) ? 1.0 : 0.0);
    ph = fma(mul64(cs, icb), fma(DL - 0.5, pL, mul64(DR - 0.5, pR)), half64(pL + pR));
  } else {
    DL = subL ? mul64(MpL, 2.0 - ML) : (negative(ML) ? 0.0 : 1.0);
    DR = subR ? -mul64(MmR, 2.0 + MR) : (negative(MR) ? 1.0 : 0.0);
    ph = fma(DL, pL, mul64(DR, pR));
  }
  const double mL = mul64(mul64(rL, cs), Cp), mR = mul64(mul64(rR, cs), Cm);
  F[0] = mL + mR;
  F[1] = fma(mL, unL, fma(mR, unR, ph));
#pragma unroll
  for (int d = 0; d < D; d++) F[2 + d] = fma(mL, utL[d], mul64(mR, utR[d]));
  F[2 + D] = fma(mL, HL, mul64(mR, HR));
}

}  // namespace ibm
