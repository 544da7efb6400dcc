// Device arithmetic of the FD-CGKS hot path, templated on the compute type R
// (double for the FP64 path, float for the mixed path).  Everything here is
// __host__ __device__ so that the same source can be instantiated on the host
// with an operation-counting scalar to obtain exact algorithmic flop counts.
//
// Paper: "Finite Difference Implementation of a High-order Space-Time Coupled
// Compact Gas-Kinetic Scheme" (Zhao, Chen, Xu).
#pragma once

#include <math.h>
#include <string.h>

#include "fdcgks_gauss_table.h"

#if defined(__CUDACC__)
#define FD_HD __host__ __device__ __forceinline__
#else
#define FD_HD inline
#endif

namespace fdk {

// ---------------------------------------------------------------------------
// scalar helpers (overload points for other scalar types)
// ---------------------------------------------------------------------------
FD_HD double s_sqrt(double x) { return sqrt(x); }
FD_HD float s_sqrt(float x) { return sqrtf(x); }
FD_HD double s_rsqrt(double x) {
#if defined(__CUDA_ARCH__)
  return rsqrt(x);
#else
  return 1.0 / sqrt(x);
#endif
}
FD_HD float s_rsqrt(float x) {
#if defined(__CUDA_ARCH__)
  return rsqrtf(x);
#else
  return 1.0f / sqrtf(x);
#endif
}
template <class R> FD_HD R s_rsqrt(R x) { return R(1) / s_sqrt(x); }   // other scalar types
FD_HD double s_exp(double x) { return exp(x); }
FD_HD float s_exp(float x) { return expf(x); }
FD_HD double s_erfc(double x) { return erfc(x); }
FD_HD float s_erfc(float x) { return erfcf(x); }
FD_HD double s_tanh(double x) { return tanh(x); }
FD_HD float s_tanh(float x) { return tanhf(x); }
FD_HD double s_abs(double x) { return fabs(x); }
FD_HD float s_abs(float x) { return fabsf(x); }
FD_HD double s_min(double a, double b) { return fmin(a, b); }
FD_HD float s_min(float a, float b) { return fminf(a, b); }
FD_HD double s_max(double a, double b) { return fmax(a, b); }
FD_HD float s_max(float a, float b) { return fmaxf(a, b); }
FD_HD double s_expm1(double x) { return expm1(x); }
FD_HD float s_expm1(float x) { return expm1f(x); }

// The FP64 part of the arithmetic (collision time and time coefficients) runs
// in Wide<R>::T: double for both compute types; an instrumented scalar type
// maps to its own wide counterpart.
template <class R> struct Wide { typedef double T; };
template <class R> FD_HD typename Wide<R>::T to_w(R x) { return (typename Wide<R>::T)x; }
template <class R> FD_HD R from_w(typename Wide<R>::T x) { return (R)x; }

// Division in the compute type: IEEE in FP64; in FP32 on the device the
// fast division x * (1/y) with an approximate reciprocal (2 ulp), which is
// below the FP32 path's own error.  Denominators here are bounded away from
// 0 and from 2^126.
FD_HD double s_div(double a, double b) { return a / b; }
FD_HD float s_div(float a, float b) {
#if defined(__CUDA_ARCH__)
  return __fdividef(a, b);
#else
  return a / b;
#endif
}

// erfc(x) given ex2 = exp(-x^2), which the caller has already computed.
// FP64: erfc(|x|) = exp(-x^2) erfcx(|x|) with the library's scaled function
// erfcx, and erfc(x) = 2 - erfc(-x) for x < 0, so the exponential is not
// evaluated twice (1.7 % of the FP64 point kernel's time on the 1024^2
// vortex).  FP32: the library erfcf, which keeps a few ulp of relative
// accuracy where erfc is small, while an absolute-error approximation (e.g.
// Abramowitz & Stegun 7.1.26, |error| <= 1.5e-7, written as a polynomial times
// exp(-x^2)) is off by up to 1e-3 relative there; that inconsistency between
// the half-space moments of the two sides seeded a grid-scale mode across the
// strong shock of the 1000 x 500 viscous shock tube in the mixed path.
FD_HD double s_erfc_e(double x, double ex2) {
#if defined(__CUDA_ARCH__)
  const double r = ex2 * erfcx(fabs(x));
  return x >= 0.0 ? r : 2.0 - r;
#else
  (void)ex2;   // host builds (tests, the flop counter): the C library has no erfcx
  return erfc(x);
#endif
}
FD_HD float s_erfc_e(float x, float ex2) { (void)ex2; return erfcf(x); }

// the words of an FP64 value and the bits of an FP32 one
FD_HD void words_of(double x, unsigned& hi, unsigned& lo) {
#if defined(__CUDA_ARCH__)
  hi = (unsigned)__double2hiint(x);
  lo = (unsigned)__double2loint(x);
#else
  unsigned long long b;
  memcpy(&b, &x, sizeof(b));
  hi = (unsigned)(b >> 32);
  lo = (unsigned)b;
#endif
}
FD_HD double of_words(unsigned hi, unsigned lo) {
#if defined(__CUDA_ARCH__)
  return __hiloint2double((int)hi, (int)lo);
#else
  const unsigned long long b = (unsigned long long)hi << 32 | lo;
  double x;
  memcpy(&x, &b, sizeof(x));
  return x;
#endif
}
FD_HD unsigned bits_of(float x) {
#if defined(__CUDA_ARCH__)
  return __float_as_uint(x);
#else
  unsigned b;
  memcpy(&b, &x, sizeof(b));
  return b;
#endif
}
FD_HD float of_bits(unsigned b) {
#if defined(__CUDA_ARCH__)
  return __uint_as_float(b);
#else
  float x;
  memcpy(&x, &b, sizeof(x));
  return x;
#endif
}

// FP32 copy of an FP64 value, rounded toward zero (for estimates and small terms):
// shifts of its words, which cost the integer pipe 5 operations where a
// conversion takes a slot of the FP64 pipe.  Zero below 2^-126, infinite from
// 2^128 on; NaN becomes infinite.
FD_HD float est_f32(double x) {
  unsigned hi, lo;
  words_of(x, hi, lo);
  const unsigned a = hi & 0x7fffffffu;
  unsigned m = (a - 0x38000000u) << 3 | lo >> 29;
  m = a < 0x38100000u ? 0u : a >= 0x47f00000u ? 0x7f800000u : m;
  return of_bits(m | (hi & 0x80000000u));
}

// exp(-y^2) and erfc(y), which the half-space moments take together.
template <class R>
FD_HD void exp_erfc(R y, R& e, R& ec) {
  e = s_exp(-y * y);
  ec = s_erfc_e(y, e);
}

// FP64: both from one table and one Taylor expansion about the nearest x =
// k/256 (a table method as P. T. P. Tang's for exp, ACM TOMS 15, 1989).  With
// d = |y| - x, |d| <= 1/512,
//   exp(-y^2) = exp(-x^2) P(d),  P = exp(-2 x d - d^2) = sum p_n d^n,
//   erfc(|y|) = erfc(x) - 2/sqrt(pi) exp(-x^2) d sum p_n d^n/(n+1),
//   p_0 = 1, p_1 = -2x, p_2 = 2x^2 - 1, p_3 = 2x - 4x^3/3,
//   p_{n+1} = -(2 x p_n + 2 p_{n-1})/(n+1),
// the terms from n = 4 on (below 8e-10) in FP32: 23 slots of the FP64 pipe for
// the pair where the library's exp and erfcx take 60, and both within 2 ulp (no
// rounding of y^2 enters).  512^2 vortex, FP64 points 3.89 -> 3.62 ms per step.
// Beyond |y| = 3 the library's functions.
#if defined(__CUDACC__)
FDK_GAUSS_TABLE(static __device__, gauss_table_dev)
#endif
FDK_GAUSS_TABLE(static, gauss_table_host)
// FP32 to FP64 by shifts, off the FP64 pipe (exact for normal numbers; below
// 2^-126 the result is off by at most 2^-127, a zero becomes 2^-127)
FD_HD double f32_to_f64(float x) {
  const unsigned b = bits_of(x);
  return of_words((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + 0x38000000u), b << 29);
}
FD_HD void exp_erfc(double y, double& e, double& ec) {
  const double a = fabs(y);
  if (!(a < 3.0)) {
    e = s_exp(-y * y);
    ec = s_erfc_e(y, e);
    return;
  }
  const double magic = 6755399441055744.0;   // 1.5 * 2^52: adds round to an integer in the low word
  const double s = a * FDK_GAUSS_STEPS + magic;
  unsigned sh, k;
  words_of(s, sh, k);
#if defined(__CUDA_ARCH__)
  const double E = gauss_table_dev[k][0], C = gauss_table_dev[k][1];
#else
  const double E = gauss_table_host[k][0], C = gauss_table_host[k][1];
#endif
  const double x = (s - magic) * (1.0 / FDK_GAUSS_STEPS), d = a - x;
  // FP32: q = p_4 + p_5 d + p_6 d^2, r = p_4/5 + p_5 d/6
  const float xf = (float)(int)k * (1.0f / FDK_GAUSS_STEPS), df = est_f32(d), wf = xf * xf;
  const float f2 = 2.0f * wf - 1.0f, f3 = xf * (2.0f - (4.0f / 3.0f) * wf);
  const float f4 = -0.5f * (xf * f3 + f2), f5 = -0.4f * (xf * f4 + f3), f6 = (-1.0f / 3.0f) * (xf * f5 + f4);
  const double q = f32_to_f64(f4 + df * (f5 + df * f6)), r = f32_to_f64(0.2f * f4 + df * ((1.0f / 6.0f) * f5));
  const double w = x * x, p2 = 2.0 * w - 1.0, p3 = x * (2.0 - (4.0 / 3.0) * w);
  const double P = d * (-2.0 * x + d * (p2 + d * (p3 + d * q)));   // less 1
  const double Q = d + d * (d * (-x + d * (p2 * (1.0 / 3.0) + d * (0.25 * p3 + d * r))));
  e = E + E * P;
  const double c = C - (1.12837916709551257390 * E) * Q;   // 2/sqrt(pi)
  ec = y >= 0.0 ? c : 2.0 - c;
}

// value at which tanh(z) rounds to exactly 1 in FP32
template <class R> struct TanhSat;
template <> struct TanhSat<float> { static constexpr float z = 9.5f; };
// FP64: the value from which (1 - e)/(1 + e), e = e^(-2z), rounds to 1: e = 2^-54,
// z = 27 ln 2.  tanh itself rounds to 1 from 27.5 ln 2 = 19.0615 on; between the
// two chi is 1 where it is 1 - 2^-53 rounded, an ulp of a weight.
const double GENO_SAT64 = 18.715;

// ---------------------------------------------------------------------------
// constants of one run, in compute precision
// ---------------------------------------------------------------------------
template <class R>
struct GenoK {
  int linear;        // 1: chi = 1 everywhere (linear scheme)
  int r;             // exponent of GENO-IS-linear
  R eps_a, eps_w, C, tanhC, inv_tanhC;
  R d_iface[3];      // ideal weights of the interface sub-stencils (App. C1/C2 order)
  R d_node[3];       // ideal weights of the node sub-stencils (Sec. 3.2 order, central first)
};

template <class R>
struct GasK {
  R K;               // internal degrees of freedom, (4 - 2 gamma)/(gamma - 1)
  R gm1;             // gamma - 1 = 2/(K + 2)
  R c4K;             // 4/(K + 2)
  R prfix;           // 1/Pr - 1 (heat-flux correction)
  double mu, c1, c2, dt, inv_dt;
  R mu_r, c1_r, c2_r, dt_r, inv_dt_r;   // the same in the compute type
};

// dt/tau above which the time coefficients show no cancellation and the FP32
// path evaluates them in FP32 (e^{-dt/tau} < 0.02); from 1 to it they are
// computed in FP64 with expm1, up to 1 by float-float series (time_coef_small)
const double TIME_COEF_FP32_RATIO = 4.0;

template <class R> FD_HD R rpow(R x, int r) { return r == 3 ? x * x * x : x * x; }

// ---------------------------------------------------------------------------
// GENO blend (Sec. 3.2, Eqs. GENO-nonlinear, GENO-IS-linear, GENO-1d-IS-HL)
// of a high-order value/derivative with ENO-weighted sub-stencil values and
// derivatives (the same weights serve both).
// ---------------------------------------------------------------------------
template <class R> struct IsF32 { static constexpr bool v = false; };
template <> struct IsF32<float> { static constexpr bool v = true; };

// FP32 rounding floor of the smoothness indicators: the indicators are
// squares of differences of O(|Q|) values, which FP32 resolves only to about
// u |Q| (u = 2^-24); below (64 u |Q|)^2 they measure rounding, not the data.
// The FP32 path adds it to eps_a, so that data varying by less than about
// 4e-6 of their magnitude count as smooth (FP64: no floor).
template <class R>
FD_HD R geno_floor(R qmax) {
  if (IsF32<R>::v) {
    const R e = R(64.0 * 5.9604644775390625e-8) * qmax;
    return e * e;
  }
  return R(0);
}

// Sufficient test for chi = 1 (TanhSat, GENO_SAT64), which smooth data pass:
// alpha = 2 aH/(aH + aL) with aH >= 1, so C alpha > z wherever
// aL = 1 + (tau/(ISL + eps))^r < 2C/z - 1.  C = 20; the bounds on
// tau/(ISL + eps) are the r-th roots of 2C/z - 2 (0.13732 in FP64, where z =
// GENO_SAT64, 2.2105 in FP32), rounded down.  It takes a product where the quotients of the path
// function take divisions (FP32) or 14 more FP64 operations.
template <class R> struct GenoSmooth { static constexpr double c2 = 0.370560, c3 = 0.515910; };
template <> struct GenoSmooth<float> { static constexpr float c2 = 1.48670f, c3 = 1.30260f; };
template <class R>
FD_HD bool geno_smooth(R tau, R ISL, R ea, int r) {
  return tau < R(r == 3 ? GenoSmooth<R>::c3 : GenoSmooth<R>::c2) * (ISL + ea);
}

template <class R>
FD_HD R geno_chi(const GenoK<R>& g, R IS0, R IS1, R IS2, R floor = R(0)) {
  if (g.linear) return R(1);
  R ISL = s_min(IS0, s_min(IS1, IS2));
  R ISH = s_max(IS0, s_max(IS1, IS2));
  R tau = s_abs(R(0.5) * (IS1 + IS2) - IS0);
  if (geno_smooth(tau, ISL, g.eps_a + floor, g.r)) return g.inv_tanhC;
  if constexpr (IsF32<R>::v) {
    // FP32: quotient form (the product form could overflow for large IS)
    const R ea = g.eps_a + floor;
    R aH = R(1) + rpow(s_div(tau, ISH + ea), g.r);
    R aL = R(1) + rpow(s_div(tau, ISL + ea), g.r);
    const R z = g.C * s_div(R(2) * aH, aH + aL);
    // tanh(z) is exactly 1 in this precision above the saturation point
    if (z > R(TanhSat<R>::z)) return g.inv_tanhC;
    return s_tanh(z) * g.inv_tanhC;
  } else {
    // tanh(C alpha) with alpha = 2 aH/(aH + aL), aH = 1 + (tau/h)^r, aL = 1 +
    // (tau/l)^r, over the common denominator h^r l^r; tanh z as
    // (1 - e^-2z)/(1 + e^-2z), one exponential and two reciprocals (tanh(C) is
    // 1).  A floor is added to eps_a only when one is given (the FP64
    // linearisation of a mixed run)
    R ea = g.eps_a;
    if (floor != R(0)) ea = ea + floor;
    const R hr = rpow(ISH + ea, g.r), lr = rpow(ISL + ea, g.r), tr = rpow(tau, g.r);
    const R a = (hr + tr) * lr, b = (lr + tr) * hr;
    const R z = (R(2) * g.C) * (a * (R(1) / (a + b)));
    if (z > R(GENO_SAT64)) return g.inv_tanhC;
    const R e = s_exp(R(-2) * z);
    return (R(1) - e) * (R(1) / (R(1) + e));
  }
}

// Scales four numbers by 2^-512 where the last, the sum of the others, is finite and
// above 2^864 (1e260): in their exponents, which all exceed 2^-510 then, so that it
// costs no slot of the FP64 pipe and no branch.
FD_HD void scale_vast(double w[3], double& sum) {
  unsigned hi, lo;
  words_of(sum, hi, lo);
  const unsigned first = (1023u + 864u) << 20, inf = 0x7ff00000u;
  const unsigned down = hi - first < inf - first ? 512u << 20 : 0u;
  sum = of_words(hi - down, lo);
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    words_of(w[k], hi, lo);
    w[k] = of_words(hi - down, lo);
  }
}
template <class R> FD_HD void scale_vast(R[3], R&) {}   // other scalar types

// Weights of the three sub-stencils up to the factor returned (FP64: the
// reciprocal of their sum, which is applied once to what they weight; FP32:
// 1, the weights are normalised, which keeps their range).  In FP64 they reach
// the eighth power of the data's differences, and times a ninth would overflow
// from differences of 1e34 on: the largest are scaled down.
template <class R>
FD_HD R geno_weights(const GenoK<R>& g, const R d[3], R IS0, R IS1, R IS2, R w[3]) {
  R e0 = IS0 + g.eps_w, e1 = IS1 + g.eps_w, e2 = IS2 + g.eps_w;
  R s0 = e0 * e0, s1 = e1 * e1, s2 = e2 * e2;
  if (IsF32<R>::v) {
    R t0 = s_div(d[0], s0), t1 = s_div(d[1], s1), t2 = s_div(d[2], s2);
    R inv = s_div(R(1), t0 + t1 + t2);
    w[0] = t0 * inv;
    w[1] = t1 * inv;
    w[2] = t2 * inv;
    return R(1);
  }
  // d_k/s_k normalised = d_k P_k / sum_m d_m P_m with P_k the product of the other two s
  w[0] = d[0] * (s1 * s2);
  w[1] = d[1] * (s0 * s2);
  w[2] = d[2] * (s0 * s1);
  R sum = w[0] + (w[1] + w[2]);
  scale_vast(w, sum);
  return R(1) / sum;
}

// The floor of an FP64 evaluation: (fscale max|Q|)^2 when fscale is given
// (fscale = 64 u reproduces the FP32 path's floor in FP64, for the reverse
// pass of a mixed run), else none; the FP32 path always takes its own.
template <class R>
FD_HD R geno_floor_of(R qmax, R fscale) {
  if (IsF32<R>::v) return geno_floor(qmax);
  if (fscale != R(0)) {
    const R e = fscale * qmax;
    return e * e;
  }
  return R(0);
}

// FP32 estimate of the saturation test (geno_smooth) of the FP64 path: true
// only where the FP64 indicators pass it too.  The indicators are positive
// definite forms of the estimated differences (smallest eigenvalue 0.24), so
// each estimate is within 5e-5 of its indicator and tau within 1e-4 of the
// largest; both margins are on the safe side.  An infinite or NaN indicator
// fails the test.
FD_HD bool geno_smooth_est(float I0, float I1, float I2, float ea, int r) {
  const float lo = fminf(I0, fminf(I1, I2)), hi = fmaxf(I0, fmaxf(I1, I2));
  const float tau = fabsf(0.5f * (I1 + I2) - I0);
  return tau + 2e-4f * hi < (r == 3 ? 0.51585f : 0.37050f) * (0.9999f * lo + ea);
}
FD_HD float is_grad_est(float b, float xh) {   // the sub-stencil with an averaged gradient
  const float t = b - xh, u = 2.0f * b - xh;
  return (13.0f / 3.0f) * t * t + u * u;
}
FD_HD float is_three_est(float t, float u) { return (13.0f / 12.0f) * t * t + 0.25f * u * u; }

// whether the FP64 path screens its indicators in FP32 (FP64 runs at 1/64 of
// the FP32 rate, and smooth data need no FP64 indicators at all)
template <class R> struct GenoScreen { static constexpr bool v = false; };
template <> struct GenoScreen<double> { static constexpr bool v = true; };
FD_HD void screen_iface(const GenoK<double>& g, double b0, double b1, double b2, double x0, double x3, float hf,
                        bool& sl, bool& sr) {
  const float c0 = est_f32(b0), c1 = est_f32(b1), c2 = est_f32(b2);
  const float y0 = est_f32(x0) * hf, y3 = est_f32(x3) * hf, ea = (float)g.eps_a;
  const float t01 = c1 - c0, t12 = c2 - c1;
  sl = geno_smooth_est(is_grad_est(c0, y0), is_three_est(t01, c0 + c1), is_three_est(t12, c2 - 3.0f * c1), ea, g.r);
  sr = geno_smooth_est(is_grad_est(c2, y3), is_three_est(t12, c1 + c2), is_three_est(t01, c0 - 3.0f * c1), ea, g.r);
}
FD_HD bool screen_node(const GenoK<double>& g, double b0, double b1, double x0, double x2, float hf) {
  const float c0 = est_f32(b0), c1 = est_f32(b1);
  return geno_smooth_est(is_three_est(c1 - c0, c0 + c1), is_grad_est(c0, est_f32(x0) * hf),
                         is_grad_est(c1, est_f32(x2) * hf), (float)g.eps_a, g.r);
}
template <class R>
FD_HD void screen_iface(const GenoK<R>&, R, R, R, R, R, float, bool&, bool&) {}
template <class R>
FD_HD bool screen_node(const GenoK<R>&, R, R, R, R, float) { return false; }
template <class R> FD_HD float screen_h(R) { return 0.0f; }
// the spacing for the screen: infinite, which fails every test, where FP32 does not
// hold it (subnormal) or where the gradients that est_f32 flushes (below 2^-126)
// would count, h 2^-126 against the root of eps_a (3e-8): from 2^80 on, 2^-46
FD_HD float screen_h(double h) {
  const float hf = (float)h;
  return hf >= 1.17549435e-38f && hf < 1.2089258e24f ? hf : INFINITY;
}

// left and right states at the interface between Q[1] and Q[2] of a 4-point
// line, with averaged gradients Qx[0..3] of the same 4 nodes (Sec. 3.1 Eq.
// 7th-compact-recons; App. C1 and C2).  h: spacing, ih = 1/h; fscale: see
// geno_floor_of.  Everything is written in the differences b_k = Q[k+1] - Q[k]
// (values relative to the node on their side), which all formulas share: 20
// FP64 operations a component on smooth data (about 100 with every indicator
// in FP64).  512^2 vortex, ms per step: FP64 points 5.55 -> 4.25, nodal 1.24 ->
// 0.57 (without the screen 4.96 and 0.92; with conversions on the FP64 pipe
// instead of est_f32's shifts 4.34 and 0.64); mixed points 0.174 -> 0.153.
template <class R>
FD_HD void recon_interface(const GenoK<R>& g, const R Q[4], const R Qx[4], R h, R ih,
                           R& vl, R& dl, R& chil, R& vr, R& dr, R& chir, R fscale = R(0)) {
  const R c64 = R(1.0 / 64.0), c30 = R(1.0 / 30.0);
  const R b0 = Q[1] - Q[0], b1 = Q[2] - Q[1], b2 = Q[3] - Q[2];
  // shared high-order derivative (identical for left and right)
  const R PHx = (b0 + b2 + R(46) * b1) * (ih * c30) - R(0.3) * (Qx[1] + Qx[2]);
  const R PHl = R(22) * b1 + b2 - R(7) * b0 + (Qx[0] + R(22) * Qx[1] - R(7) * Qx[2]) * h;      // times 64
  const R PHr = R(7) * b2 - R(22) * b1 - b0 + (R(7) * Qx[1] - R(22) * Qx[2] - Qx[3]) * h;
  bool smooth_l = g.linear, smooth_r = g.linear;
  if (GenoScreen<R>::v && !g.linear && fscale == R(0))
    screen_iface(g, b0, b1, b2, Qx[0], Qx[3], screen_h(h), smooth_l, smooth_r);
  chil = chir = g.linear ? R(1) : g.inv_tanhC;
  vl = Q[1] + c64 * PHl;
  vr = Q[2] + c64 * PHr;
  dl = dr = PHx;
  if (smooth_l && smooth_r) return;
  const R fl = geno_floor_of(s_max(s_max(s_abs(Q[0]), s_abs(Q[1])), s_max(s_abs(Q[2]), s_abs(Q[3]))), fscale);
  const R t01 = b1 - b0, t12 = b2 - b1;
  const R s01 = R(13.0 / 12.0) * t01 * t01, s12 = R(13.0 / 12.0) * t12 * t12;
  // ---- left state (App. C1) ----
  if (!smooth_l) {
    const R xh = Qx[0] * h;
    R t = b0 - xh, u = R(2) * b0 - xh;
    const R IS0 = R(13.0 / 3.0) * t * t + u * u;
    u = b0 + b1;
    const R IS1 = s01 + R(0.25) * u * u;
    u = b2 - R(3) * b1;
    const R IS2 = s12 + R(0.25) * u * u;
    const R chi = geno_chi(g, IS0, IS1, IS2, fl);
    chil = chi;
    if (chi != R(1)) {
      R w[3];
      const R om = (R(1) - chi) * geno_weights(g, g.d_iface, IS0, IS1, IS2, w);
      const R PL = w[0] * (R(1.25) * b0 - R(0.75) * xh) + w[1] * (R(0.125) * b0 + R(0.375) * b1) +
                   w[2] * (R(0.625) * b1 - R(0.125) * b2);
      const R PLx = w[0] * (R(3) * b0 * ih - R(2) * Qx[0]) + (w[1] + w[2]) * (b1 * ih);
      vl = Q[1] + (chi * (c64 * PHl) + om * PL);
      dl = chi * PHx + om * PLx;
    }
  }
  // ---- right state (App. C2, formulas for interface j+1/2) ----
  if (!smooth_r) {
    const R xh = Qx[3] * h;
    R t = b2 - xh, u = R(2) * b2 - xh;
    const R IS0 = R(13.0 / 3.0) * t * t + u * u;
    u = b1 + b2;
    const R IS1 = s12 + R(0.25) * u * u;
    u = b0 - R(3) * b1;
    const R IS2 = s01 + R(0.25) * u * u;
    const R chi = geno_chi(g, IS0, IS1, IS2, fl);
    chir = chi;
    if (chi != R(1)) {
      R w[3];
      const R om = (R(1) - chi) * geno_weights(g, g.d_iface, IS0, IS1, IS2, w);
      const R PL = w[0] * (R(0.75) * xh - R(1.25) * b2) - w[1] * (R(0.125) * b2 + R(0.375) * b1) +
                   w[2] * (R(0.125) * b0 - R(0.625) * b1);
      const R PLx = w[0] * (R(3) * b2 * ih - R(2) * Qx[3]) + (w[1] + w[2]) * (b1 * ih);
      vr = Q[2] + (chi * (c64 * PHr) + om * PL);
      dr = chi * PHx + om * PLx;
    }
  }
}

// rho > 0 and 2 E rho > m_x^2 + m_y^2 (positive pressure), both finite: the
// test of the positivity safeguard of the interface states
template <class R>
FD_HD bool physical_state(const R W[4]) {
  return W[0] > R(0) && R(2) * W[3] * W[0] > W[1] * W[1] + W[2] * W[2] && W[0] < R(INFINITY) &&
         W[3] < R(INFINITY);
}

// derivative at the middle node of a 3-point line (Sec. 3.1 Eq.
// 6th-compact-recons; App. C3 with the Sec. 3.2 sub-stencil order)
template <class R>
FD_HD R recon_node(const GenoK<R>& g, const R Q[3], const R Qx[3], R h, R ih, R fscale = R(0)) {
  const R b0 = Q[1] - Q[0], b1 = Q[2] - Q[1], b = b0 + b1;
  const R PHx = (Qx[0] + R(46) * Qx[1] + Qx[2]) * R(1.0 / 30.0) - (R(0.3) * ih) * b;
  if (g.linear) return PHx;
  if (GenoScreen<R>::v && fscale == R(0) && screen_node(g, b0, b1, Qx[0], Qx[2], screen_h(h))) return PHx;
  const R x0 = Qx[0] * h, x2 = Qx[2] * h;
  R t = b1 - b0;
  const R IS0 = R(13.0 / 12.0) * t * t + R(0.25) * b * b;
  t = b0 - x0;
  R u = R(2) * b0 - x0;
  const R IS1 = R(13.0 / 3.0) * t * t + u * u;
  t = b1 - x2;
  u = R(2) * b1 - x2;
  const R IS2 = R(13.0 / 3.0) * t * t + u * u;
  const R chi =
      geno_chi(g, IS0, IS1, IS2, geno_floor_of(s_max(s_abs(Q[1]), s_max(s_abs(Q[0]), s_abs(Q[2]))), fscale));
  if (chi == R(1)) return PHx;
  R w[3];
  const R om = (R(1) - chi) * geno_weights(g, g.d_node, IS0, IS1, IS2, w);
  const R PLx = w[0] * (R(0.5) * b * ih) + w[1] * (R(2) * b0 * ih - Qx[0]) + w[2] * (R(2) * b1 * ih - Qx[2]);
  return chi * PHx + om * PLx;
}

// ---------------------------------------------------------------------------
// heat flux of the energy equation relative to (U0, V0) from the moments
// F = int u psi f and W = int psi f of one distribution (x-normal)
template <class R>
FD_HD R heat_flux_x(const R F[4], const R W[4], R U0, R V0) {
  return F[3] - U0 * W[3] - U0 * F[1] - V0 * F[2] + (R(1.5) * U0 * U0 + R(0.5) * V0 * V0) * W[1] +
         U0 * V0 * W[2] - R(0.5) * U0 * (U0 * U0 + V0 * V0) * W[0];
}
// ---------------------------------------------------------------------------
// Time coefficients of the interface distribution, integrated over
// [0, delta] for delta = dt/2 and dt and fitted to f^n + t f_t^n (App. A1).
// The terms cancel where dt/tau is small: TW is FP64 there, unless the series
// of time_coef_small replace this form.
// ---------------------------------------------------------------------------
template <class TW>
struct TimeCoef {
  TW cn[6], ct[6];
  TW E, e1;   // exp(-dt/tau), 1 - exp(-dt/tau)
};

// integrals over [0, d] of the equilibrium coefficients c1..c3 of f(0,t);
// the initial-data coefficients follow from c1 + c4 = 1, c2 + c5 = -tau,
// c3 + c6 = t - tau
template <class TW>
FD_HD void time_integrals_d(TW tau, TW d, TW E, TW e1, TW C[3]) {
  C[0] = d - tau * e1;
  C[1] = -tau * d * (TW(1) + E) + TW(2) * tau * tau * e1;
  C[2] = TW(0.5) * d * d - tau * d + tau * tau * e1;
}

template <class TW>
FD_HD TimeCoef<TW> time_coef(TW tau, TW dt, TW inv_dt) {
  TimeCoef<TW> t;
  // one transcendental: em = exp(-dt/(2 tau)) - 1, then
  // exp(-dt/tau) - 1 = em (em + 2) without cancellation.  Beyond
  // dt/(2 tau) = 40 expm1 rounds to -1 in FP64 (from 37.5 on) and FP32; smooth
  // inviscid flow lies there and is spared the division, expm1 and 25 products
  if (TW(0.5) * dt > TW(40) * tau) {
    // em = -1: the fits in closed form, with r = tau/dt
    const TW r = tau * inv_dt, tr = tau * r, r4 = TW(4) * r * r;
    t.E = TW(0);
    t.e1 = TW(1);
    t.cn[3] = TW(3) * r;
    t.cn[4] = TW(-6) * tr;
    t.cn[5] = TW(-3) * tr;
    t.ct[0] = TW(4) * r * inv_dt;
    t.ct[4] = TW(2) * r4;
    t.ct[5] = r4;
    t.cn[0] = TW(1) - t.cn[3];
    t.cn[1] = -tau - t.cn[4];
    t.cn[2] = -tau - t.cn[5];
    t.ct[1] = -t.ct[4];
    t.ct[2] = TW(1) - r4;
    t.ct[3] = -t.ct[0];
    return t;
  }
  const TW em = s_expm1(-TW(0.5) * dt / tau);
  TW Eh = TW(1) + em, e1h = -em;
  t.E = Eh * Eh;
  t.e1 = -em * (em + TW(2));
  TW Ch[3], Cf[3];
  time_integrals_d(tau, TW(0.5) * dt, Eh, e1h, Ch);
  time_integrals_d(tau, dt, t.E, t.e1, Cf);
  for (int k = 0; k < 3; ++k) {
    // linear-in-time fit of App. A1: f^n = (4 fbar(dt/2) - fbar(dt))/dt,
    // f_t^n = 4 (fbar(dt) - 2 fbar(dt/2))/dt^2
    t.cn[k] = (TW(4) * Ch[k] - Cf[k]) * inv_dt;
    t.ct[k] = TW(4) * (Cf[k] - TW(2) * Ch[k]) * inv_dt * inv_dt;
  }
  // fits of c4..c6: the fit of (c1 + c4) = 1 is 1 (value) and 0 (slope),
  // of (c2 + c5) = -tau is -tau and 0, of (c3 + c6) = t - tau is -tau and 1
  t.cn[3] = TW(1) - t.cn[0];
  t.ct[3] = -t.ct[0];
  t.cn[4] = -tau - t.cn[1];
  t.ct[4] = -t.ct[1];
  t.cn[5] = -tau - t.cn[2];
  t.ct[5] = TW(1) - t.ct[2];
  return t;
}

// Float-float numbers h + l (|l| a few ulp of h at most, so that l l' counts for
// nothing): sums and products of some 44 bits from FP32 operations (Dekker 1971,
// Knuth's TwoSum).  add_rn and mul_rn are rounded by themselves, never fused.
FD_HD float add_rn(float a, float b) {
#if defined(__CUDA_ARCH__)
  return __fadd_rn(a, b);
#else
  volatile float r = a + b;
  return r;
#endif
}
FD_HD float mul_rn(float a, float b) {
#if defined(__CUDA_ARCH__)
  return __fmul_rn(a, b);
#else
  volatile float r = a * b;
  return r;
#endif
}
FD_HD float s_fma(float a, float b, float c) { return fmaf(a, b, c); }
template <class R> FD_HD R add_rn(R a, R b) { return a + b; }   // other scalar types
template <class R> FD_HD R mul_rn(R a, R b) { return a * b; }
template <class R> FD_HD R s_fma(R a, R b, R c) { return a * b + c; }

template <class R>
struct FF {
  R h, l;
};
template <class R> FD_HD FF<R> ff_neg(FF<R> a) { return {-a.h, -a.l}; }
template <class R> FD_HD FF<R> ff_scale(FF<R> a, R k) { return {a.h * k, a.l * k}; }   // k a power of two
template <class R> FD_HD R ff_round(FF<R> a) { return add_rn(a.h, a.l); }
template <class R>
FD_HD FF<R> ff_quick(R a, R b) {   // a + b exactly, |a| >= |b|
  const R s = add_rn(a, b);
  return {s, add_rn(b, -add_rn(s, -a))};
}
template <class R>
FD_HD FF<R> ff_sum(R a, R b) {     // a + b exactly
  const R s = add_rn(a, b), v = add_rn(s, -a);
  return {s, add_rn(add_rn(a, -add_rn(s, -v)), add_rn(b, -v))};
}
template <class R>
FD_HD FF<R> ff_add(FF<R> a, FF<R> b) {   // |a| >= |b|
  const FF<R> s = ff_quick(a.h, b.h);
  return {s.h, add_rn(s.l, add_rn(a.l, b.l))};
}
template <class R>
FD_HD FF<R> ff_mul(FF<R> a, FF<R> b) {
  const R p = mul_rn(a.h, b.h);
  return {p, s_fma(a.h, b.l, s_fma(a.l, b.h, s_fma(a.h, b.h, -p)))};
}
template <class R>
FD_HD FF<R> ff_div(FF<R> a, FF<R> b) {
  const R i = s_div(R(1), b.h), q = mul_rn(a.h, i);
  return {q, mul_rn(add_rn(s_fma(-q, b.h, a.h), s_fma(-q, b.l, a.l)), i)};
}
template <class R> FD_HD FF<R> ff_one_less(FF<R> a) { return ff_add(FF<R>{R(1), R(0)}, ff_neg(a)); }
// an FP64 value to 46 bits or more: one slot of the FP64 pipe
template <class R> FD_HD FF<R> ff_split(double v) { return {R(v), R(0)}; }
template <>
FD_HD FF<float> ff_split<float>(double v) {
  const float h = est_f32(v);
  return {h, est_f32(v - f32_to_f64(h))};
}

// The same for q = tau/dt >= 1, for the FP32 path without FP64's pipe: inserting
// exp(-y) = sum (-y)^n/n! in the integrals, with x = 1/q, every term that
// cancels drops out and two power series in x remain,
//   p = sum_{n>=3} (-1)^n (4/2^n - 1)/n! x^(n-3),
//   r = -sum_{n>=3} (-1)^n 4 (1 - 2/2^n)/n! x^(n-3),
// from which, with w = 1 - x r and m = w/4 - 2 p,
//   cn0 = x^2 p,  cn1 = dt x m,  cn2 = -dt x p,
//   ct0 = x w/dt,  ct1 = 2 (x r - x^2 p) - 3/2 x w,  ct2 = x r,
//   1 - E = x (1 - x^2 p - x w/2).
// The series' terms to n = 8 are summed by a compensated Horner rule (Graillat,
// Langlois and Louvet 2005), those to n = 16 (below 2^-14 of the sum, the next
// below 2^-42) in FP32 in front of it, and the rest is float-float, so that a
// coefficient is its exact value rounded once: the error is at most 0.500 ulp
// of FP32, which the FP64 form reaches for x > 1e-2 (0.54 at 1e-3, 13 at 1e-4:
// its terms cancel to third order), where four plain FP32 series were 4 to 9 ulp
// off.  Viscous tube 1000x500, ms per step: 0.47 with those series, 0.51 so, 1.07
// with the FP64 form.
template <class R>
FD_HD TimeCoef<R> time_coef_small(FF<R> q, FF<R> dt, FF<R> inv_dt) {
  const int FIRST = 3, SPLIT = 8, LAST = 16;
  const FF<R> x = ff_div(FF<R>{R(1), R(0)}, q);
  R ps = R(0), rs = R(0), pe = R(0), re = R(0);   // the sums and their errors
  auto step = [&](R& s, R& e, double c) {
    const R ch = R((float)c), cl = R((float)(c - (double)(float)c)), t = mul_rn(s, x.h);
    const FF<R> u = ff_quick(ch, t);
    e = s_fma(e, x.h, s_fma(s, x.l, add_rn(s_fma(s, x.h, -t), add_rn(u.l, cl))));
    s = u.h;
  };
#pragma unroll
  for (int n = LAST; n >= FIRST; --n) {
    double f = 1.0, h = 1.0;   // n!, 2^-n
    for (int k = 1; k <= n; ++k) { f *= k; h *= 0.5; }
    const double sg = n % 2 ? -1.0 : 1.0, a = sg * (4.0 * h - 1.0) / f, b = -sg * 4.0 * (1.0 - 2.0 * h) / f;
    if (n > SPLIT) {
      ps = s_fma(ps, x.h, R(a));
      rs = s_fma(rs, x.h, R(b));
    } else {
      step(ps, pe, a);
      step(rs, re, b);
    }
  }
  const FF<R> p = {ps, pe}, r = {rs, re};
  const FF<R> xp = ff_mul(x, p), xr = ff_mul(x, r), xxp = ff_mul(x, xp), w = ff_one_less(xr), xw = ff_mul(x, w);
  const FF<R> xm = ff_mul(x, ff_add(ff_scale(w, R(0.25)), ff_scale(p, R(-2))));
  TimeCoef<R> t;
  t.cn[0] = ff_round(xxp);
  t.cn[1] = ff_round(ff_mul(dt, xm));
  t.cn[2] = -ff_round(ff_mul(dt, xp));
  t.ct[0] = ff_round(ff_mul(inv_dt, xw));
  t.ct[1] = -ff_round(ff_add(ff_add(xw, ff_scale(xw, R(0.5))), ff_scale(ff_add(xr, ff_neg(xxp)), R(-2))));
  t.ct[2] = ff_round(xr);
  t.cn[3] = ff_round(ff_one_less(xxp));
  t.ct[3] = -t.ct[0];
  t.cn[4] = -ff_round(ff_mul(dt, ff_add(q, xm)));
  t.ct[4] = -t.ct[1];
  t.cn[5] = -ff_round(ff_mul(dt, ff_add(q, ff_neg(xp))));
  t.ct[5] = ff_round(w);
  const FF<R> e1 = ff_mul(x, ff_one_less(ff_add(ff_scale(xw, R(0.5)), xxp)));
  t.e1 = ff_round(e1);
  t.E = ff_round(ff_one_less(e1));
  return t;
}
// the same for FP32 arguments (x = dt/tau, implied by the others), for tests
template <class R>
FD_HD TimeCoef<R> time_coef_small(R x, R tau, R dt, R inv_dt) {
  (void)x;
  const FF<R> d = {dt, R(0)};
  (void)inv_dt;
  return time_coef_small(ff_div(FF<R>{tau, R(0)}, d), d, ff_div(FF<R>{R(1), R(0)}, d));
}

// ---------------------------------------------------------------------------
// Closed-form moments.  A slope a = (d ln g) of a Maxwellian is fixed by the
// gradients of its primitive variables; with c = v - V the tangential
// peculiar velocity and s0..s3 the coefficients of 1, u, c, (u^2 + c^2 + xi^2)/2,
//   s3 = theta'/theta^2, s2 = V'/theta, s1 = U'/theta - U s3,
//   s0 = rho'/rho - (K+2)/2 theta'/theta - U s1 - U^2 s3 / 2,   theta = p/rho,
// which needs no moment system.  In the variable c odd moments vanish and
// <c^2 + xi^2> = N theta, <(c^2 + xi^2)^2> = N (N+2) theta^2 with N = K + 1,
// so a slope-weighted moment is a polynomial in u alone.  Whole-space moments
// (the equilibrium state g0 and the compatibility conditions) are then the
// Euler flux, its time derivative and the Navier-Stokes stress and heat flux.
// D1: the one-dimensional gas, V = 0 and no y-derivatives; component 2 is
// neither read nor written.
// ---------------------------------------------------------------------------

// conservative W with its primitive variables; th = p/rho, en = rho E/rho
template <class R>
struct GasState {
  R rho, ir, U, V, p, th, en;
};
template <bool D1 = false, class R>
FD_HD GasState<R> gas_state(const R W[4], R gm1) {
  GasState<R> g;
  g.rho = W[0];
  g.ir = s_div(R(1), W[0]);
  g.U = W[1] * g.ir;
  g.V = D1 ? R(0) : W[2] * g.ir;
  g.en = W[3] * g.ir;
  if (IsF32<R>::v) {   // squares of one factor: every kernel contracts them alike, so their results agree
    g.th = gm1 * (g.en - R(0.5) * (D1 ? g.U * g.U : g.U * g.U + g.V * g.V));
    g.p = g.rho * g.th;
  } else {
    g.p = gm1 * (W[3] - R(0.5) * (D1 ? W[1] * g.U : W[1] * g.U + W[2] * g.V));
    g.th = g.p * g.ir;
  }
  return g;
}

// rho times a derivative of the primitive variables: d = rho', u = rho U',
// v = rho V', t = rho theta'.  Everything they enter is linear in them and
// wanted per unit volume, so the weight saves the products with 1/rho here and
// with rho there (some 40 of a solve's 900 FP64 operations).
template <class R>
struct PrimGrad {
  R d, u, v, t;
};
// from the derivative D of the conservative variables
template <bool D1 = false, class R>
FD_HD PrimGrad<R> prim_grad(const GasState<R>& g, R gm1, const R D[4]) {
  PrimGrad<R> q;
  q.d = D[0];
  q.u = D[1] - g.U * D[0];
  if (D1) {
    q.v = R(0);
    q.t = gm1 * (D[3] - g.en * D[0] - g.U * q.u);
  } else {
    q.v = D[2] - g.V * D[0];
    q.t = gm1 * (D[3] - g.en * D[0] - g.U * q.u - g.V * q.v);
  }
  return q;
}
// time derivative from the x- and y-derivatives (compatibility
// <(a u + b v + A) psi> = 0: the Euler equations)
template <bool D1 = false, class R>
FD_HD PrimGrad<R> prim_rate(const GasState<R>& g, R gm1, const PrimGrad<R>& x, const PrimGrad<R>& y) {
  PrimGrad<R> q;
  if (D1) {
    q.d = -(g.U * x.d + x.u);
    q.u = -(g.U * x.u + g.th * x.d + x.t);
    q.v = R(0);
    q.t = -(g.U * x.t + gm1 * g.th * x.u);
    return q;
  }
  const R div = x.u + y.v;
  q.d = -(g.U * x.d + g.V * y.d + div);
  q.u = -(g.U * x.u + g.V * y.u + g.th * x.d + x.t);
  q.v = -(g.U * x.v + g.V * y.v + g.th * y.d + y.t);
  q.t = -(g.U * x.t + g.V * y.t + gm1 * g.th * div);
  return q;
}
// derivative of the conservative variables; hN = (K + 2)/2
template <bool D1 = false, class R>
FD_HD void cons_rate(const GasState<R>& g, R hN, const PrimGrad<R>& q, R W[4]) {
  W[0] = q.d;
  W[1] = g.U * q.d + q.u;
  if (D1) {
    W[3] = g.en * q.d + g.U * q.u + hN * q.t;
    return;
  }
  W[2] = g.V * q.d + q.v;
  W[3] = g.en * q.d + g.U * q.u + g.V * q.v + hN * q.t;
}
// Euler x-flux of g and its derivative for the derivative q (Wq: of W)
template <bool D1 = false, class R>
FD_HD void euler_flux(const GasState<R>& g, const R W[4], R F[4]) {
  F[0] = W[1];
  F[1] = g.U * W[1] + g.p;
  if (!D1) F[2] = g.V * W[1];
  F[3] = g.U * (W[3] + g.p);
}
template <bool D1 = false, class R>
FD_HD void euler_flux_rate(const GasState<R>& g, const PrimGrad<R>& q, const R Wq[4], R F[4]) {
  const R pq = g.th * q.d + q.t;
  F[0] = Wq[1];
  F[1] = g.U * (Wq[1] + q.u) + pq;
  if (!D1) F[2] = g.V * Wq[1] + g.U * q.v;
  F[3] = q.u * (g.en + g.th) + g.U * (Wq[3] + pq);
}
// rho <u psi (a u + b v + A)>: minus the Navier-Stokes stress and heat flux
// over the collision time (the density component is 0)
template <bool D1 = false, class R>
FD_HD void stress_flux(const GasState<R>& g, R K, R gm1, const PrimGrad<R>& x, const PrimGrad<R>& y, R S[4]) {
  S[0] = R(0);
  if (D1) {
    S[1] = g.th * ((R(2) - gm1) * x.u);
    S[3] = g.U * S[1] + (R(0.5) * K + R(2)) * (g.th * x.t);
    return;
  }
  S[1] = g.th * (R(2) * x.u - gm1 * (x.u + y.v));
  S[2] = g.th * (x.v + y.u);
  S[3] = g.U * S[1] + g.V * S[2] + (R(0.5) * K + R(2)) * (g.th * x.t);
}

// ---------------------------------------------------------------------------
// One side of the interface: the half-space moments M[n] = <u^n> over u > 0
// (sign +1) or u < 0 (sign -1), and the slope polynomials D = a u + b v and A
// integrated over c and xi against 1, c and (c^2 + xi^2)/2, both times rho.
// With weights k3 + k4 D + k5 A the moments are, for T_k = <s u^k>,
//   T_k = e0 M_k + e1 M_{k+1} + e2 M_{k+2} + e3 M_{k+3},
//   <s u^k c> = c0 M_k + c1 M_{k+1} + c2 M_{k+2},
//   <s u^k (u^2 + c^2 + xi^2)/2> = T_{k+2}/2 + N theta/2 T_k + X0 M_k + X1 M_{k+1}.
// ---------------------------------------------------------------------------
template <class R>
struct HalfSide {
  R M[7];
  R rho, V, Nh;                              // Nh = N theta/2
  R e0, e1, e2, e3, X0, X1, c0, c1, c2;      // D
  R Ae0, Ae1, Ae2, AX0, Ac0;                 // A
};

template <class R>
FD_HD void half_moments(const GasState<R>& g, int sign, R sl, R M[7]) {
  const R x = sl * g.U;                        // U sqrt(lambda)
  R e, ec;
  exp_erfc(sign > 0 ? -x : x, e, ec);
  const R isqpi2 = R(0.56418958354775628695);   // 1/sqrt(pi); sl th = 1/(2 sqrt(lambda))
  M[0] = R(0.5) * ec;
  M[1] = g.U * M[0] + R(sign) * isqpi2 * (e * (sl * g.th));
  R nth = g.th;
#pragma unroll
  for (int n = 0; n < 5; ++n) {
    M[n + 2] = g.U * M[n + 1] + nth * M[n];
    if (n < 4) nth = nth + g.th;
  }
}

template <bool D1 = false, class R>
FD_HD void half_side(const GasState<R>& g, R N, R ith, const PrimGrad<R>& gx, const PrimGrad<R>& gy,
                     const PrimGrad<R>& gt, HalfSide<R>& s) {
  s.rho = g.rho;
  s.V = g.V;
  s.Nh = R(0.5) * N * g.th;
  const R cU = R(0.5) * g.U * g.U;
  // slope coefficients; the constant one with N theta s3 / 2 added (its
  // integral over c and xi)
  const R ta = gx.t * ith, a3 = ta * ith, a1 = gx.u * ith - g.U * a3;
  const R a0 = gx.d - R(0.5) * ta - g.U * a1 - cU * a3;
  s.e3 = R(0.5) * a3;
  s.X1 = s.Nh * ta;
  if (D1) {
    s.e1 = a0;
    s.e2 = a1;
  } else {
    const R tb = gy.t * ith, b3 = tb * ith, b1 = gy.u * ith - g.U * b3;
    const R b0 = gy.d - R(0.5) * tb - g.U * b1 - cU * b3;
    s.e0 = g.V * b0 + gy.v;
    s.e1 = a0 + g.V * b1;
    s.e2 = a1 + R(0.5) * g.V * b3;
    s.X0 = g.V * (s.Nh * tb) + g.th * gy.v;
    s.c0 = g.V * gy.v + g.th * (b0 + tb);
    s.c1 = gx.v + g.th * b1;
    s.c2 = R(0.5) * tb;
  }
  const R tA = gt.t * ith, A3 = tA * ith;
  s.Ae1 = gt.u * ith - g.U * A3;
  s.Ae0 = gt.d - R(0.5) * tA - g.U * s.Ae1 - cU * A3;
  s.Ae2 = R(0.5) * A3;
  s.AX0 = s.Nh * tA;
  if (!D1) s.Ac0 = gt.v;
}

// adds rho <psi s> to Wm and rho <u psi s> to F for s = k3 + k4 D + k5 A
template <bool D1 = false, class R>
FD_HD void half_flux(const HalfSide<R>& s, R k3, R k4, R k5, R F[4], R Wm[4]) {
  const R q3 = s.rho * k3, q4 = k4, q5 = k5;
  const R e0 = D1 ? q3 + q5 * s.Ae0 : q3 + q4 * s.e0 + q5 * s.Ae0, e1 = q4 * s.e1 + q5 * s.Ae1, e2 = q4 * s.e2 + q5 * s.Ae2;
  const R e3 = q4 * s.e3;
  const R X0 = D1 ? q5 * s.AX0 : q4 * s.X0 + q5 * s.AX0, X1 = q4 * s.X1;
  const R* M = s.M;
  R T[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) T[k] = e0 * M[k] + (e1 * M[k + 1] + (e2 * M[k + 2] + e3 * M[k + 3]));
  const R E0 = R(0.5) * T[2] + s.Nh * T[0] + X0 * M[0] + X1 * M[1];
  const R E1 = R(0.5) * T[3] + s.Nh * T[1] + X0 * M[1] + X1 * M[2];
  Wm[0] += T[0];
  Wm[1] += T[1];
  F[0] += T[1];
  F[1] += T[2];
  if (D1) {
    Wm[3] += E0;
    F[3] += E1;
    return;
  }
  const R c0 = q4 * s.c0 + q5 * s.Ac0, c1 = q4 * s.c1, c2 = q4 * s.c2;
  const R C0 = c0 * M[0] + c1 * M[1] + c2 * M[2], C1 = c0 * M[1] + c1 * M[2] + c2 * M[3];
  const R hV = R(0.5) * s.V;
  Wm[2] += C0 + s.V * T[0];
  Wm[3] += E0 + s.V * (C0 + hV * T[0]);
  F[2] += C1 + s.V * T[1];
  F[3] += E1 + s.V * (C1 + hV * T[1]);
}

// ---------------------------------------------------------------------------
// Interface solve with x as the normal (App. A1-A2, Eq. eq:W-model).
// Inputs: left/right reconstructed states, their normal (x) derivatives and
// the shared tangential (y) derivative.  want_n = false skips the outputs
// that the second S2O4 stage does not use (F^, W^ values).
//
// The distribution is g0 (k0 + k1 (a0 u + b0 v) + k2 A0) on the whole space
// plus g (k3 + k4 (a u + b v) + k5 A) on each half, k = cn for the value and
// ct for the time slope; each set's polynomial is formed first, so a side's
// moments are taken once per set instead of once per basis term: 855 flops
// instead of the 1667 of moment tables and moment-system solves, and 114
// instead of 402 for the nodal flux below (GB300, vortex 512^2, ms per step,
// this form alone: FP64 points 7.80 -> 5.55, nodal 1.63 -> 1.24; mixed points
// 0.223 -> 0.174, nodal 0.062 -> 0.051; with rho-weighted gradients FP64 points
// 3.41 -> 3.15).  The FP64 kernels are bound by the FP64 pipe, which
// takes 16 clocks of an SM per warp instruction whatever the occupancy, the
// FP32 ones by instruction issue: fewer operations is what both need.
// ---------------------------------------------------------------------------
template <class R>
struct IfaceOut {
  R F[4], Ft[4], Wl[4], Wr[4], Wlt[4], Wrt[4];
};

// the power of two below a density, and its inverse
FD_HD void density_unit(float rho, float& unit, float& inv) {
  unsigned e = bits_of(rho) >> 23 & 255u;
  e = e < 1u ? 1u : e > 253u ? 253u : e;
  unit = of_bits(e << 23);
  inv = of_bits((254u - e) << 23);
}
template <class R> FD_HD void density_unit(R, R& unit, R& inv) { unit = inv = R(1); }   // other scalar types

template <bool D1 = false, class R>
FD_HD void iface_solve_x(const GasK<R>& gas, const R Wl_[4], const R Wr_[4], const R Wln_[4], const R Wrn_[4],
                         const R Wt_[4], bool want_n, IfaceOut<R>& o) {
  // The slopes carry the density (PrimGrad): in FP32 their products with theta^-2
  // leave the range for densities far from 1 where the specific ones would not.
  // The solve is linear in the density's unit, so there the unit is the power of
  // two below the left density (exact).  Elsewhere a test and branches not taken,
  // us per step: 33^2 22.6 -> 22.9, 1024^2 876 -> 878, an ensemble of 40 925 -> 935.
  R unit = R(1), Wl[4], Wr[4], Wln[4], Wrn[4], Wt[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) { Wl[k] = Wl_[k]; Wr[k] = Wr_[k]; Wln[k] = Wln_[k]; Wrn[k] = Wrn_[k]; Wt[k] = Wt_[k]; }
  if (IsF32<R>::v && !(Wl_[0] > R(1e-9) && Wl_[0] < R(1e9))) {
    R inv;
    density_unit(Wl_[0], unit, inv);
#pragma unroll
    for (int k = 0; k < 4; ++k) { Wl[k] *= inv; Wr[k] *= inv; Wln[k] *= inv; Wrn[k] *= inv; Wt[k] *= inv; }
  }
  const R K = gas.K, gm1 = gas.gm1, N = K + R(1), hN = R(0.5) * K + R(1);
  const GasState<R> gl = gas_state<D1>(Wl, gm1), gr = gas_state<D1>(Wr, gm1);
  HalfSide<R> sl, sr;
  const R ql = s_rsqrt(R(2) * gl.th), qr = s_rsqrt(R(2) * gr.th);   // sqrt(lambda)
  half_moments(gl, +1, ql, sl.M);
  half_moments(gr, -1, qr, sr.M);

  // equilibrium state from the particles crossing the interface
  R W0[4];
  {
    const R ml = gl.rho * sl.M[0], mr = gr.rho * sr.M[0];
    W0[0] = ml + mr;
    W0[1] = gl.rho * sl.M[1] + gr.rho * sr.M[1];
    if (D1) {
      W0[2] = R(0);
      W0[3] = R(0.5) * (gl.rho * sl.M[2] + gr.rho * sr.M[2] + N * (gl.p * sl.M[0] + gr.p * sr.M[0]));
    } else {
      W0[2] = gl.V * ml + gr.V * mr;
      W0[3] = R(0.5) * (gl.rho * sl.M[2] + gr.rho * sr.M[2] + (ml * (gl.V * gl.V) + mr * (gr.V * gr.V)) +
                        N * (gl.p * sl.M[0] + gr.p * sr.M[0]));
    }
  }
  const GasState<R> g0 = gas_state<D1>(W0, gm1);

  // gradients (x: normal, y: tangential) and time derivatives of each state
  R x1[4], W0q[4];
  PrimGrad<R> gtl, gtr;
  {
    const PrimGrad<R> gx = prim_grad<D1>(gl, gm1, Wln), gy = prim_grad<D1>(gl, gm1, Wt);
    gtl = prim_rate<D1>(gl, gm1, gx, gy);
    half_side<D1>(gl, N, R(2) * ql * ql, gx, gy, gtl, sl);
  }
  {
    const PrimGrad<R> gx = prim_grad<D1>(gr, gm1, Wrn), gy = prim_grad<D1>(gr, gm1, Wt);
    gtr = prim_rate<D1>(gr, gm1, gx, gy);
    half_side<D1>(gr, N, R(2) * qr * qr, gx, gy, gtr, sr);
  }
  R FE[4], FQ[4], FS[4];   // g0: Euler flux, its time derivative, stress
  {
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (!D1 || k != 2) x1[k] = R(0.5) * (Wln[k] + Wrn[k]);
    const PrimGrad<R> gx = prim_grad<D1>(g0, gm1, x1), gy = prim_grad<D1>(g0, gm1, Wt), gt = prim_rate<D1>(g0, gm1, gx, gy);
    cons_rate<D1>(g0, hN, gt, W0q);
    euler_flux<D1>(g0, W0, FE);
    euler_flux_rate<D1>(g0, gt, W0q, FQ);
    stress_flux<D1>(g0, K, gm1, gx, gy, FS);
  }

  // collision time and time coefficients: FP64 with expm1 where they cancel
  // (dt/tau small); in the FP32 path FP32 where dt/tau > 4, where they do not,
  // and where dt/tau <= 1 float-float, as exact as FP64's when rounded to FP32
  // (viscous runs lie there: the FP64 form's 85 slots of the FP64 pipe cost
  // more than the rest of the FP32 solve)
  typedef typename Wide<R>::T TW;
  R cn[6], ct[6], E, e1;
  R ip0r = R(0);                               // 1/p0, needed with viscosity only
  if (gas.mu_r != R(0)) ip0r = s_div(R(1), g0.p);
  if (IsF32<R>::v && unit != R(1)) ip0r = s_div(ip0r, unit);
  R taur = gas.c1_r * gas.dt_r + gas.mu_r * ip0r + gas.c2_r * gas.dt_r * s_div(s_abs(gl.p - gr.p), gl.p + gr.p);
  if (IsF32<R>::v && gas.dt_r > R(TIME_COEF_FP32_RATIO) * taur) {
    TimeCoef<R> tc = time_coef(taur, gas.dt_r, gas.inv_dt_r);
#pragma unroll
    for (int k = 0; k < 6; ++k) { cn[k] = tc.cn[k]; ct[k] = tc.ct[k]; }
    E = tc.E;
    e1 = tc.e1;
  } else if (IsF32<R>::v && !(gas.dt_r > taur)) {
    // tau/dt = c1 + c2 |pl - pr|/(pl + pr) + (mu/dt)/p0
    FF<R> dp = ff_sum(gl.p, -gr.p);
    if (dp.h < R(0)) dp = ff_neg(dp);
    const FF<R> qj = ff_mul(ff_split<R>(gas.c2), ff_div(dp, ff_sum(gl.p, gr.p))), q1 = ff_split<R>(gas.c1);
    FF<R> q = ff_sum(q1.h, qj.h);
    q.l = q.l + (q1.l + qj.l);
    if (gas.mu_r != R(0)) {
      const FF<R> qm = ff_mul(ff_split<R>(gas.mu * gas.inv_dt), FF<R>{ip0r, R(0)}), s = ff_sum(q.h, qm.h);
      q = {s.h, s.l + (q.l + qm.l)};
    }
    TimeCoef<R> tc = time_coef_small(q, ff_split<R>(gas.dt), ff_split<R>(gas.inv_dt));
#pragma unroll
    for (int k = 0; k < 6; ++k) { cn[k] = tc.cn[k]; ct[k] = tc.ct[k]; }
    E = tc.E;
    e1 = tc.e1;
  } else {
    TW pl = to_w(gl.p), pr = to_w(gr.p);
    TW ip0 = to_w(ip0r);
    TW dtw = TW(gas.dt);
    TW tau = TW(gas.c1) * dtw + TW(gas.mu) * ip0 + TW(gas.c2) * dtw * (s_abs(pl - pr) * (TW(1) / (pl + pr)));
    TimeCoef<TW> tc = time_coef(tau, dtw, TW(gas.inv_dt));
#pragma unroll
    for (int k = 0; k < 6; ++k) { cn[k] = from_w<R>(tc.cn[k]); ct[k] = from_w<R>(tc.ct[k]); }
    E = from_w<R>(tc.E);
    e1 = from_w<R>(tc.e1);
  }

  // <psi (a0 u + b0 v)> = -W0q and <psi A0> = W0q (compatibility); the fluxes
  // of the two terms are FS - FQ and FQ
  R F[4], We[4];
  auto used = [](int k) { return !D1 || k != 2; };
  if (D1) F[2] = We[2] = R(0);
  if (want_n) {
    const R kq = cn[2] - cn[1];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (!used(k)) continue;
      F[k] = cn[0] * FE[k] + kq * FQ[k] + cn[1] * FS[k];
      We[k] = cn[0] * W0[k] + kq * W0q[k];
    }
    half_flux<D1>(sr, cn[3], cn[4], cn[5], F, We);
    half_flux<D1>(sl, cn[3], cn[4], cn[5], F, We);
    // Prandtl-number correction of the energy flux
    if (gas.prfix != R(0)) F[3] += gas.prfix * heat_flux_x(F, We, g0.U, g0.V);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (!used(k)) continue;
      // interface flow variables, Eq. (eq:W-model) with tau_0 = tau
      o.F[k] = F[k];
      o.Wl[k] = o.Wr[k] = We[k];
    }
    if (E != R(0)) {
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        if (!used(k)) continue;
        o.Wl[k] = e1 * We[k] + E * Wl[k];
        o.Wr[k] = e1 * We[k] + E * Wr[k];
      }
    }
  }
  const R kq = ct[2] - ct[1];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    if (!used(k)) continue;
    F[k] = ct[0] * FE[k] + kq * FQ[k] + ct[1] * FS[k];
    We[k] = ct[0] * W0[k] + kq * W0q[k];
  }
  half_flux<D1>(sl, ct[3], ct[4], ct[5], F, We);
  half_flux<D1>(sr, ct[3], ct[4], ct[5], F, We);
  if (gas.prfix != R(0)) F[3] += gas.prfix * heat_flux_x(F, We, g0.U, g0.V);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    if (!used(k)) continue;
    o.Ft[k] = F[k];
    o.Wlt[k] = o.Wrt[k] = We[k];
  }
  // the initial states' part, with the one-sided time derivatives W_t = -rho
  // <(a u + b v) psi>: nothing is left of it (E = 0, e1 = 1) where dt/tau > 80,
  // as in smooth inviscid flow (512^2 vortex, points per step: FP64 3.62 ->
  // 3.41 ms, mixed 0.140 -> 0.137)
  if (E != R(0)) {
    R Wlq[4], Wrq[4];
    cons_rate<D1>(gl, hN, gtl, Wlq);
    cons_rate<D1>(gr, hN, gtr, Wrq);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (!used(k)) continue;
      o.Wlt[k] = e1 * We[k] + E * Wlq[k];
      o.Wrt[k] = e1 * We[k] + E * Wrq[k];
    }
  }
  if (IsF32<R>::v && unit != R(1)) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (!used(k)) continue;
      o.Ft[k] *= unit;
      o.Wlt[k] *= unit;
      o.Wrt[k] *= unit;
      if (want_n) { o.F[k] *= unit; o.Wl[k] *= unit; o.Wr[k] *= unit; }
    }
  }
}

// y-normal solve through the x <-> y transposition of the equations; the
// transposition is a register select, so one copy of the x-normal solve
// serves both normals
template <class R>
FD_HD void swap_uv(const R a[4], R b[4], bool sw) {
  b[0] = a[0];
  b[1] = sw ? a[2] : a[1];
  b[2] = sw ? a[1] : a[2];
  b[3] = a[3];
}

template <class R>
FD_HD void iface_solve(const GasK<R>& gas, int normal, const R Wl[4], const R Wr[4], const R Wln[4],
                       const R Wrn[4], const R Wt[4], bool want_n, IfaceOut<R>& o) {
  const bool sw = normal != 0;
  R a[4], b[4], c[4], d[4], e[4];
  swap_uv(Wl, a, sw); swap_uv(Wr, b, sw); swap_uv(Wln, c, sw); swap_uv(Wrn, d, sw); swap_uv(Wt, e, sw);
  IfaceOut<R> t;
  iface_solve_x(gas, a, b, c, d, e, want_n, t);
  swap_uv(t.Ft, o.Ft, sw); swap_uv(t.Wlt, o.Wlt, sw); swap_uv(t.Wrt, o.Wrt, sw);
  if (want_n) { swap_uv(t.F, o.F, sw); swap_uv(t.Wl, o.Wl, sw); swap_uv(t.Wr, o.Wr, sw); }
}

// ---------------------------------------------------------------------------
// Nodal flux from smooth local data (Sec. 2.1): f = g(1 - tau(a u + b v + A)),
// f_t = A g.  Outputs x-flux F, y-flux G and their time derivatives;
// want_n = false computes the time derivatives only (F, G are set to 0): the
// second S2O4 stage uses no other nodal output.
// ---------------------------------------------------------------------------
template <class R>
FD_HD void nodal_flux(const GasK<R>& gas, const R W[4], const R Wx[4], const R Wy[4], R F[4], R G[4], R Ft[4],
                      R Gt[4], bool want_n = true) {
  const R K = gas.K, gm1 = gas.gm1;
  const GasState<R> g = gas_state(W, gm1);
  const PrimGrad<R> gx = prim_grad(g, gm1, Wx), gy = prim_grad(g, gm1, Wy), gt = prim_rate(g, gm1, gx, gy);
  R Wq[4];
  cons_rate(g, R(0.5) * K + R(1), gt, Wq);
  // f_t = A g: the time derivative of the Euler fluxes; its heat flux relative
  // to the fixed (U, V) is (K + 4)/2 p (U_t, V_t).  y-flux by the
  // transposition u <-> v
  const R qf = gas.prfix * (R(0.5) * K + R(2)) * g.th;
  euler_flux_rate(g, gt, Wq, Ft);
  Ft[3] += qf * gt.u;
  const GasState<R> s = {g.rho, g.ir, g.V, g.U, g.p, g.th, g.en};
  const PrimGrad<R> sx = {gx.d, gx.v, gx.u, gx.t}, sy = {gy.d, gy.v, gy.u, gy.t}, st = {gt.d, gt.v, gt.u, gt.t};
  const R Ws[4] = {W[0], W[2], W[1], W[3]}, Wsq[4] = {Wq[0], Wq[2], Wq[1], Wq[3]};
  R x[4], y[4];
  euler_flux_rate(s, st, Wsq, x);
  Gt[0] = x[0]; Gt[1] = x[2]; Gt[2] = x[1]; Gt[3] = x[3] + qf * gt.v;
  if (!want_n) {
#pragma unroll
    for (int k = 0; k < 4; ++k) F[k] = G[k] = R(0);
    return;
  }
  // F = Euler - tau stress, the heat flux (K + 4)/2 p theta' over Pr
  R tau = gas.c1_r * gas.dt_r;                                       // c1 dt + mu/p
  if (gas.mu_r != R(0)) tau = tau + gas.mu_r * s_div(R(1), g.p);
  euler_flux(g, W, F);
  stress_flux(g, K, gm1, gx, gy, x);
  x[3] += qf * gx.t;
#pragma unroll
  for (int k = 1; k < 4; ++k) F[k] = F[k] - tau * x[k];
  euler_flux(s, Ws, x);
  stress_flux(s, K, gm1, sy, sx, y);
  y[3] += qf * gy.t;
#pragma unroll
  for (int k = 1; k < 4; ++k) x[k] = x[k] - tau * y[k];
  G[0] = x[0]; G[1] = x[2]; G[2] = x[1]; G[3] = x[3];
}

// The x-flux of nodal_flux for the one-dimensional gas (V = 0, no
// y-derivative); component 2 is neither read nor written.
template <class R>
FD_HD void nodal_flux_1d(const GasK<R>& gas, const R W[4], const R Wx[4], R F[4], R Ft[4], bool want_n) {
  const R K = gas.K, gm1 = gas.gm1;
  const GasState<R> g = gas_state<true>(W, gm1);
  const PrimGrad<R> gx = prim_grad<true>(g, gm1, Wx), gt = prim_rate<true>(g, gm1, gx, gx);
  R Wq[4], x[4];
  cons_rate<true>(g, R(0.5) * K + R(1), gt, Wq);
  const R qf = gas.prfix * (R(0.5) * K + R(2)) * g.th;
  euler_flux_rate<true>(g, gt, Wq, Ft);
  Ft[3] += qf * gt.u;
  if (!want_n) return;
  R tau = gas.c1_r * gas.dt_r;                                       // c1 dt + mu/p
  if (gas.mu_r != R(0)) tau = tau + gas.mu_r * s_div(R(1), g.p);
  euler_flux<true>(g, W, F);
  stress_flux<true>(g, K, gm1, gx, gx, x);
  x[3] += qf * gx.t;
  F[1] = F[1] - tau * x[1];
  F[3] = F[3] - tau * x[3];
}

// ---------------------------------------------------------------------------
// Compact numerical flux (Eqs. fd-conservative-flux, -flux-1, -flux-2).
// Fi = {F_{j-1/2}, F_{j+1/2}, F_{j+3/2}}, Fn0 = F_j, Fn1 = F_{j+1}
// ---------------------------------------------------------------------------
template <class R>
FD_HD R compact_flux(int variant, R chi, R Fim, R Fi0, R Fip, R Fn0, R Fn1) {
  R Fbar = (Fim + R(46) * Fi0 + Fip - R(9) * (Fn0 + Fn1)) * R(1.0 / 30.0);
  R Flow = variant == 62 ? Fi0 : (R(8) * Fi0 - Fn0 - Fn1) * R(1.0 / 6.0);
  return (R(1) - chi) * Flow + chi * Fbar;
}

// Difference of the compact fluxes at j+1/2 and j-1/2 over the node j.
// Fi = {F_{j-3/2}, F_{j-1/2}, F_{j+1/2}, F_{j+3/2}}, Fn = {F_{j-1}, F_j, F_{j+1}}.
// SMOOTH: both interfaces take the high-order flux (chi = 1), whose difference
// is (F_{j+3/2} - F_{j-3/2} + 45 (F_{j+1/2} - F_{j-1/2}) - 9 (F_{j+1} - F_{j-1}))/30,
// 6 operations instead of the two blended fluxes' 22.
template <bool SMOOTH, class R>
FD_HD R compact_flux_diff(int variant, R chim, R chip, R Fmm, R Fm, R Fp, R Fpp, R Nm, R N0, R Np) {
  if (SMOOTH) return (R(45) * (Fp - Fm) + (Fpp - Fmm) - R(9) * (Np - Nm)) * R(1.0 / 30.0);
  return compact_flux(variant, chip, Fm, Fp, Fpp, N0, Np) - compact_flux(variant, chim, Fmm, Fm, Fp, Nm, N0);
}

}  // namespace fdk
