// The FP64 Dormand-Prince 5(4) integrator of Hamilton's equations (Eq.
// Hamilton) shared by the forward, backward and adjoint kernels: the lane
// state of one ray, the step-size controller, and one step attempt with the
// null-cone branch switching, the step-reach bound and the escape event.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "rt_device.cuh"
#include "rt_internal.h"

namespace rtk {
namespace {

constexpr unsigned FULL = 0xffffffffu;

__device__ __forceinline__ void rhs64(const RayConst<double>& c, const double* y, double* f) {
  ham_rhs64<double>(c, y[0], y[1], y[2], y[3], y[4], y[5], f[0], f[1], f[2], f[3], f[4], f[5]);
}

// FP32 <-> FP64 by integer operations.  The conversion instructions issue on
// the FP64 pipe at its rate (64 cycles a warp); these cost it nothing.
// narrow(): toward zero; below 2^-126 zero, above FP32's range infinity, NaN
// stays NaN.  widen(): exact for zero and normal values; infinity and NaN stay
// what they are (a subnormal float becomes zero).
__device__ __forceinline__ float narrow(double d) {
  const int hi = __double2hiint(d), a = hi & 0x7fffffff;
  int f = __funnelshift_l(__double2loint(d), a - 0x38000000, 3);
  if (a < 0x38100000) f = 0;
  if (a >= 0x47f00000) f = (a > 0x7ff00000 || (a == 0x7ff00000 && __double2loint(d))) ? 0x7fc00000
                                                                                      : 0x7f800000;
  return __int_as_float(f | (hi & 0x80000000));
}
__device__ __forceinline__ double widen(float v) {
  const int b = __float_as_int(v), a = b & 0x7fffffff;
  int hi = (a >> 3) + 0x38000000;
  if (a < 0x00800000) hi = 0;
  if (a >= 0x7f800000) hi = 0x7ff00000 | (a > 0x7f800000 ? 0x80000 : 0);
  return __hiloint2double(hi | (b & 0x80000000),
                          (a < 0x00800000 || a >= 0x7f800000) ? 0 : (a << 29));
}
// the larger magnitude, compared as integers (a comparison of doubles is an
// FP64-pipe instruction)
__device__ __forceinline__ double max_abs(double a, double b) {
  const long long x = __double_as_longlong(a) & 0x7fffffffffffffffll;
  const long long y = __double_as_longlong(b) & 0x7fffffffffffffffll;
  return __longlong_as_double(x > y ? x : y);
}
// Reciprocal, quotient and inverse square root to rounding, for arguments in FP32's
// range (in_fp32: 2^-100 <= x < 2^100) from the FP32 unit's estimate at the leading 21
// bits and one step of Chebyshev's iteration of order three in FP64 (Traub, Iterative
// Methods for the Solution of Equations, 1964: t - f/f' - f^2 f''/(2 f'^3)), for all
// others by CUDA's functions (a tolerance may be as small as the smallest double).  A division takes ten FP64
// instructions of 64 cycles and rsqrt() has a longer path around its special values; an
// attempt has six quotients, a group's attempt twelve inverse roots: 4096 rays of the
// aligned star 371 ms, 382 ms with CUDA's functions throughout; 16 x 251 rays of the
// rotating one 540 and 562 ms.  CUDA's functions stand in copies of their own: inlined
// at every use they cost the double-float kernel, which waits for instructions, 2 %.
__device__ __forceinline__ bool in_fp32(double x) {
  return (unsigned)(__double2hiint(x) - 0x39b00000) < 0x0c800000u;
}
static __device__ __noinline__ double quotient_any(double a, double b) { return a / b; }
static __device__ __noinline__ double rsqrt_any(double x) { return rsqrt(x); }
__device__ __forceinline__ float lead_in_fp32(double x) {
  return __int_as_float((unsigned)__double2hiint(x) * 8u + 0x40000000u);
}
__device__ __forceinline__ double widen_normal(float v) {
  const int b = __float_as_int(v);
  return __hiloint2double((b >> 3) + 0x38000000, b << 29);
}
// f = 1/r - x: r (1 + d + d^2) with d = 1 - x r; the estimate is off by at most 2^-23 and
// its argument by 2^-20, so |d| < 2^-19 and the rest, d^3, is below 2^-57.
__device__ __forceinline__ double recip_in_fp32(double x) {
  float v;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(v) : "f"(lead_in_fp32(x)));
  const double r = widen_normal(v);
  const double d = fma(-x, r, 1.0);
  return fma(r, fma(d, d, d), r);
}
__device__ __forceinline__ double recip(double x) {
  return in_fp32(x) ? recip_in_fp32(x) : quotient_any(1.0, x);
}
__device__ __forceinline__ double quotient(double a, double b) {
  return in_fp32(b) ? a * recip_in_fp32(b) : quotient_any(a, b);
}
// The squared error norm's sum: (err(i) / sc_i)^2 over the six components, sc = atol +
// rtol max(|y|, |yn|), with one test of the range for all six quotients.
template <class Err>
__device__ __forceinline__ double error_sum(double atol, double rtol, const double* y,
                                            const double* yn, const Err& err) {
  double sc[6], s = 0.0;
  bool plain = true;
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    sc[i] = atol + rtol * max_abs(y[i], yn[i]);
    plain = plain && in_fp32(sc[i]);
  }
  if (plain) {
#pragma unroll
    for (int i = 0; i < 6; ++i) {
      const double q = err(i) * recip_in_fp32(sc[i]);
      s += q * q;
    }
  } else {
#pragma unroll
    for (int i = 0; i < 6; ++i) {
      const double q = quotient_any(err(i), sc[i]);
      s += q * q;
    }
  }
  return s;
}
// f = 1/y^2 - x: y (1 + e/2 + 3 e^2/8) with e = 1 - x y^2; the estimate is off by at most
// 2^-22 and its argument by 2^-20, so |e| < 2^-19 and the rest, 5 e^3/16, is below 2^-58.
__device__ __forceinline__ double inv_sqrt(double x) {
  if (!in_fp32(x)) return rsqrt_any(x);
  float v;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(v) : "f"(lead_in_fp32(x)));
  const double y = widen_normal(v);
  const double e = fma(-x, y * y, 1.0);
  return fma(y * e, fma(0.375, e, 0.5), y);
}

// The controller's factor 0.9 err^(-1/5), clamped to [0.2, 5] (no growth after a
// rejection), from the squared error norm q: err^(-1/5) = q^(-1/10), a
// single-precision estimate y corrected by the series of (1 - r)^(-1/10) in the
// residual r = 1 - q y^10 (at most ~1e-5), y (1 + r/10 + 11 r^2/200).  The clamp
// is decided on the high words (positive numbers order like their bits).
__device__ __forceinline__ double step_factor_sq(double q, bool accepted, bool last_rej) {
  const int hq = __double2hiint(q);
  double fac = 5.0;
  if (hq >= 0x426d1a94) {                         // q > 1e12
    fac = 0.2;
  } else if (hq >= 0x3d719799) {                  // q > 1e-12
    const double y = widen(exp2f(-0.1f * log2f(narrow(q))));
    const double y2 = y * y, y4 = y2 * y2;
    const double r = fma(-q, (y4 * y) * (y4 * y), 1.0);
    fac = 0.9 * fma(y, r * fma(0.055, r, 0.1), y);
    const int hf = __double2hiint(fac);
    if (hf >= 0x40140000) fac = 5.0;
    if (__double_as_longlong(fac) < __double_as_longlong(0.2)) fac = 0.2;
  }
  if ((!accepted || last_rej) && __double2hiint(fac) >= 0x3ff00000) fac = 1.0;
  return fac;
}

// Hairer's two-evaluation initial step (order 5).
__device__ double initial_step(const RayConst<double>& c, const double* y0, const double* f0,
                               double rtol, double atol, double hmax) {
  double dnf = 0.0, dny = 0.0;
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    const double sk = atol + rtol * fabs(y0[i]);
    dnf += (f0[i] / sk) * (f0[i] / sk);
    dny += (y0[i] / sk) * (y0[i] / sk);
  }
  double h = (dnf <= 1e-10 || dny <= 1e-10) ? 1e-6 : sqrt(dny / dnf) * 0.01;
  h = fmin(h, hmax);
  double y1[6], f1[6];
#pragma unroll
  for (int i = 0; i < 6; ++i) y1[i] = y0[i] + h * f0[i];
  rhs64(c, y1, f1);
  double der2 = 0.0;
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    const double sk = atol + rtol * fabs(y0[i]);
    der2 += ((f1[i] - f0[i]) / sk) * ((f1[i] - f0[i]) / sk);
  }
  der2 = sqrt(der2) / h;
  const double der12 = fmax(fabs(der2), sqrt(dnf));
  const double h1 = (der12 <= 1e-15) ? fmax(1e-6, h * 1e-3) : pow(0.01 / der12, 0.2);
  return fmin(fmin(100.0 * h, h1), hmax);
}

struct Lane {
  RayConst<double> c;
  double y[6], f0[6];
  double h, lam;
  int na, nr;
  bool last_rej;
  bool switching;      // the current attempt ends just past a null-cone crossing
  double h_resume;     // step size to resume with after that crossing
  double R_km, ma_eV;
};

// The Goldreich-Julian density |2 Omega . B / e| has a kink on the null cone
// Omega . B = 0 (Eq. GJDensity): dk/dlambda jumps there, which an embedded
// error estimate cannot resolve inside a step.  Each step integrates the
// smooth continuation of the side it starts on (c.sig); when an accepted step
// ends on the other side, the crossing is located on the continuous extension,
// the step is redone to end just past it, and the side is switched there.
constexpr double SWITCH_MIN_FRACTION = 1e-6;
constexpr double SWITCH_OVERSHOOT = 1e-10;

// Squared angular distance of ray i's start point from the Goldreich-Julian
// null cone F = 3 n_z (m.n) - m_z = 0, (F / |grad_n F|)^2 (the gradient on
// the unit sphere); 1e300 for the other plasmas.  Rays guided along the cone for
// thousands of steps start within 1e-2 rad of it.
__device__ __forceinline__ double cone_dist2(const StarDev& s, const double* state, int64_t n,
                                             int64_t i) {
  if (s.plasma != PLASMA_GJ) return 1e300;
  const double x0 = state[i], x1 = state[n + i], x2 = state[2 * n + i];
  double sp, cpsi;
  sincos(state[7 * n + i], &sp, &cpsi);
  const double m0 = s.sin_tm * cpsi, m1 = s.sin_tm * sp, m2 = s.cos_tm;
  const double ir = rsqrt(x0 * x0 + x1 * x1 + x2 * x2);
  const double n0 = x0 * ir, n1 = x1 * ir, n2 = x2 * ir;
  const double mu = m0 * n0 + m1 * n1 + m2 * n2;
  const double F = 3.0 * n2 * mu - m2;
  // grad_n F = 3 (mu e_z + n_z m) minus its radial part 6 mu n_z n
  const double c = 6.0 * mu * n2;
  const double g0 = 3.0 * n2 * m0 - c * n0, g1 = 3.0 * n2 * m1 - c * n1,
               g2 = 3.0 * (mu + n2 * m2) - c * n2;
  return (F * F) / (g0 * g0 + g1 * g1 + g2 * g2);
}

// Cost-ordered claims and finished rays.  A ray finished in one pass has had
// its state overwritten, and the cost bucket of its new state may match a
// later pass.  Stores therefore write the state, fence, then the status
// (status_after_state), and a claim that read the state for the bucket
// re-reads the status after a fence (status_still): a claim that saw any of
// the new state sees the ray finished.
__device__ __forceinline__ void status_after_state(const TraceParams& p, int64_t i, int st) {
  __threadfence();
  p.status[i] = (uint8_t)st;
}
__device__ __forceinline__ bool status_still(const TraceParams& p, int64_t i, int want) {
  __threadfence();
  return *(volatile const uint8_t*)(p.status + i) == want;
}

// Cost bucket for the cost-ordered claim (TraceParams::order): 0 for a start
// within 1e-3 rad of the null cone, 1 within 1e-2 rad, 2 otherwise.
__device__ __forceinline__ int cost_bucket(const StarDev& s, const double* state, int64_t n,
                                           int64_t i) {
  const double d2 = cone_dist2(s, state, n, i);
  return (d2 < 1e-6) ? 0 : (d2 < 1e-4) ? 1 : 2;
}

// Observer of accepted steps (forward tracing needs none).
struct NoHook {
  __device__ __forceinline__ void on_accept(const Lane&, const double*, const double*,
                                            const double*, const double*, const double*,
                                            const double*, const double*, const double*,
                                            const double*, double) {}
};

// The last th in [0, 1] on the non-negative side of side_val, given
// side_val(0) = flo >= 0 > fhi = side_val(1): Illinois (regula falsi that
// halves the retained end's value), with a bisection step whenever the
// bracket did not halve over two steps, run to the last representable th.
// Returns lo (side_val >= 0); *hi_out the first th past it.
// T is the type of th and of the values (double, or float in the mixed
// kernel); [lo, hi] the starting bracket.
template <class S, class T>
__device__ __forceinline__ T last_nonneg(const S& side_val, T flo, T fhi, T* hi_out, T lo = T(0),
                                         T hi = T(1)) {
  int last = 0;
  T width = hi - lo;
  for (int it = 0; it < 200; ++it) {
    T mid = (lo * fhi - hi * flo) / (fhi - flo);
    if ((it & 1) && hi - lo > T(0.5) * width) mid = T(0.5) * (lo + hi);
    if (!(mid > lo && mid < hi)) mid = T(0.5) * (lo + hi);
    if (mid <= lo || mid >= hi) break;
    if (it & 1) width = hi - lo;
    const T fm = side_val(mid);
    if (fm >= T(0)) {
      lo = mid;
      flo = fm;
      if (last > 0) fhi *= T(0.5);
      last = 1;
    } else {
      hi = mid;
      fhi = fm;
      if (last < 0) flo *= T(0.5);
      last = -1;
    }
  }
  *hi_out = hi;
  return lo;
}

// Plain Illinois on the bracket [lo, hi] (side(lo) = flo >= 0 > fhi =
// side(hi)), updated in place, until it is at most tol x hi wide, stops
// shrinking, or maxit evaluations were spent.  Superlinear for a simple root;
// no bisection steps (the caller finishes with last_nonneg if needed).
template <class S, class T>
__device__ __forceinline__ void illinois(const S& side, T& lo, T& hi, T& flo, T& fhi, T tol,
                                         int maxit) {
  int last = 0;
  for (int it = 0; it < maxit && hi - lo > tol * hi; ++it) {
    T mid = (lo * fhi - hi * flo) / (fhi - flo);
    if (!(mid > lo && mid < hi)) mid = T(0.5) * (lo + hi);
    if (mid <= lo || mid >= hi) break;
    const T fm = side(mid);
    if (fm >= T(0)) {
      lo = mid;
      flo = fm;
      if (last > 0) fhi *= T(0.5);
      last = 1;
    } else {
      hi = mid;
      fhi = fm;
      if (last < 0) flo *= T(0.5);
      last = -1;
    }
  }
}

// Event location on the continuous extension: the root th in [0, 1] of a
// function given in FP64 (f64) and, to FP32 rounding, by a cheap FP32 model
// (f32), with f64(0) = flo >= 0 > fhi = f64(1).  The FP32 model's root (plain
// Illinois to 2^-22 relative) is widened by SEED_WIDEN on each side; where FP64
// values at the two ends confirm it, the secant through them is off by
// ~SEED_WIDEN^2 times the relative curvature, and one more secant step from an
// FP64 value there leaves only rounding.  Otherwise (a grazing crossing, or
// rounding of the model) last_nonneg from [0, 1].
//
// On this GPU a search runs at one or two live lanes of its warp while every
// FP64 instruction costs the same 64 cycles: three FP64 evaluations and two
// divisions, against fifteen or more evaluations, each with a division, of the
// guarded Illinois from [0, 1].  The FP32 part costs the FP64 pipe nothing (the
// model is built with narrow()).
constexpr float SEED_TOL32 = 0x1p-22f;
constexpr float SEED_WIDEN = 0x1p-19f;
template <class S64, class S32>
__device__ __forceinline__ double event_root(const S64& f64, const S32& f32, double flo,
                                             double fhi) {
  float l = 0.0f, u = 1.0f, fl = narrow(flo), fu = narrow(fhi);
  if (!(fl >= 0.0f)) fl = 0.0f;
  if (!(fu < 0.0f)) fu = -1e-30f;
  illinois(f32, l, u, fl, fu, SEED_TOL32, 40);
  const double a = widen(fmaxf(0.0f, l - SEED_WIDEN)), b = widen(fminf(1.0f, u + SEED_WIDEN));
  const double fa = f64(a), fb = f64(b);
  if (fa >= 0.0 && fb < 0.0) {
    const double slope = (b - a) * recip(fa - fb);      // -1 / f'
    double th = fma(fa, slope, a);
    th = fma(f64(th), slope, th);
    if (th >= a && th <= b) return th;
  }
  double hi;
  return last_nonneg(f64, flo, fhi, &hi);
}

__device__ __forceinline__ float to_f32(float v) { return v; }
__device__ __forceinline__ float to_f32(double v) { return narrow(v); }

// FP32 model of the null-cone side function sig F(x(th)), F = 3 z (m.x) -
// m_z |x|^2, along the continuous extension x(th) = y + d(th), d(th) =
// th (r2 + (1 - th) (r3 + th (r4 + (1 - th) r5))): F(y + d) = F0 + gF.d +
// 3 d_z (m.d) - m_z |d|^2 with F0 = F(y) from FP64 and gF = grad F(y).
struct ConeModel32 {
  float sg, F0, m0, m1, m2, gF[3], r2[3], r3[3], r4[3], r5[3];
  // y, R2..R5: the first three (position) components
  template <class Y, class T>
  __device__ __forceinline__ void init(float sig, float F0f, float cm0, float cm1, float cm2,
                                       const Y* y, const T* R2, const T* R3, const T* R4,
                                       const T* R5) {
    sg = sig;
    F0 = F0f;
    m0 = cm0;
    m1 = cm1;
    m2 = cm2;
    const float y0 = to_f32(y[0]), y1 = to_f32(y[1]), y2 = to_f32(y[2]);
    const float mx = m0 * y0 + m1 * y1 + m2 * y2;
    gF[0] = 3.0f * y2 * m0 - 2.0f * m2 * y0;
    gF[1] = 3.0f * y2 * m1 - 2.0f * m2 * y1;
    gF[2] = 3.0f * mx + 3.0f * y2 * m2 - 2.0f * m2 * y2;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      r2[i] = to_f32(R2[i]);
      r3[i] = to_f32(R3[i]);
      r4[i] = to_f32(R4[i]);
      r5[i] = to_f32(R5[i]);
    }
  }
  __device__ __forceinline__ float operator()(float th) const {
    float d[3];
#pragma unroll
    for (int i = 0; i < 3; ++i)
      d[i] = th * (r2[i] + (1.0f - th) * (r3[i] + th * (r4[i] + (1.0f - th) * r5[i])));
    const float md = m0 * d[0] + m1 * d[1] + m2 * d[2];
    const float dd = d[0] * d[0] + d[1] * d[1] + d[2] * d[2];
    return sg * (F0 + (gF[0] * d[0] + gF[1] * d[1] + gF[2] * d[2]) + (3.0f * d[2] * md - m2 * dd));
  }
};

// FP32 model of r_out^2 - |x(th)|^2 on the same extension: c0 - 2 y.d - |d|^2,
// c0 = r_out^2 - |y|^2 from FP64.
struct EscapeModel32 {
  float c0, y[3], r2[3], r3[3], r4[3], r5[3];
  template <class Y, class T>
  __device__ __forceinline__ void init(float c0f, const Y* yd, const T* R2, const T* R3,
                                       const T* R4, const T* R5) {
    c0 = c0f;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      y[i] = to_f32(yd[i]);
      r2[i] = to_f32(R2[i]);
      r3[i] = to_f32(R3[i]);
      r4[i] = to_f32(R4[i]);
      r5[i] = to_f32(R5[i]);
    }
  }
  __device__ __forceinline__ float operator()(float th) const {
    float d[3];
#pragma unroll
    for (int i = 0; i < 3; ++i)
      d[i] = th * (r2[i] + (1.0f - th) * (r3[i] + th * (r4[i] + (1.0f - th) * r5[i])));
    return c0 - (2.0f * (y[0] * d[0] + y[1] * d[1] + y[2] * d[2]) +
                 (d[0] * d[0] + d[1] * d[1] + d[2] * d[2]));
  }
};

// One attempted Dormand-Prince step.  Returns -1 to continue, else the final
// ray status.  hook.on_accept sees every accepted step (start, end, stages).
template <class Hook>
__device__ int advance(const TraceParams& p, Lane& L, Hook& hook) {
  if (L.na >= p.max_steps || L.na + L.nr >= 4 * p.max_steps) return RAY_MAXSTEPS;
  bool clipped = false;
  double h = L.h;
  {
    // displacement of one step at most STEP_REACH x the distance to the centre
    const double v2 = L.f0[0] * L.f0[0] + L.f0[1] * L.f0[1] + L.f0[2] * L.f0[2];
    const double r2 = L.y[0] * L.y[0] + L.y[1] * L.y[1] + L.y[2] * L.y[2];
    if (h * h * v2 > STEP_REACH * STEP_REACH * r2) h = STEP_REACH * sqrt(r2 / v2);
  }
  if (p.lambda_max > 0.0 && L.lam + h >= p.lambda_max) {
    h = p.lambda_max - L.lam;
    clipped = true;
  }
  const double* y = L.y;
  const double* k1 = L.f0;
  double t[6], k2[6], k3[6], k4[6], k5[6], k6[6], k7[6], yn[6];
#pragma unroll
  for (int i = 0; i < 6; ++i) t[i] = y[i] + h * (DP::a21 * k1[i]);
  rhs64(L.c, t, k2);
#pragma unroll
  for (int i = 0; i < 6; ++i) t[i] = y[i] + h * (DP::a31 * k1[i] + DP::a32 * k2[i]);
  rhs64(L.c, t, k3);
#pragma unroll
  for (int i = 0; i < 6; ++i)
    t[i] = y[i] + h * (DP::a41 * k1[i] + DP::a42 * k2[i] + DP::a43 * k3[i]);
  rhs64(L.c, t, k4);
#pragma unroll
  for (int i = 0; i < 6; ++i)
    t[i] = y[i] + h * (DP::a51 * k1[i] + DP::a52 * k2[i] + DP::a53 * k3[i] + DP::a54 * k4[i]);
  rhs64(L.c, t, k5);
#pragma unroll
  for (int i = 0; i < 6; ++i)
    t[i] = y[i] + h * (DP::a61 * k1[i] + DP::a62 * k2[i] + DP::a63 * k3[i] + DP::a64 * k4[i] +
                       DP::a65 * k5[i]);
  rhs64(L.c, t, k6);
#pragma unroll
  for (int i = 0; i < 6; ++i)
    yn[i] = y[i] + h * (DP::b1 * k1[i] + DP::b3 * k3[i] + DP::b4 * k4[i] + DP::b5 * k5[i] +
                        DP::b6 * k6[i]);
  rhs64(L.c, yn, k7);
  const double s = error_sum(p.atol, p.rtol, y, yn, [&](int i) {
    return h * (DP::e1 * k1[i] + DP::e3 * k3[i] + DP::e4 * k4[i] + DP::e5 * k5[i] +
                DP::e6 * k6[i] + DP::e7 * k7[i]);
  });
  // the squared error norm; <= 1 accepts
  const double en2 = s * (1.0 / 6.0);
  if ((__double2hiint(en2) & 0x7ff00000) == 0x7ff00000) {   // infinite or NaN
    ++L.nr;
    L.h = h * 0.2;
    L.last_rej = true;
    return (L.h < 1e-12) ? RAY_NAN : -1;
  }
  const bool ok = en2 <= 1.0;
  const bool gj = (L.c.plasma == PLASMA_GJ);
  if (ok && gj && !L.switching &&
      L.c.sig * gj_side<double>(L.c.m0, L.c.m1, L.c.m2, yn[0], yn[1], yn[2]) < 0.0) {
    // the step crossed the null cone: the crossing on the continuous extension,
    // then redo the step to end just past it
    double r3[3], r4[3], r5[3], r2[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      r2[i] = yn[i] - y[i];
      r3[i] = h * k1[i] - r2[i];
      r4[i] = r2[i] - h * k7[i] - r3[i];
      r5[i] = h * (DP::d1 * k1[i] + DP::d3 * k3[i] + DP::d4 * k4[i] + DP::d5 * k5[i] +
                   DP::d6 * k6[i] + DP::d7 * k7[i]);
    }
    // s(th) = sig (3 z (m.x) - m_z |x|^2), whose sign is the side
    const double sgn = L.c.sig;
    auto side_val = [&](double th) {
      double xd[3];
#pragma unroll
      for (int i = 0; i < 3; ++i)
        xd[i] = y[i] + th * (r2[i] + (1.0 - th) * (r3[i] + th * (r4[i] + (1.0 - th) * r5[i])));
      const double mx = L.c.m0 * xd[0] + L.c.m1 * xd[1] + L.c.m2 * xd[2];
      const double rr = xd[0] * xd[0] + xd[1] * xd[1] + xd[2] * xd[2];
      return sgn * (3.0 * xd[2] * mx - L.c.m2 * rr);
    };
    double flo = side_val(0.0), fhi = side_val(1.0);
    ConeModel32 m32;
    m32.init(narrow(sgn), narrow(sgn * flo), narrow(L.c.m0), narrow(L.c.m1), narrow(L.c.m2), y, r2,
             r3, r4, r5);
    if (!(flo >= 0.0)) flo = 0.0;                  // the start is on its own side
    if (!(fhi < 0.0)) fhi = -1e-300;
    const double lo = event_root(side_val, m32, flo, fhi);
    ++L.nr;
    if (lo < SWITCH_MIN_FRACTION) {
      L.c.sig = -L.c.sig;             // already at the cone: switch here
      rhs64(L.c, L.y, L.f0);
      L.h = h;
    } else {
      L.h_resume = h;
      L.h = h * lo * (1.0 + SWITCH_OVERSHOOT);
      L.switching = true;
    }
    return -1;
  }
  if (ok) {
    ++L.na;
    hook.on_accept(L, y, yn, k1, k2, k3, k4, k5, k6, k7, h);
    const double rnew2 = yn[0] * yn[0] + yn[1] * yn[1] + yn[2] * yn[2];
    if (rnew2 >= p.r_out * p.r_out) {
      // locate |x(th)| = r_out on the continuous extension
      double r3[6], r4[6], r5[6];
#pragma unroll
      for (int i = 0; i < 6; ++i) {
        const double r2 = yn[i] - y[i];
        r3[i] = h * k1[i] - r2;
        r4[i] = r2 - h * k7[i] - r3[i];
        r5[i] = h * (DP::d1 * k1[i] + DP::d3 * k3[i] + DP::d4 * k4[i] + DP::d5 * k5[i] +
                     DP::d6 * k6[i] + DP::d7 * k7[i]);
        t[i] = r2;
      }
      // r_out^2 - |x(th)|^2 changes sign on [0, 1]
      const double ro2 = p.r_out * p.r_out;
      auto inside = [&](double th) {
        double xd[3];
#pragma unroll
        for (int i = 0; i < 3; ++i)
          xd[i] = y[i] + th * (t[i] + (1.0 - th) * (r3[i] + th * (r4[i] + (1.0 - th) * r5[i])));
        return ro2 - (xd[0] * xd[0] + xd[1] * xd[1] + xd[2] * xd[2]);
      };
      double flo = ro2 - (y[0] * y[0] + y[1] * y[1] + y[2] * y[2]);
      if (!(flo >= 0.0)) flo = 0.0;
      double fhi = ro2 - rnew2;
      if (!(fhi < 0.0)) fhi = -1e-300;
      EscapeModel32 e32;
      e32.init(narrow(flo), y, t, r3, r4, r5);
      const double th = event_root(inside, e32, flo, fhi);
#pragma unroll
      for (int i = 0; i < 6; ++i)
        yn[i] = y[i] + th * (t[i] + (1.0 - th) * (r3[i] + th * (r4[i] + (1.0 - th) * r5[i])));
#pragma unroll
      for (int i = 0; i < 6; ++i) L.y[i] = yn[i];
      L.lam += th * h;
      return RAY_ESCAPED;
    }
#pragma unroll
    for (int i = 0; i < 6; ++i) {
      L.y[i] = yn[i];
      L.f0[i] = k7[i];
    }
    L.lam += h;
    if (rnew2 <= p.r_capture * p.r_capture) return RAY_CAPTURED;
    if (clipped) return RAY_LAMBDA_END;
    if (gj && L.c.sig * gj_side<double>(L.c.m0, L.c.m1, L.c.m2, L.y[0], L.y[1], L.y[2]) < 0.0) {
      L.c.sig = -L.c.sig;             // past the cone: continue on the other side
      rhs64(L.c, L.y, L.f0);
    }
    if (L.switching) {
      L.h = L.h_resume;
      L.switching = false;
    } else {
      L.h = h * step_factor_sq(en2, true, L.last_rej);
    }
    L.last_rej = false;
    return -1;
  }
  ++L.nr;
  L.h = h * step_factor_sq(en2, false, L.last_rej);
  L.last_rej = true;
  return (L.h < 1e-12) ? RAY_STIFF : -1;
}

}  // namespace
}  // namespace rtk
