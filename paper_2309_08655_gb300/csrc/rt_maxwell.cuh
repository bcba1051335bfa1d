// Inverse distribution of the Maxwellian speed (Sec. 4.3, Eq. GaussianDist).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "rt_device.cuh"

namespace rtk {
namespace sampling {

constexpr double TWO_OVER_SQRTPI = 1.12837916709551257390;

// Inverse CDF of the Maxwellian speed x = |k_inf| / k0, density
// (4/sqrt(pi)) x^2 exp(-x^2).  Lower half: erf(x) - c x e^{-x^2} = u; upper
// half: erfc(x) + c x e^{-x^2} = 1 - u (exact for u >= 1/2), which keeps the
// tail well conditioned.  Safeguarded Newton iteration.
// The start of the FP64 iteration: the same safeguarded Newton iteration in
// FP32 (FP32 exp, erf and erfc issue on the fast pipe) to ~1e-5.  Where FP32
// cannot resolve the equation (u below ~1e-8: erf(x) and x e^{-x^2} cancel) the
// FP64 iteration starts from a poor point and takes more steps, nothing else.
__device__ __forceinline__ float maxwell_seed(bool upper, float v) {
  const float c = (float)TWO_OVER_SQRTPI;
  float lo = 0.0f, hi = 30.0f;
  float x = 1.0876520317f;   // median
  for (int it = 0; it < 40; ++it) {
    const float ex = expf(-x * x);
    const float q = upper ? erfcf(x) + c * x * ex : erff(x) - c * x * ex;
    const float dq = 2.0f * c * x * x * ex * (upper ? -1.0f : 1.0f);
    const bool below = upper ? (q > v) : (q < v);
    if (below) lo = x; else hi = x;
    float xn = x - (q - v) / dq;
    if (!(xn > lo && xn < hi)) xn = 0.5f * (lo + hi);
    if (fabsf(xn - x) <= 1e-5f * x || hi - lo <= 1e-6f * hi) return xn;
    x = xn;
  }
  return x;
}

// The whole iteration, for the tails outside the table.
static __device__ __noinline__ double maxwell_newton(double u) {
  const bool upper = u > 0.5;
  const double v = upper ? 1.0 - u : u;
  double lo = 0.0, hi = 30.0;
  double x = (double)maxwell_seed(upper, (float)v);
  if (!(x > lo && x < hi)) x = 1.0876520317;   // median
  for (int it = 0; it < 200; ++it) {
    const double ex = exp(-x * x);
    const double q = upper ? erfc(x) + TWO_OVER_SQRTPI * x * ex
                           : erf(x) - TWO_OVER_SQRTPI * x * ex;
    const double dq = 2.0 * TWO_OVER_SQRTPI * x * x * ex * (upper ? -1.0 : 1.0);
    // bracket update: the CDF increases with x, the tail decreases
    const bool below = upper ? (q > v) : (q < v);
    if (below) lo = x; else hi = x;
    double xn = x - (q - v) / dq;
    if (!(xn > lo && xn < hi)) xn = 0.5 * (lo + hi);
    // converged: a Newton step of a few ulps (one of exactly 1-2 ulps can
    // recur for ever where q - v is a rounding-level difference)
    if (fabs(xn - x) <= 1e-15 * x || hi - lo <= 4e-16 * hi) {
      x = xn;
      break;
    }
    x = xn;
  }
  return x;
}

// x with distribution u.  The FP32 iteration above finds the cell of the table
// (maxwell_table.inc, written at build time by maxwell.py), and the reversed
// Taylor series of the distribution about the cell's centre gives x to
// rounding: 12 FP64 instructions on a warp without a branch, where the Newton
// iteration took three or four rounds of exp and of both erf and erfc (lanes on
// either side of the median part ways).  Outside [1/32, 4), 2.4e-5 of the
// samples, the iteration itself.
#include "maxwell_table.inc"

__device__ __forceinline__ double maxwell_speed(int fa_model, double u) {
  if (fa_model == FA_DELTA) return 1.0;
  const double w = 1.0 - u;
  const bool upper = u > 0.5;
  const float s = maxwell_seed(upper, (float)(upper ? w : u));
  if (!(s >= 0x1p-5f && s < 4.0f)) return maxwell_newton(u);
  // cell: 7 leading mantissa bits below 2, 8 in [2, 4); its centre by the bits
  const uint32_t b = __float_as_uint(s);
  const bool high = s >= 2.0f;
  const uint32_t k = high ? b >> 15 : b >> 16;
  const int cell = high ? (int)(k - (0x40000000u >> 15)) + MAXWELL_LOW_CELLS
                        : (int)(k - (0x3d000000u >> 16));
  const double x0 = (double)__uint_as_float(high ? (k << 15) | 0x4000u : (k << 16) | 0x8000u);
  const double2* row = (const double2*)maxwell_table[cell];
  const double2 r0 = __ldg(row), r1 = __ldg(row + 1), r2 = __ldg(row + 2), r3 = __ldg(row + 3),
                r4 = __ldg(row + 4);
  const double t = ((cell >= MAXWELL_FIRST_UPPER ? w : u) - r0.x) * r0.y;
  double p = r4.y;
  p = p * t + r4.x;
  p = p * t + r3.y;
  p = p * t + r3.x;
  p = p * t + r2.y;
  p = p * t + r2.x;
  p = p * t + r1.y;
  p = p * t + r1.x;
  return x0 + (t + (t * t) * p);
}

}  // namespace sampling
}  // namespace rtk
