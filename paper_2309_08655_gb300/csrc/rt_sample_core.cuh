// Forward Monte-Carlo sampling of the resonant conversion surface: the
// per-sample computation shared by the sampling kernel (FP64) and the adjoint
// (dual numbers carrying derivatives with respect to the star parameters).
//
// Per sample (Sec. 3, Eqs. AxionCollInt and ForwardTracingEquation1; Sec. 4.2,
// Eq. PowerCurved; Sec. 4.3, Eq. GaussianDist): a direction n uniform on the
// sphere, a momentum direction khat uniform in the static orthonormal frame,
// the asymptotic axion speed from the Maxwellian, and the rotation phase.
// With khat and omega_inf = -k_t held fixed, the kinematic resonance
// k^a_mu = k^gamma_mu (Sec. 2.4, Sec. 4) on the radial line through n is the
// root of
//   G(r) = P(r) (1 + K2 s2) - (1 + K2),   K2(r) = omega_inf^2 / A(r) - 1,
// (units of m_a; s2 = sin^2 of the angle between khat and the dipole
// direction, constant along the line), obtained by substituting the axion's
// on-shell k into the anisotropic dispersion relation (Eq. AnisotrpoicDisp);
// G > 0 exactly where the LO photon is heavier than the axion.  For the
// isotropic plasma G = P - 1.
//
// Weight.  The power is the phase-space integral
//   P = int d^3k_loc dV sqrt(A) delta(E_gamma - E_a) Psi f_a,
//   Psi = (pi/2) g^2 |B|^2 (E^4 s2 / D) E,  D = c2 P (P - 2E^2) + E^4
// (Eq. PowerCurved with Eq. AngleDefAniso and Eq. CPAnisoCurved; isotropic:
// Psi = (pi/2) g^2 |B|^2 s2 E).  In the sample coordinates (n, khat, k_inf):
//   dV = A^{-1/2} r^2 dr dOmega_n,  d^3k_loc = (k k_inf / A) dk_inf dOmega_k,
//   int dr delta(h) = 1/|h'|,  f_a / pdf(k_inf) = n_inf / (4 pi k_inf^2),
// so W = 4 pi r^2 k n_inf Psi / (A k_inf |h'|), with h = E_gamma - E_a along the
// line and h' = G' / (2 E (E^2 - y_minus)), y_minus = K2 P c2 / E^2 the other
// root of the dispersion quadratic (isotropic: h' = P' / (2E)).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "rt_device.cuh"
#include "rt_dual.cuh"
#include "rt_maxwell.cuh"
#include "rt_sample_types.cuh"

namespace rtk {
namespace sampling {

struct Line {
  int disp, plasma;
  double rs, W2, s2, PR, pa, nz;
};

// P(r) and dP/dr along the radial line.
__device__ __forceinline__ void line_plasma(const Line& L, double r, double& P, double& dP) {
  switch (L.plasma) {
    case PLASMA_GJ: {
      const double ir = 1.0 / r;
      P = L.PR * ir * ir * ir;
      dP = -3.0 * P * ir;
      break;
    }
    case PLASMA_HOMOG: P = L.pa; dP = 0.0; break;
    case PLASMA_LINEAR_Z: P = L.pa * r * L.nz; dP = L.pa * L.nz; break;
    case PLASMA_RADIAL: {
      const double ir = 1.0 / r;
      P = L.pa * ir * ir * ir;
      dP = -3.0 * P * ir;
      break;
    }
    case PLASMA_TWISTED: {
      const double ir = 1.0 / r;
      P = L.PR * ir * ir * ir * ir;
      dP = -4.0 * P * ir;
      break;
    }
    default: P = 0.0; dP = 0.0; break;
  }
}

// G and G' in FP32 for the start of the FP64 root iteration; omega_inf^2 - 1
// (W2m1, a few 1e-6) is passed apart so that K2 keeps its FP32 precision.
__device__ __forceinline__ float line_G32(const Line& L, float W2m1, float r, float* dG) {
  const float ir = 1.0f / r;
  float P = 0.0f, dP = 0.0f;
  switch (L.plasma) {
    case PLASMA_GJ: P = (float)L.PR * ir * ir * ir; dP = -3.0f * P * ir; break;
    case PLASMA_HOMOG: P = (float)L.pa; break;
    case PLASMA_LINEAR_Z: P = (float)L.pa * r * (float)L.nz; dP = (float)(L.pa * L.nz); break;
    case PLASMA_RADIAL: P = (float)L.pa * ir * ir * ir; dP = -3.0f * P * ir; break;
    case PLASMA_TWISTED: P = (float)L.PR * ir * ir * ir * ir; dP = -4.0f * P * ir; break;
    default: break;
  }
  if (L.disp == DISP_ISO) {
    *dG = dP;
    return P - 1.0f;
  }
  const float rsr = (float)L.rs * ir;
  const float A = 1.0f - rsr;
  const float K2 = (W2m1 + rsr) / A;
  const float s2 = (float)L.s2;
  const float dK2 = -(1.0f + W2m1) * rsr * ir / (A * A);
  *dG = dP * (1.0f + K2 * s2) + P * s2 * dK2 - dK2;
  return P * (1.0f + K2 * s2) - (1.0f + K2);
}

__device__ __forceinline__ double line_G(const Line& L, double r, double* dG) {
  double P, dP;
  line_plasma(L, r, P, dP);
  if (L.disp == DISP_ISO) {
    if (dG) *dG = dP;
    return P - 1.0;
  }
  const double A = 1.0 - L.rs / r;
  const double K2 = L.W2 / A - 1.0;
  if (dG) {
    const double dK2 = -L.W2 * L.rs / (r * r * A * A);
    *dG = dP * (1.0 + K2 * L.s2) + P * L.s2 * dK2 - dK2;
  }
  return P * (1.0 + K2 * L.s2) - (1.0 + K2);
}


__device__ __forceinline__ double val(double x) { return x; }
__device__ __forceinline__ double tabs(double x) { return fabs(x); }

// The root r of G as a function of the constants: G(r; c) = 0 gives
// dr = -dG_c / G_r (the value stays the one the bracketed iteration found).
__device__ __forceinline__ double root_of(double r, double /*G*/, double /*dGdr*/) { return r; }

template <class T>
__device__ __forceinline__ void line_plasma_t(int plasma, const T& PR, double pa, double nz,
                                              const T& r, T& P, T& dP) {
  switch (plasma) {
    case PLASMA_GJ: {
      const T ir = rt_rcp(r);
      P = PR * ir * ir * ir;
      dP = T(-3.0) * P * ir;
      break;
    }
    case PLASMA_HOMOG: P = T(pa); dP = T(0.0); break;
    case PLASMA_LINEAR_Z: P = T(pa) * r * T(nz); dP = T(pa * nz); break;
    case PLASMA_RADIAL: {
      const T ir = rt_rcp(r);
      P = T(pa) * ir * ir * ir;
      dP = T(-3.0) * P * ir;
      break;
    }
    case PLASMA_TWISTED: {
      const T ir = rt_rcp(r);
      P = PR * ir * ir * ir * ir;
      dP = T(-4.0) * P * ir;
      break;
    }
    default: P = T(0.0); dP = T(0.0); break;
  }
}

// The root of G on the line for the profiles that fall as a power of r, where
// G decreases through a single root (0: not found this way).  The bracket and
// the Newton iteration run in FP32, to ~1e-6; in FP64 G alone is evaluated,
// and its quotient with the FP32 slope (good to 1e-6) converges in two steps.
// Every lane does the same two or three FP64 evaluations of G, where the
// bracketing in FP64 and a Newton iteration to the last bit took five to ten,
// each with its own count.
__device__ __forceinline__ double line_root_power(const Line& L, float W2m1) {
  if (L.plasma != PLASMA_GJ && L.plasma != PLASMA_RADIAL && L.plasma != PLASMA_TWISTED)
    return 0.0;
  float lo = 1.0f, hi = 2.0f, dG = 0.0f;
  for (int it = 0; !(line_G32(L, W2m1, hi, &dG) < 0.0f); ++it) {
    if (it > 40) return 0.0;
    lo = hi;
    hi *= 2.0f;
  }
  float x = 0.5f * (lo + hi);
  for (int it = 0; it < 40; ++it) {
    const float g = line_G32(L, W2m1, x, &dG);
    if (g > 0.0f) lo = x; else hi = x;
    float xn = x - g / dG;
    if (!(xn > lo && xn < hi)) xn = 0.5f * (lo + hi);
    const bool done = fabsf(xn - x) <= 1e-5f * x || hi - lo <= 1e-6f * hi;
    x = xn;
    if (done) break;
  }
  (void)line_G32(L, W2m1, x, &dG);
  if (!(dG < 0.0f)) return 0.0;
  const float idG = 1.0f / dG;
  double r = (double)x;
  for (int it = 0; it < 8; ++it) {
    const float step = (float)line_G(L, r, nullptr) * idG;
    r = fmax(r - (double)step, 1.0);
    if (fabsf(step) <= 1e-10f * x) return r;
  }
  return 0.0;
}

// The root of G for any profile (0: G does not change sign): bracketed by
// doubling, then safeguarded Newton to a few ulps from a start that the same
// iteration finds in FP32.
static __device__ __noinline__ double line_root(const Line L, float W2m1) {
  double lo = 1.0, hi = 2.0;
  int n = 0;
  while (!(line_G(L, hi, nullptr) < 0.0)) {
    lo = hi;
    hi *= 2.0;
    if (++n > 60) return 0.0;
  }
  double r = 0.5 * (lo + hi);
  {
    float flo = (float)lo, fhi = (float)hi, fr = (float)r;
    for (int it = 0; it < 40; ++it) {
      float dG;
      const float g = line_G32(L, W2m1, fr, &dG);
      if (g > 0.0f) flo = fr; else fhi = fr;
      float rn = fr - g / dG;
      if (!(rn > flo && rn < fhi)) rn = 0.5f * (flo + fhi);
      const bool done = fabsf(rn - fr) <= 1e-5f * fr || fhi - flo <= 1e-6f * fhi;
      fr = rn;
      if (done) break;
    }
    if ((double)fr > lo && (double)fr < hi) r = (double)fr;
  }
  for (int it = 0; it < 200; ++it) {
    double dG;
    const double g = line_G(L, r, &dG);
    if (g > 0.0) lo = r; else hi = r;
    double rn = r - g / dG;
    if (!(rn > lo && rn < hi)) rn = 0.5 * (lo + hi);
    const bool done = fabs(rn - r) <= 1e-15 * r || hi - lo <= 4e-16 * hi;
    r = rn;
    if (done) break;
  }
  return r;
}

// Gradient of G (units 1/R) at the point x (units of R) of the leaf selected by
// (khat = q, W2 = omega_inf^2): the header's G with the angular factors and
// A evaluated at x itself (dual numbers over x).  Along the radial line it is
// G' of the root search; across it, the tilt of the conversion surface.
__device__ __forceinline__ void grad_G(const SampConst<double>& s, double m0, double m1,
                                       double m2, const double* q, double W2, const double* x,
                                       double* g) {
  typedef Dual<3> D3;
  D3 X[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) X[i] = D3::var(x[i], i);
  const D3 r = rt_sqrt(X[0] * X[0] + X[1] * X[1] + X[2] * X[2]);
  const D3 ir = D3(1.0) / r;
  const D3 n0 = X[0] * ir, n1 = X[1] * ir, n2 = X[2] * ir;
  const D3 mu = D3(m0) * n0 + D3(m1) * n1 + D3(m2) * n2;
  const D3 A = D3(1.0) - D3(s.rs) * ir;
  const D3 K2 = D3(W2) / A - D3(1.0);
  D3 P(0.0);
  switch (s.plasma) {
    case PLASMA_GJ: P = D3(s.cp) * ir * ir * ir * dabs(D3(3.0) * n2 * mu - D3(m2)); break;
    case PLASMA_TWISTED: P = D3(s.cp) * (D3(1.0) - mu * mu) * ir * ir * ir * ir; break;
    case PLASMA_HOMOG: P = D3(s.plasma_a); break;
    case PLASMA_LINEAR_Z: P = D3(s.plasma_a) * X[2]; break;
    case PLASMA_RADIAL: P = D3(s.plasma_a) * ir * ir * ir; break;
    default: break;
  }
  D3 G;
  if (s.disp == DISP_ISO) {
    G = P - D3(1.0);
  } else {
    const D3 b0 = D3(3.0) * mu * n0 - D3(m0), b1 = D3(3.0) * mu * n1 - D3(m1),
             b2 = D3(3.0) * mu * n2 - D3(m2);
    const D3 kb = D3(q[0]) * b0 + D3(q[1]) * b1 + D3(q[2]) * b2;
    const D3 s2 = D3(1.0) - kb * kb / (D3(3.0) * mu * mu + D3(1.0));
    G = P * (D3(1.0) + K2 * s2) - (D3(1.0) + K2);
  }
#pragma unroll
  for (int i = 0; i < 3; ++i) g[i] = G.d[i];
}

// One sample from its six uniforms (the sample coordinates and the weight
// of the header comment).  inv_n: 1 / (number of samples).
template <class T>
__device__ void sample_core(const SampConst<T>& s, const double* u, double nsamp,
                            SampOut<T>& o) {
  // direction of the conversion point and of the momentum
  const double ct = 1.0 - 2.0 * u[0];
  const double st = sqrt(fmax(0.0, (1.0 - ct) * (1.0 + ct)));
  double sph, cph;
  sincospi(2.0 * u[1], &sph, &cph);
  const double n0 = st * cph, n1 = st * sph, n2 = ct;
  const double ck = 1.0 - 2.0 * u[2];
  const double sk = sqrt(fmax(0.0, (1.0 - ck) * (1.0 + ck)));
  double spk, cpk;
  sincospi(2.0 * u[3], &spk, &cpk);
  const double q0 = sk * cpk, q1 = sk * spk, q2 = ck;
  // asymptotic axion speed and the Killing energy omega_inf / m_a = 1 + delta
  const double xs = maxwell_speed(s.fa_model, u[4]);
  const double kinf = xs * s.v0;
  const double delta = kinf * kinf / (sqrt(1.0 + kinf * kinf) + 1.0);
  const double om = 1.0 + delta;
  const bool uniform_phase = s.phase_mode == PHASE_UNIFORM;
  const double psi = uniform_phase ? 2.0 * PI * u[5] : s.psi_fixed;
  double sps, cps;
  if (uniform_phase) sincospi(2.0 * u[5], &sps, &cps);   // no argument reduction by pi
  else sincos(psi, &sps, &cps);
  const T m0 = s.sin_tm * T(cps), m1 = s.sin_tm * T(sps), m2 = s.cos_tm;
  // dipole direction b = 3 (m.n) n - m (depends on n only)
  const T mu = m0 * T(n0) + m1 * T(n1) + m2 * T(n2);
  const T b0 = T(3.0) * mu * T(n0) - m0, b1 = T(3.0) * mu * T(n1) - m1,
          b2 = T(3.0) * mu * T(n2) - m2;
  const T bb = T(3.0) * mu * mu + T(1.0);
  const T kb = T(q0) * b0 + T(q1) * b1 + T(q2) * b2;
  const T c2 = kb * kb / bb;
  const T s2 = T(1.0) - c2;
  // the angular factor of P along the radial line: Goldreich-Julian
  // |3 n_z (m.n) - m_z|; twisted magnetosphere sin^2 of the magnetic colatitude
  const T PR = (s.plasma == PLASMA_TWISTED) ? s.cp * (T(1.0) - mu * mu)
                                            : s.cp * tabs(T(3.0) * T(n2) * mu - m2);
  Line L;
  L.disp = s.disp;
  L.plasma = s.plasma;
  L.rs = val(s.rs);
  L.W2 = om * om;
  L.s2 = val(s2);
  L.PR = val(PR);
  L.pa = s.plasma_a;
  L.nz = n2;
  o.delta = delta;
  o.psi = psi;
  o.ok = line_G(L, 1.0, nullptr) > 0.0;
  if (!o.ok) return;
  const float W2m1 = (float)(delta * (2.0 + delta));   // omega_inf^2 - 1
  double r = line_root_power(L, W2m1);
  if (r == 0.0) r = line_root(L, W2m1);
  if (r == 0.0) {
    o.ok = false;
    return;
  }
  // twisted magnetosphere: no conversion on open field lines, the dipole
  // lines r / sin^2(theta) = L that reach the light cylinder (L >= r_LC)
  if (s.plasma == PLASMA_TWISTED && r >= s.rlc * (1.0 - val(mu) * val(mu))) {
    o.ok = false;
    return;
  }
  // G in the working type at the root, for the root's dependence on the constants
  T rT;
  if constexpr (std::is_same<T, double>::value) {
    rT = r;
  } else {
    double dGr;
    line_G(L, r, &dGr);
    T P, dP;
    line_plasma_t(s.plasma, PR, s.plasma_a, n2, T(r), P, dP);
    T G;
    if (s.disp == DISP_ISO) {
      G = P - T(1.0);
    } else {
      const T A = T(1.0) - s.rs * T(1.0 / r);
      const T K2 = T(L.W2) / A - T(1.0);
      G = P * (T(1.0) + K2 * s2) - (T(1.0) + K2);
    }
    rT = root_of(r, G, dGr);
  }
  // quantities at the resonance.  One reciprocal each for r and A, one rsqrt
  // for E and one quotient for the whole weight: an FP64 division is ten
  // instructions of a pipe that takes 64 cycles for each.
  T P, dP;
  line_plasma_t(s.plasma, PR, s.plasma_a, n2, rT, P, dP);
  const T ir = rt_rcp(rT);
  const T rsr = s.rs * ir;
  const T A = T(1.0) - rsr;
  const T qA = rt_rsqrt(A);
  const T iA = qA * qA;
  const T K2 = T(L.W2) * iA - T(1.0);          // on shell with the rounded omega_inf^2
  const T E2 = T(1.0) + K2;
  const T kloc = rt_sqrt(K2);
  // dh/dr = dG / hden with hden = 2 E (E^2 - y_minus) = 2 hE / E (isotropic: 2 E),
  // the shape factor E^4 s2 / D = shape / D
  T dG, hE, shape, D;
  if (s.disp == DISP_ISO) {
    dG = dP;
    hE = E2;
    shape = s2;
    D = T(1.0);
  } else {
    const T dK2 = -T(L.W2) * rsr * ir * iA * iA;
    const T E4 = E2 * E2;
    dG = dP * (T(1.0) + K2 * s2) + P * s2 * dK2 - dK2;
    hE = E4 - K2 * P * c2;
    D = c2 * P * (P - T(2.0) * E2) + E4;
    shape = E4 * s2;
  }
  // w = W1 Psi, W1 = 4 pi r^2 (kloc / kinf) n_inf / (A |dh/dr|) and
  // Psi = (pi/2) g^2 (B0/2)^2 r^-6 bb (shape / D) E, the sizes in eV
  const T pre = T(PI * PI * s.g_eV * s.g_eV * s.w_unit) * s.n_inf * s.B0_eV2 * s.B0_eV2 *
                (s.R_eV * s.R_eV * s.R_eV);
  const T ir2 = ir * ir;
  o.w = pre * (ir2 * ir2) * bb * kloc * hE * shape / (T(nsamp * kinf) * A * tabs(dG) * D);
  if constexpr (std::is_same<T, double>::value) {
    if (s.weight_mode == WEIGHT_UNIT_P || s.weight_mode == WEIGHT_RENORM) {
      // conversion probability set to one (Sec. 5.1): divide by
      // P_agamma = Psi / |k . dE| (Eq. CPAnisoCurved), dE the proper-frame
      // gradient of h = E_gamma - E_a; dh = dG / (2 E (E^2 - y_minus)) (as h')
      const double q[3] = {q0, q1, q2};
      const double xr[3] = {rT * n0, rT * n1, rT * n2};
      double g[3];
      grad_G(s, m0, m1, m2, q, L.W2, xr, g);
      const double gn = g[0] * n0 + g[1] * n1 + g[2] * n2;
      const double sA = sqrt(A);
      double kg = 0.0;
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        const double ni = (i == 0) ? n0 : (i == 1) ? n1 : n2;
        kg += q[i] * (g[i] + (sA - 1.0) * gn * ni);
      }
      // W1 |k . dE|: the factor 1 / hden of dE and of dh cancel
      const double r_eV = rT * s.R_eV;
      const double W1 = 4.0 * PI * r_eV * r_eV * (kloc / kinf) * s.n_inf / (A * fabs(dG));
      o.w = W1 * (kloc * s.ma_eV * fabs(kg)) / nsamp * s.w_unit;
      if (s.weight_mode == WEIGHT_RENORM) {
        // Eq. reweight: x (1 cm^-3 / n_a(r)) (m_a / |k_a|) / sqrt(1 - r_s / r), the
        // focused density of the monochromatic distribution n_inf k_c / k0,
        // k_c^2 = k0^2 + m_a^2 r_s / r (Sec. 4.3)
        const double kc_over_k0 = sqrt(s.v0 * s.v0 + s.rs / rT) / s.v0;
        o.w *= (s.per_cm3 / (s.n_inf * kc_over_k0)) / kloc / sA;
      }
    }
  }
  // photon phase-space point: orthonormal k = |k| khat; covariant Cartesian
  // k = k_o + (1/sqrt(A) - 1) (n.k_o) n
  const T nko = kloc * T(n0 * q0 + n1 * q1 + n2 * q2);
  const T cr = (qA - T(1.0)) * nko;
  o.x[0] = rT * T(n0);
  o.x[1] = rT * T(n1);
  o.x[2] = rT * T(n2);
  o.k[0] = kloc * T(q0) + cr * T(n0);
  o.k[1] = kloc * T(q1) + cr * T(n1);
  o.k[2] = kloc * T(q2) + cr * T(n2);
}

// Squared angle within which a Goldreich-Julian sample counts as next to the
// null cone: 1e-2 rad (the cost-ordered claims' two nearest buckets), with room
// for this test's FP32 rounding.
constexpr float GUIDED_DIST2 = 1.05e-4f;

// Whether a sample lies within GUIDED_DIST2 of the null cone, (F / |grad_n F|)^2 as
// cone_dist2 of rt_integrator.cuh, in FP32.
__device__ __forceinline__ bool next_to_null_cone(const SampConst<double>& s, const double* x,
                                                  double psi) {
  if (s.plasma != PLASMA_GJ) return false;
  const float x0 = (float)x[0], x1 = (float)x[1], x2 = (float)x[2];
  float sp, cp;
  sincosf((float)psi, &sp, &cp);
  const float st = (float)s.sin_tm, m2 = (float)s.cos_tm;
  const float ir = rsqrtf(x0 * x0 + x1 * x1 + x2 * x2), n2 = x2 * ir;
  const float mu = st * (cp * x0 + sp * x1) * ir + m2 * n2;
  const float F = 3.0f * n2 * mu - m2, c = 6.0f * mu * n2;
  const float g2 = 9.0f * (mu * mu + n2 * n2) + 18.0f * mu * n2 * m2 - c * c;
  return F * F < GUIDED_DIST2 * g2;
}

// The state of one sample (not its weight) by iterating the speed and the
// resonance radius to the last bit in FP64.  For the samples next to the null
// cone: a ray guided along it for thousands of steps carries a last-bit change of
// its start to another end point (in the mixed-precision trace, to another bin or
// fate), so these starts keep this arithmetic, operation for operation.
__device__ __forceinline__ void sample_state_iterated(const SampConst<double>& s, const double* u,
                                                      SampOut<double>& o) {
  const double ct = 1.0 - 2.0 * u[0];
  const double st = sqrt(fmax(0.0, (1.0 - ct) * (1.0 + ct)));
  double sph, cph;
  sincospi(2.0 * u[1], &sph, &cph);
  const double n0 = st * cph, n1 = st * sph, n2 = ct;
  const double ck = 1.0 - 2.0 * u[2];
  const double sk = sqrt(fmax(0.0, (1.0 - ck) * (1.0 + ck)));
  double spk, cpk;
  sincospi(2.0 * u[3], &spk, &cpk);
  const double q0 = sk * cpk, q1 = sk * spk, q2 = ck;
  const double kinf = (s.fa_model == FA_DELTA ? 1.0 : maxwell_newton(u[4])) * s.v0;
  const double delta = kinf * kinf / (sqrt(1.0 + kinf * kinf) + 1.0);
  const double om = 1.0 + delta;
  const double psi = (s.phase_mode == PHASE_UNIFORM) ? 2.0 * PI * u[5] : s.psi_fixed;
  double sps, cps;
  sincos(psi, &sps, &cps);
  const double m0 = s.sin_tm * cps, m1 = s.sin_tm * sps, m2 = s.cos_tm;
  const double mu = m0 * n0 + m1 * n1 + m2 * n2;
  const double b0 = 3.0 * mu * n0 - m0, b1 = 3.0 * mu * n1 - m1, b2 = 3.0 * mu * n2 - m2;
  const double bb = 3.0 * mu * mu + 1.0;
  const double kb = q0 * b0 + q1 * b1 + q2 * b2;
  const double c2 = kb * kb / bb;
  Line L;
  L.disp = s.disp;
  L.plasma = s.plasma;
  L.rs = s.rs;
  L.W2 = om * om;
  L.s2 = 1.0 - c2;
  L.PR = s.cp * fabs(3.0 * n2 * mu - m2);
  L.pa = s.plasma_a;
  L.nz = n2;
  o.delta = delta;
  o.psi = psi;
  o.ok = line_G(L, 1.0, nullptr) > 0.0;
  if (!o.ok) return;
  const double r = line_root(L, (float)(delta * (2.0 + delta)));
  if (r == 0.0) {
    o.ok = false;
    return;
  }
  const double A = 1.0 - s.rs / r;
  const double K2 = L.W2 / A - 1.0;
  const double kloc = sqrt(K2);
  const double nko = kloc * (n0 * q0 + n1 * q1 + n2 * q2);
  const double cr = (1.0 / sqrt(A) - 1.0) * nko;
  o.x[0] = r * n0;
  o.x[1] = r * n1;
  o.x[2] = r * n2;
  o.k[0] = kloc * q0 + cr * n0;
  o.k[1] = kloc * q1 + cr * n1;
  o.k[2] = kloc * q2 + cr * n2;
}

}  // namespace sampling
}  // namespace rtk
