// Types of the conversion-surface sampling (rt_sample_core.cuh) that host code
// and other translation units need.
#pragma once

namespace rtk {
namespace sampling {

// Sample constants in the working type T: double for sampling, a dual number
// for the derivatives of the initial state and the weight with respect to the
// star parameters (the adjoint).  Only the fields a parameter can move are T.
template <class T>
struct SampConst {
  T rs, cp, sin_tm, cos_tm, B0_eV2, R_eV, n_inf, ma_eV;
  double v0, psi_fixed, plasma_a, g_eV, w_unit;
  double rlc;     // light-cylinder radius / R (twisted model: open field lines excluded)
  double per_cm3; // 1 cm^-3 in eV^3 (the renormalised weights)
  int disp, plasma, fa_model, phase_mode;
  int weight_mode;
};

template <class T>
struct SampOut {
  T x[3], k[3];   // scaled state: x / R, covariant k / m_a
  T w;            // weight [W]
  double delta, psi;
  bool ok;
};

}  // namespace sampling
}  // namespace rtk
