// Six lanes per ray: the group integrator of the FP64 tail mode (rt_tail.cu)
// and of the express lane of cost-ordered tracing (rt_trace.cu).
//
// On GB300 an FP64 warp instruction occupies its SM sub-partition for the same
// 64 cycles whether 1 or 32 lanes are live, so once the work queue has drained
// a warp that still holds a few long rays (those guided along the
// Goldreich-Julian null cone take 10^4 - 10^5 steps) spends the FP64 pipe on
// one lane per instruction.  Such rays are parked by the persistent kernel
// (their complete integrator state, so the continuation is the same
// computation) and continued with one lane per state component: lane c
// of a six-lane group owns y_c, its stage derivatives and the stage sums, and
// the right-hand side's scalars are shared out over the lanes.  The steps, the
// error norm, the controller and the events are those of advance() in
// rt_integrator.cuh; the arithmetic of the component sums and of the error-norm
// sum is ordered differently, so results agree with the lane-per-ray path to
// rounding.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "rt_device.cuh"
#include "rt_guided.cuh"
#include "rt_integrator.cuh"
#include "rt_internal.h"

namespace rtk {

namespace {

constexpr int GROUP = 6;           // lanes per ray
constexpr int GROUPS_PER_WARP = 5;

__device__ __forceinline__ int find_star(const TraceParams& p, int64_t i) {
  if (p.nstars <= 1) return 0;
  int lo = 0, hi = p.nstars - 1;   // offsets[s] <= i < offsets[s + 1]
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (p.offsets[mid] <= i) lo = mid; else hi = mid - 1;
  }
  return lo;
}

__device__ void load_lane(const TraceParams& p, int64_t i, Lane& L) {
  const StarDev& s = p.stars[find_star(p, i)];
  const int64_t n = p.n;
  L.R_km = s.R_km;
  L.ma_eV = s.ma_eV;
  const double iR = 1.0 / s.R_km, im = 1.0 / s.ma_eV;
  L.y[0] = p.state[i] * iR;
  L.y[1] = p.state[n + i] * iR;
  L.y[2] = p.state[2 * n + i] * iR;
  L.y[3] = p.state[3 * n + i] * im;
  L.y[4] = p.state[4 * n + i] * im;
  L.y[5] = p.state[5 * n + i] * im;
  const double om = 1.0 + p.state[6 * n + i];
  const double psi = p.state[7 * n + i];
  double sp, cpsi;
  sincos(psi, &sp, &cpsi);
  L.c.rs = s.rs_prop;
  L.c.cp = s.cp;
  L.c.pa = s.plasma_a;
  L.c.W2 = om * om;
  L.c.iW2 = 1.0 / (om * om);
  L.c.m0 = s.sin_tm * cpsi;
  L.c.m1 = s.sin_tm * sp;
  L.c.m2 = s.cos_tm;
  L.c.disp = s.dispersion;
  L.c.plasma = s.plasma;
  L.c.sig = gj_side<double>(L.c.m0, L.c.m1, L.c.m2, L.y[0], L.y[1], L.y[2]);
  L.switching = false;
  L.h_resume = 0.0;
  rhs64(L.c, L.y, L.f0);
  const double hmax = (p.lambda_max > 0.0) ? p.lambda_max : 1e30;
  L.h = initial_step(L.c, L.y, L.f0, p.rtol, p.atol, hmax);
  L.lam = 0.0;
  L.na = 0;
  L.nr = 0;
  if (p.claim_status == RAY_PROMOTED) {   // resume a ray handed over by the FP32 pass
    if (p.nacc) L.na = p.nacc[i];
    if (p.nrej) L.nr = p.nrej[i];
  }
  L.last_rej = false;
}

// A READY ray's park record: the start of load_lane.
__device__ void fresh_record(const TraceParams& p, int64_t ray, double* pe) {
  Lane L;
  load_lane(p, ray, L);
#pragma unroll
  for (int j = 0; j < 6; ++j) pe[j] = L.y[j];
  pe[6] = L.h;
  pe[7] = 0.0;
  pe[8] = L.c.sig;
  pe[9] = 0.0;
  pe[10] = 0.0;
  pe[11] = 0.0;
  pe[12] = (double)ray;
  pe[13] = 0.0;
}

// The group's right-hand side as passes over a small register file in shared
// memory.
//
// An FP64 instruction costs a warp 64 cycles whether the lanes of a group do the
// same work or six different products, and a launch of guided rays ends with its
// longest ray: what counts is the number of FP64 instructions one after another,
// and what stands between them.  So the scalar coefficients of the anisotropic
// Goldreich-Julian and twisted media are formed in passes: in each, the six lanes
// take one multiply-add whose operands they read from slots of their own choice,
// and store the result to a slot.  The slot numbers are one table, read into
// registers when a ray is taken up, so a pass is three loads, the multiply-add and
// a store: 32 FP64 instructions a right-hand side, where every lane forming every
// scalar takes 105.  A lone guided ray: 12.8 us an attempt (26 k cycles, of which
// about 310 FP64 instructions take 20 k), 33 us with the prefix formed by every
// lane; operands exchanged by shuffles and picked by selects took 13 other
// instructions for each FP64 one, 23.5 us.
//
// Slots: the point, the ray's constants, plain numbers, then what the passes
// leave.
enum Slot : int {
  S_X = 0,                                      // x0 x1 x2 k0 k1 k2
  S_M = 6, S_M3 = 9,                            // m, 3 m
  S_RS = 12, S_CPS, S_FB, S_W2, S_IW2,          // rs, cp sig, W2, 1/W2
  S_0, S_1, S_N1, S_2, S_N2, S_3, S_FA, S_QA, S_QB,    // F = FA . + FB, qn = QA . + QB
  S_IR, S_DOT,                                  // 1/r; x.k, m.x, k.m, |x|^2, 3 m.x
  S_Q = S_DOT + 6,                              // 1/sqrt(A) (0-2), 1/|b| (3-5)
  S_P1 = S_Q + 6                                // pass n at S_P1 + 6 (n - 1)
};
constexpr int PASSES = 14;
constexpr int SLOTS = S_P1 + 6 * PASSES;

constexpr int res(int pass, int lane) { return S_P1 + 6 * (pass - 1) + lane; }

// what the passes leave
enum Value : int {
  V_KR = res(1, 0), V_MU = res(1, 1), V_NZ = res(1, 2), V_IR2 = res(1, 3), V_MU3 = res(1, 4),
  V_U = res(1, 5),
  V_A = res(2, 0), V_QA = S_Q, V_IB = S_Q + 3,
  V_IR3 = res(3, 0), V_MN = res(3, 1), V_UKR = res(3, 2), V_DA = res(3, 3), V_KR2 = res(3, 4),
  V_MKR = res(3, 5),
  V_G3 = res(4, 0), V_F = res(4, 1), V_QN = res(4, 2), V_SA = res(4, 3), V_IA = res(4, 4),
  V_IB2 = res(4, 5),
  V_P = res(5, 0), V_T = res(5, 1), V_BX0 = res(5, 2), V_OPSA = res(5, 3), V_IA2 = res(5, 4),
  V_DAQ = res(5, 5),
  V_C1 = res(6, 0), V_OKR = res(6, 1), V_PA = res(6, 2), V_QM = res(6, 3), V_W2IA2 = res(6, 4),
  V_A3 = res(6, 5),
  V_UU = res(7, 0), V_IBIW2 = res(7, 1), V_C1KR = res(7, 2), V_PA2 = res(7, 3), V_S1 = res(7, 4),
  V_AIW2 = res(7, 5),
  V_KP = res(8, 0), V_M3U = res(8, 1), V_NIB2 = res(8, 2), V_NAIW2 = res(8, 3),
  V_NC1 = res(8, 4), V_NP = res(8, 5),
  V_KP2 = res(9, 0), V_A1 = res(9, 1), V_QIB = res(9, 2), V_NA3 = res(9, 3),
  V_ONEM = res(10, 0), V_GM = res(10, 1), V_D = res(10, 2), V_KQ = res(10, 3),
  V_NA1 = res(10, 4),
  V_W = res(11, 0), V_GMR = res(11, 1), V_BX = res(11, 2), V_S = res(11, 3), V_Z = res(11, 4),
  V_WQM = res(12, 0), V_GMZ = res(12, 1), V_CK = res(12, 2), V_VS = res(12, 3), V_WQZ = res(12, 4),
  V_NGA1 = res(12, 5),
  V_CM = res(13, 0), V_E = res(13, 1),
  V_CN = res(14, 0)
};

// Operands of pass n (2 and up to 14): result = a b + c per lane.  Pass 1 (the
// products with 1/r) and the dot products before it are written out.  The media
// differ in the plasma's terms, P = g F and dP = t (qn n + qm m + qz e_z) with
// t = g / r, as ham_rhs64:
//   Goldreich-Julian  g = cp sig r^-3, F = 3 mu n_z - m_z, qn = -15 mu n_z + 3 m_z,
//                     qm = 3 n_z, qz = 3 mu
//   twisted           g = cp r^-4, F = 1 - mu^2, qn = 6 mu^2 - 4, qm = -2 mu, qz = 0
#define RT_PASSES(RA, RB, MA, MB, QMA, QMB, QZ) {                                             \
    /* A, and |b|^2 = 3 mu^2 + 1 */                                                           \
    {{V_U, S_N1, S_1}, {V_U, S_N1, S_1}, {V_U, S_N1, S_1}, {V_MU3, V_MU, S_1},                \
     {V_MU3, V_MU, S_1}, {V_MU3, V_MU, S_1}},                                                 \
    /* r^-3, mu n_z, (rs/r) kr, dA/dr, kr^2, mu kr */                                         \
    {{RA, RB, S_0}, {MA, MB, S_0}, {V_U, V_KR, S_0}, {S_RS, V_IR2, S_0},                      \
     {V_KR, V_KR, S_0}, {V_MU, V_KR, S_0}},                                                   \
    /* g3 = cp sig r^-3, F, qn, sqrt(A), 1/A, 1/|b|^2 */                                      \
    {{S_CPS, V_IR3, S_0}, {S_FA, V_MN, S_FB}, {S_QA, V_MN, S_QB}, {V_A, V_QA, S_0},           \
     {V_QA, V_QA, S_0}, {V_IB, V_IB, S_0}},                                                   \
    /* P, t, -2 (rs/r) kr, 1 + 2 sqrt(A), 1/A^2, dA/dr / sqrt(A) */                           \
    {{V_G3, V_F, S_0}, {V_G3, S_IR, S_0}, {S_N2, V_UKR, S_0}, {S_2, V_SA, S_1},               \
     {V_IA, V_IA, S_0}, {V_DA, V_QA, S_0}},                                                   \
    /* c1, opsA kr, P A, qm, W2/A^2, a3 */                                                    \
    {{V_MU, V_OPSA, S_0}, {V_OPSA, V_KR, S_0}, {V_P, V_A, S_0}, {QMA, QMB, S_0},              \
     {S_W2, V_IA2, S_0}, {V_MKR, V_DAQ, S_0}},                                                \
    /* U, 1/(|b| W2), c1 kr, 2 P A, W2/A^2 + 3 kr^2, A/W2 */                                  \
    {{V_C1, V_KR, S_DOT + 5}, {V_IB, S_IW2, S_0}, {V_C1, V_KR, S_0}, {S_2, V_PA, S_0},        \
     {S_3, V_KR2, V_W2IA2}, {V_A, S_IW2, S_0}},                                               \
    /* Kp, 3 mu U, and the negatives of 1/|b|^2, A/W2, c1, P */                               \
    {{V_UU, V_IB, S_0}, {V_MU3, V_UU, S_0}, {S_N1, V_IB2, S_0}, {S_N1, V_AIW2, S_0},          \
     {S_N1, V_C1, S_0}, {S_N1, V_P, S_0}},                                                    \
    /* Kp^2, a1, Kp/(|b| W2), -a3 */                                                          \
    {{V_KP, V_KP, S_0}, {V_M3U, V_NIB2, V_OKR}, {V_KP, V_IBIW2, S_0}, {S_N1, V_A3, S_0},      \
     {S_0, S_0, S_0}, {S_0, S_0, S_0}},                                                       \
    /* 1 - A Kp^2/W2, gm, a1 mu + c1 kr, Kp^2/W2, -a1 */                                      \
    {{V_NAIW2, V_KP2, S_1}, {V_PA2, V_QIB, S_0}, {V_A1, V_MU, V_C1KR}, {V_KP2, S_IW2, S_0},   \
     {S_N1, V_A1, S_0}, {S_0, S_0, S_0}},                                                     \
    /* w, gm/r, bx, s, z = (a1 mu + c1 kr)/r - a3 */                                          \
    {{V_T, V_ONEM, S_0}, {V_GM, S_IR, S_0}, {V_GM, V_NC1, V_BX0}, {V_NP, V_KQ, V_S1},         \
     {S_IR, V_D, V_NA3}, {S_0, S_0, S_0}},                                                    \
    /* w qm, gm z, Ck, dA/dr s, w qz, -gm a1 / r */                                           \
    {{V_W, V_QM, S_0}, {V_GM, V_Z, S_0}, {V_BX, S_IR, S_0}, {V_DA, V_S, S_0},                 \
     {V_W, QZ, S_0}, {V_GMR, V_NA1, S_0}},                                                    \
    /* Cm, w qn + gm z */                                                                     \
    {{S_1, V_WQM, V_NGA1}, {V_W, V_QN, V_GMZ}, {S_0, S_0, S_0}, {S_0, S_0, S_0},              \
     {S_0, S_0, S_0}, {S_0, S_0, S_0}},                                                       \
    /* Cn */                                                                                  \
    {{S_1, V_E, V_VS}, {S_0, S_0, S_0}, {S_0, S_0, S_0}, {S_0, S_0, S_0}, {S_0, S_0, S_0},    \
     {S_0, S_0, S_0}}}
__constant__ unsigned char c_pass[2][PASSES - 1][GROUP][3] = {
    RT_PASSES(V_IR2, S_IR, V_MU, V_NZ, S_3, V_NZ, V_MU3),
    RT_PASSES(V_IR2, V_IR2, V_MU, V_MU, S_N2, V_MU, S_0)};
#undef RT_PASSES

// A lane's view of its group's slots: byte offsets of its operands.
struct GroupFile {
  double* s;                        // the group's SLOTS slots
  unsigned off[PASSES - 1][3];
  int cc, j;                        // component, and component mod 3
  unsigned gm;
};

__device__ __forceinline__ void file_init(GroupFile& f, double* slots, int cc, unsigned gm) {
  f.s = slots;
  f.cc = cc;
  f.j = cc < 3 ? cc : cc - 3;
  f.gm = gm;
}

__device__ __forceinline__ double slot_at(const GroupFile& f, unsigned off) {
  return *(const double*)((const char*)f.s + off);
}

// The ray's constants, and the plain numbers (every lane of the group).
__device__ __forceinline__ void file_ray(GroupFile& f, const RayConst<double>& c) {
  const bool gj = c.plasma == PLASMA_GJ;
#pragma unroll
  for (int p = 0; p < PASSES - 1; ++p)
#pragma unroll
    for (int q = 0; q < 3; ++q) f.off[p][q] = 8u * c_pass[gj ? 0 : 1][p][f.cc][q];
  __syncwarp(f.gm);
  double* s = f.s;
  if (f.cc == 0) {
    s[S_M] = c.m0;
    s[S_M + 1] = c.m1;
    s[S_M + 2] = c.m2;
    s[S_M3] = 3.0 * c.m0;
    s[S_M3 + 1] = 3.0 * c.m1;
    s[S_M3 + 2] = 3.0 * c.m2;
    s[S_RS] = c.rs;
    s[S_CPS] = gj ? c.cp * c.sig : c.cp;
    s[S_FA] = gj ? 3.0 : -1.0;
    s[S_FB] = gj ? -c.m2 : 1.0;
    s[S_QA] = gj ? -15.0 : 6.0;
    s[S_QB] = gj ? 3.0 * c.m2 : -4.0;
    s[S_W2] = c.W2;
    s[S_IW2] = c.iW2;
    s[S_0] = 0.0;
    s[S_1] = 1.0;
    s[S_N1] = -1.0;
    s[S_2] = 2.0;
    s[S_N2] = -2.0;
    s[S_3] = 3.0;
  }
  __syncwarp(f.gm);
}

// Own component (0-2: dx_j/dl, 3-5: dk_j/dl) of the right-hand side at the point
// whose own component is yc.  *r2 = |x|^2 and *F the null-cone factor there (any
// positive multiple of it: its sign is the side; meaningful for Goldreich-Julian).
__device__ __forceinline__ double rhs_group(const GroupFile& f, const RayConst<double>& c,
                                            double yc, double* r2, double* F) {
  double* s = f.s;
  __syncwarp(f.gm);
  s[S_X + f.cc] = yc;
  __syncwarp(f.gm);
  if ((c.plasma != PLASMA_GJ && c.plasma != PLASMA_TWISTED) || c.disp == DISP_ISO) {
    // every lane evaluates the whole right-hand side and keeps its component
    double y[6], g[6];
#pragma unroll
    for (int q = 0; q < 6; ++q) y[q] = s[S_X + q];
    rhs64(c, y, g);
    *r2 = y[0] * y[0] + y[1] * y[1] + y[2] * y[2];
    *F = c.plasma == PLASMA_GJ ? 3.0 * y[2] * (c.m0 * y[0] + c.m1 * y[1] + c.m2 * y[2]) - c.m2 * *r2
                               : 1.0;
    double out = g[0];
#pragma unroll
    for (int q = 1; q < 6; ++q) out = f.cc == q ? g[q] : out;
    return out;
  }
  // x.k, m.x, k.m, |x|^2, 3 m.x, -k.m
  const double* va = s + (f.cc == 2 || f.cc == 5 ? S_X + 3 : S_X);
  const double* vb = s + (f.cc == 0 ? S_X + 3 : f.cc == 3 ? S_X : f.cc == 4 ? S_M3 : S_M);
  double d = va[0] * vb[0] + va[1] * vb[1] + va[2] * vb[2];
  s[S_DOT + f.cc] = f.cc == 5 ? -d : d;
  __syncwarp(f.gm);
  const double rr = s[S_DOT + 3];
  const double ir = inv_sqrt(rr);
  // kr, mu, n_z, r^-2, 3 mu, rs/r
  const double v1 = f.cc == 2 ? s[S_X + 2] : f.cc == 3 ? ir : f.cc == 5 ? s[S_RS] : d;
  s[S_P1 + f.cc] = ir * v1;
  s[S_IR] = ir;                       // every lane the same value
  const double nj = ir * s[S_X + f.j];
  __syncwarp(f.gm);
  auto pass = [&](int n) {
    const unsigned* o = f.off[n - 2];
    return fma(slot_at(f, o[0]), slot_at(f, o[1]), slot_at(f, o[2]));
  };
  double* out = s + S_P1 + f.cc;
  const double p2 = pass(2);
  out[6] = p2;
  out[12] = pass(3);
  s[S_Q + f.cc] = inv_sqrt(p2);
  __syncwarp(f.gm);
#pragma unroll
  for (int n = 4; n <= PASSES; ++n) {
    out[6 * (n - 1)] = pass(n);
    __syncwarp(f.gm);
  }
  // 2 k + bx n + gm m, or -(Cn n + Ck k + Cm m + Cz e_z)
  const bool pos = f.cc < 3;
  const double al = s[pos ? (int)S_2 : (int)V_CK], be = s[pos ? (int)V_BX : (int)V_CN],
               ga = s[pos ? (int)V_GM : (int)V_CM], dz = s[f.cc == 5 ? (int)V_WQZ : (int)S_0];
  const double g = fma(be, nj, fma(al, s[S_X + 3 + f.j], fma(ga, s[S_M + f.j], dz)));
  *r2 = rr;
  *F = s[V_F];
  return pos ? g : -g;
}

// Group state: lane c of a group owns component c; the rest is replicated.
struct GLane {
  RayConst<double> c;
  double yc, f0c;      // own component of the state and of f at the state
  double r2;           // |x|^2 at the state
  double h, h_resume, lam;
  int na, nr;
  bool last_rej, switching;
  int64_t ray;
  int star;
};

// The group's three position values of v to every lane of the group.
__device__ __forceinline__ void gather3d(unsigned gm, int base, double v, double* out) {
#pragma unroll
  for (int q = 0; q < 3; ++q) out[q] = __shfl_sync(gm, v, base + q);
}

// The other side of the null cone from here on, and the derivative there.
__device__ __forceinline__ void flip_side(const GroupFile& f, GLane& L) {
  L.c.sig = -L.c.sig;
  __syncwarp(f.gm);
  if (f.cc == 0) f.s[S_CPS] = L.c.cp * L.c.sig;
  double F;
  L.f0c = rhs_group(f, L.c, L.yc, &L.r2, &F);
}

// The group's three position values of v in FP32 (for the events' models).
__device__ __forceinline__ void gather3(unsigned gm, int base, double v, float* out) {
  const float f = narrow(v);
#pragma unroll
  for (int q = 0; q < 3; ++q) out[q] = __shfl_sync(gm, f, base + q);
}

// One attempted step of the group's ray; the same decisions as advance().
__device__ __forceinline__ int advance_group(const TraceParams& p, const GroupFile& f, GLane& L,
                                             int cc, unsigned gm, int base) {
  if (L.na >= p.max_steps || L.na + L.nr >= 4 * p.max_steps) return RAY_MAXSTEPS;
  bool clipped = false;
  double h = L.h;
  {
    // |f_x|^2: the three position lanes' squares
    const double q = L.f0c * L.f0c;
    const double v2 = __shfl_sync(gm, q, base) + __shfl_sync(gm, q, base + 1) +
                      __shfl_sync(gm, q, base + 2);
    if (h * h * v2 > STEP_REACH * STEP_REACH * L.r2) h = STEP_REACH * sqrt(L.r2 / v2);
  }
  if (p.lambda_max > 0.0 && L.lam + h >= p.lambda_max) {
    h = p.lambda_max - L.lam;
    clipped = true;
  }
  const double y = L.yc;
  double K1 = L.f0c, K2, K3, K4, K5, K6, K7, r2s, Fs;
  K2 = rhs_group(f, L.c, y + h * (DP::a21 * K1), &r2s, &Fs);
  K3 = rhs_group(f, L.c, y + h * (DP::a31 * K1 + DP::a32 * K2), &r2s, &Fs);
  K4 = rhs_group(f, L.c, y + h * (DP::a41 * K1 + DP::a42 * K2 + DP::a43 * K3), &r2s, &Fs);
  K5 = rhs_group(f, L.c, y + h * (DP::a51 * K1 + DP::a52 * K2 + DP::a53 * K3 + DP::a54 * K4), &r2s,
                 &Fs);
  K6 = rhs_group(
      f, L.c, y + h * (DP::a61 * K1 + DP::a62 * K2 + DP::a63 * K3 + DP::a64 * K4 + DP::a65 * K5),
      &r2s, &Fs);
  const double yn = y + h * (DP::b1 * K1 + DP::b3 * K3 + DP::b4 * K4 + DP::b5 * K5 + DP::b6 * K6);
  double rnew2, Fnew;
  K7 = rhs_group(f, L.c, yn, &rnew2, &Fnew);
  const double e = h * (DP::e1 * K1 + DP::e3 * K3 + DP::e4 * K4 + DP::e5 * K5 + DP::e6 * K6 +
                        DP::e7 * K7);
  const double eq = quotient(e, p.atol + p.rtol * max_abs(y, yn));
  // the sum over the group: lanes c and c + 3 form the same pair sum, so every
  // lane holds the same bits
  const double pair = eq * eq + __shfl_sync(gm, eq * eq, base + (cc < 3 ? cc + 3 : cc - 3));
  const double en2 = (__shfl_sync(gm, pair, base) + __shfl_sync(gm, pair, base + 1) +
                      __shfl_sync(gm, pair, base + 2)) * (1.0 / 6.0);
  if ((__double2hiint(en2) & 0x7ff00000) == 0x7ff00000) {   // infinite or NaN
    ++L.nr;
    L.h = h * 0.2;
    L.last_rej = true;
    return (L.h < 1e-12) ? RAY_NAN : -1;
  }
  const bool ok = en2 <= 1.0;
  const bool gj = (L.c.plasma == PLASMA_GJ);
  const bool across = ok && gj && (Fnew < 0.0) != (L.c.sig < 0.0);
  const bool out = ok && rnew2 >= p.r_out * p.r_out;
  // continuous extension, own component (and the position's, in FP32)
  double r2c = 0.0, r3c = 0.0, r4c = 0.0, r5c = 0.0;
  float yx[3], r2x[3], r3x[3], r4x[3], r5x[3];
  if ((across && !L.switching) || out) {
    r2c = yn - y;
    r3c = h * K1 - r2c;
    r4c = r2c - h * K7 - r3c;
    r5c = h * (DP::d1 * K1 + DP::d3 * K3 + DP::d4 * K4 + DP::d5 * K5 + DP::d6 * K6 + DP::d7 * K7);
    gather3(gm, base, r2c, r2x);
    gather3(gm, base, r3c, r3x);
    gather3(gm, base, r4c, r4x);
    gather3(gm, base, r5c, r5x);
    gather3(gm, base, y, yx);
  }
  if (across && !L.switching) {
    // root of the side function along the continuous extension, as advance()
    const double sgn = L.c.sig;
    auto side_val = [&](double th) {
      double xd[3];
      gather3d(gm, base, y + th * (r2c + (1.0 - th) * (r3c + th * (r4c + (1.0 - th) * r5c))), xd);
      const double mx = L.c.m0 * xd[0] + L.c.m1 * xd[1] + L.c.m2 * xd[2];
      const double rr = xd[0] * xd[0] + xd[1] * xd[1] + xd[2] * xd[2];
      return sgn * (3.0 * xd[2] * mx - L.c.m2 * rr);
    };
    double flo = side_val(0.0), fhi = side_val(1.0);
    ConeModel32 m32;
    m32.init(narrow(sgn), narrow(sgn * flo), narrow(L.c.m0), narrow(L.c.m1), narrow(L.c.m2), yx,
             r2x, r3x, r4x, r5x);
    if (!(flo >= 0.0)) flo = 0.0;
    if (!(fhi < 0.0)) fhi = -1e-300;
    const double lo = event_root(side_val, m32, flo, fhi);
    ++L.nr;
    if (lo < SWITCH_MIN_FRACTION) {
      flip_side(f, L);
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
    if (out) {
      // |x(th)| = r_out on the continuous extension, as advance()
      const double ro2 = p.r_out * p.r_out;
      auto inside = [&](double th) {
        double xd[3];
        gather3d(gm, base, y + th * (r2c + (1.0 - th) * (r3c + th * (r4c + (1.0 - th) * r5c))),
                xd);
        return ro2 - (xd[0] * xd[0] + xd[1] * xd[1] + xd[2] * xd[2]);
      };
      double flo = ro2 - L.r2;
      if (!(flo >= 0.0)) flo = 0.0;
      double fhi = ro2 - rnew2;
      if (!(fhi < 0.0)) fhi = -1e-300;
      EscapeModel32 e32;
      e32.init(narrow(flo), yx, r2x, r3x, r4x, r5x);
      const double th = event_root(inside, e32, flo, fhi);
      L.yc = y + th * (r2c + (1.0 - th) * (r3c + th * (r4c + (1.0 - th) * r5c)));
      L.lam += th * h;
      return RAY_ESCAPED;
    }
    L.yc = yn;
    L.f0c = K7;
    L.r2 = rnew2;
    L.lam += h;
    if (rnew2 <= p.r_capture * p.r_capture) return RAY_CAPTURED;
    if (clipped) return RAY_LAMBDA_END;
    if (across) {
      flip_side(f, L);
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

// shared doubles of four warps
constexpr int GROUP_SLOTS = 4 * GROUPS_PER_WARP * SLOTS;

// Counts of one warp's finished rays (lane c == 0 of each group holds its own).
struct GroupCounts {
  long long acc = 0, rej = 0, traced = 0, esc = 0;
};

// Where a warp's groups get their rays: records lo + e of recs (PARKREC doubles each:
// y[6], h, h_resume, sig, flags, na, nr, ray, lambda), e = 0, 1, ... claimed with an
// atomic on *next, while lo + e < hi.
struct ParkedRays {
  const double* recs;
  unsigned long long lo, hi;
  unsigned long long* next;
  // before a free group takes one, every lane of the warp (wants: the lane's group is
  // free; busy: it holds a ray)
  __device__ __forceinline__ void poll(const TraceParams&, bool, bool) {}
  // the lanes of a free group: its next record, or NULL (*done: no more will come)
  __device__ __forceinline__ const double* take(const TraceParams&, const GroupFile& f, int base,
                                                bool* done) {
    unsigned long long e = 0;
    if (f.cc == 0) e = lo + atomicAdd(next, 1ull);
    e = __shfl_sync(f.gm, e, base);
    *done = e >= hi;
    return *done ? nullptr : recs + e * PARKREC;
  }
};

// The marked guided rays of a launch (rt_guided.cuh), from their start.
struct FreshRays {
  GuidedScan scan;
  int64_t ray = -1;
  __device__ __forceinline__ void poll(const TraceParams& p, bool wants, bool busy) {
    const int lane = threadIdx.x & 31;
    const unsigned w = __ballot_sync(0xffffffffu, wants && lane % GROUP == 0);
    const unsigned b = __ballot_sync(0xffffffffu, busy);
    ray = -1;
    if (!scan.more(p, b != 0)) return;
    ray = scan.nth(__popc(w & ((1u << (lane - lane % GROUP)) - 1u)));
    scan.drop(__popc(w));
  }
  __device__ __forceinline__ const double* take(const TraceParams& p, const GroupFile& f, int,
                                                bool* done) {
    *done = ray < 0 && !scan.open && scan.found == 0;
    if (ray < 0) return nullptr;
    double* pe = f.s + S_P1;              // the passes' slots are free between rays
    __syncwarp(f.gm);
    if (f.cc == 0) fresh_record(p, ray, pe);
    __syncwarp(f.gm);
    return pe;
  }
};

// Six-lane groups of the calling warp continue the rays of src.  ngroups (1 to
// GROUPS_PER_WARP) groups of the warp take part: one group per warp keeps a ray's
// attempts free of the other groups' divergent branches.  slots: shared memory of the
// block, GROUP_SLOTS doubles for every four warps.  Every lane of the warp must call it.
template <class Source>
__device__ void tail_groups(const TraceParams& p, Source& src, int ngroups, GroupCounts& cnt,
                            double* slots) {
  const int lane = threadIdx.x & 31;
  const int g = lane / GROUP, cc = lane % GROUP;
  const bool in_group = g < ngroups && g < GROUPS_PER_WARP;
  const int base = g * GROUP;
  const unsigned gm = in_group ? (0x3Fu << base) : 0u;
  GLane L;
  GroupFile f;
  if (in_group) file_init(f, slots + ((threadIdx.x >> 5) * GROUPS_PER_WARP + g) * SLOTS, cc, gm);
  bool have = false, done = !in_group;
  int na0 = 0, nr0 = 0;
  for (;;) {
    const bool wants = in_group && !have && !done;
    if (__ballot_sync(0xffffffffu, wants)) {
      src.poll(p, wants, have);
      if (wants) {
        const double* pe = src.take(p, f, base, &done);
        if (pe) {
          L.yc = pe[cc];
          L.h = pe[6];
          L.h_resume = pe[7];
          const double sig = pe[8];
          const int fl = (int)pe[9];
          L.last_rej = (fl & 1) != 0;
          L.switching = (fl & 2) != 0;
          L.na = (int)pe[10];
          L.nr = (int)pe[11];
          L.ray = (int64_t)pe[12];
          L.lam = pe[13];
          L.star = find_star(p, L.ray);
          const StarDev& s = p.stars[L.star];
          const double om = 1.0 + p.state[6 * p.n + L.ray];
          double sp, cpsi;
          sincos(p.state[7 * p.n + L.ray], &sp, &cpsi);
          L.c.rs = s.rs_prop;
          L.c.cp = s.cp;
          L.c.pa = s.plasma_a;
          L.c.W2 = om * om;
          L.c.iW2 = 1.0 / (om * om);
          L.c.m0 = s.sin_tm * cpsi;
          L.c.m1 = s.sin_tm * sp;
          L.c.m2 = s.cos_tm;
          L.c.disp = s.dispersion;
          L.c.plasma = s.plasma;
          L.c.sig = sig;
          file_ray(f, L.c);
          double F;
          L.f0c = rhs_group(f, L.c, L.yc, &L.r2, &F);
          na0 = L.na;
          nr0 = L.nr;
          have = true;
        }
      }
      if (__ballot_sync(0xffffffffu, in_group && !done) == 0) break;
    }
    if (have) {
      const int st = advance_group(p, f, L, cc, gm, base);
      if (st >= 0) {
        const StarDev& s = p.stars[L.star];
        const int64_t n = p.n;
        p.state[cc * n + L.ray] = (cc < 3) ? L.yc * s.R_km : L.yc * s.ma_eV;
        __syncwarp(gm);                 // the group's state writes before its status
        if (cc == 0) {
          status_after_state(p, L.ray, st);
          if (p.nacc) p.nacc[L.ray] = L.na;
          if (p.nrej) p.nrej[L.ray] = L.nr;
          if (p.ts) atomicMax(p.ts + 1 + L.star, global_ns());
          cnt.acc += L.na - na0;
          cnt.rej += L.nr - nr0;
          cnt.traced += 1;
          cnt.esc += (st == RAY_ESCAPED);
        }
        have = false;
      }
    }
  }
}

// Express SMs for K records: XRAYS_PER_SM per SM, at most an eighth of the
// device's SM identifiers.
__device__ __forceinline__ unsigned long long express_sms(unsigned long long K) {
  int nsm = 1;
  asm("mov.u32 %0, %%nsmid;" : "=r"(nsm));
  unsigned long long xs = (K + XRAYS_PER_SM - 1) / XRAYS_PER_SM;
  const unsigned long long cap = (unsigned long long)(nsm / 8 > 0 ? nsm / 8 : 1);
  return xs < cap ? xs : cap;
}

// The express records' split: the first S (two per express SM) are continued
// one group per warp, the rest (S to K) five groups per warp.
__device__ __forceinline__ unsigned long long express_solo(unsigned long long K) {
  const unsigned long long S = 2 * express_sms(K);
  return S < K ? S : K;
}

}  // namespace
}  // namespace rtk
