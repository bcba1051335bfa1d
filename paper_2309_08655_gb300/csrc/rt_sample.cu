// Sampling kernel: one thread per sample, FP64 (see rt_sample_core.cuh), the
// samples of up to SAMPLE_STARS consecutive stars in one launch.
//
// Bound by the FP64 pipe: a warp instruction takes its sub-partition 64 cycles
// whatever the number of live lanes, so the per-sample computation keeps the
// lanes of a warp on one path (the inverse distribution from a table, the root
// in two FP64 evaluations).  16 x 65536 samples of a mass scan: 1.60 ms, of which
// half goes to the samples next to the null cone, where iterating all of them to
// the last bit, one launch per star, took 28.5 ms at 5 of 32 live lanes; 4096
// samples: 279 us against 709 us.
#include <cuda_runtime.h>
#include <stdint.h>

#include "rt_device.cuh"
#include "rt_internal.h"
#include "rt_sample_core.cuh"

namespace rtk {

namespace {

using namespace sampling;

__device__ __forceinline__ SampConst<double> sample_const(const StarDev& s) {
  SampConst<double> c;
  c.rs = s.rs;
  c.cp = s.cp;
  c.sin_tm = s.sin_tm;
  c.cos_tm = s.cos_tm;
  c.B0_eV2 = s.B0_eV2;
  c.R_eV = s.R_eV;
  c.n_inf = s.n_inf;
  c.ma_eV = s.ma_eV;
  c.v0 = s.v0;
  c.psi_fixed = s.psi_fixed;
  c.plasma_a = s.plasma_a;
  c.rlc = s.rlc;
  c.g_eV = s.g_eV;
  c.w_unit = s.w_unit;
  c.disp = s.dispersion;
  c.plasma = s.plasma;
  c.fa_model = s.fa_model;
  c.phase_mode = s.phase_mode;
  c.weight_mode = s.weight_mode;
  c.per_cm3 = PER_CM3_EV3;
  return c;
}

__device__ __forceinline__ int star_of_sample(const SampleParams& p, int64_t i) {
  int star = 0;                                  // begin[star] <= i < begin[star + 1]
  for (int hi = p.nstars - 1; star < hi;) {
    const int mid = (star + hi + 1) >> 1;
    if (p.begin[mid] <= i) star = mid; else hi = mid - 1;
  }
  return star;
}

__device__ __forceinline__ void store_state(const SampleParams& p, const StarDev& s, int64_t i,
                                            const SampOut<double>& o) {
  const int64_t ld = p.ld;
  p.state[6 * ld + i] = o.delta;
  p.state[7 * ld + i] = o.psi;
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    p.state[j * ld + i] = o.ok ? o.x[j] * s.R_km : 0.0;
    p.state[(3 + j) * ld + i] = o.ok ? o.k[j] * s.ma_eV : 0.0;
  }
  p.status[i] = o.ok ? RAY_READY : RAY_NO_ROOT;
}

// The samples next to the null cone (0.7 % of a Goldreich-Julian star's) are
// listed by their block and sampled once more by sample_state_iterated, a full
// block of them at a time: scattered over the warps, their iterations would hold
// every warp for a lane or two.
constexpr int SAMPLE_BLOCK = 128;
constexpr int LISTED = 2 * SAMPLE_BLOCK;

__global__ void __launch_bounds__(SAMPLE_BLOCK) sample_kernel(const SampleParams p) {
  __shared__ int64_t listed[LISTED];
  __shared__ int nlisted;
  if (threadIdx.x == 0) nlisted = 0;
  __syncthreads();
  const int64_t n = p.begin[p.nstars], ld = p.ld;
  for (int64_t base = blockIdx.x * (int64_t)SAMPLE_BLOCK;; base += (int64_t)gridDim.x * SAMPLE_BLOCK) {
    const int64_t i = base + threadIdx.x;
    if (i < n) {
      const int star = star_of_sample(p, i);
      const StarDev& s = p.stars[star];
      const SampConst<double> c = sample_const(s);
      double u[6];
#pragma unroll
      for (int j = 0; j < 6; ++j) u[j] = p.u[j * ld + i];
      SampOut<double> o;
      sample_core(c, u, (double)p.norm[star], o);
      store_state(p, s, i, o);
      p.weight[i] = o.ok ? o.w : 0.0;
      if (o.ok && next_to_null_cone(c, o.x, o.psi)) listed[atomicAdd(&nlisted, 1)] = i;
    }
    // (base is the block's: every thread leaves the loop in the same pass)
    const bool last = base + (int64_t)gridDim.x * SAMPLE_BLOCK >= n;
    __syncthreads();
    const int m = nlisted;
    __syncthreads();
    if (m < SAMPLE_BLOCK && !last) continue;     // at most LISTED - SAMPLE_BLOCK remain
    // entry j to warp j mod 4: a few entries take a warp each, on four schedulers
    constexpr int WARPS = SAMPLE_BLOCK / 32;
    for (int j = (threadIdx.x & 31) * WARPS + (threadIdx.x >> 5); j < m; j += SAMPLE_BLOCK) {
      const int64_t q = listed[j];
      const StarDev& s = p.stars[star_of_sample(p, q)];
      const SampConst<double> c = sample_const(s);
      double u[6];
#pragma unroll
      for (int k = 0; k < 6; ++k) u[k] = p.u[k * ld + q];
      SampOut<double> o;
      sample_state_iterated(c, u, o);
      store_state(p, s, q, o);
      if (!o.ok) p.weight[q] = 0.0;
    }
    if (last) break;
    __syncthreads();
    if (threadIdx.x == 0) nlisted = 0;
    __syncthreads();
  }
}

}  // namespace

cudaError_t launch_sample(const SampleParams& p, cudaStream_t stream) {
  const int64_t n = p.begin[p.nstars];
  if (n <= 0) return cudaSuccess;
  int dev = 0, nsm = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  // resident blocks only, so that each gathers enough samples next to the cone
  // to fill its warps with them
  int occ = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, sample_kernel, SAMPLE_BLOCK, 0);
  if (e != cudaSuccess) return e;
  int64_t grid = (n + SAMPLE_BLOCK - 1) / SAMPLE_BLOCK;
  const int64_t cap = (int64_t)nsm * (occ > 0 ? occ : 1);
  if (grid > cap) grid = cap;
  sample_kernel<<<(unsigned)grid, SAMPLE_BLOCK, 0, stream>>>(p);
  return cudaGetLastError();
}

}  // namespace rtk
