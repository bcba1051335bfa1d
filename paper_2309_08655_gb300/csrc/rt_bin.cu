// Binning of escaped rays on the sky and in frequency (Sec. 2.2: the power
// reaching a bin of the sphere at infinity is the sum of the weights of the
// rays that land in it).  Sums are kept in 64-bit fixed point, so the result
// does not depend on the order of the atomics:
//   1. max_kernel      largest escaped weight (atomicMax on the bit pattern,
//                      which orders like the value for non-negative doubles);
//   2. accum_kernel    q = rint(w * 2^e) added to the 3-D histogram (global
//                      atomics) and, where a caller wants them, to the spectrum
//                      (shared memory, flushed once per block) and the sky map
//                      (global atomics); 2^e is the largest power of two with
//                      n * wmax * 2^e < 2^62;
//   3. finalize_kernel q / 2^e to float64, one warp per sky cell (or part of its
//                      row), which sums the row for the sky map (integer sums: the
//                      same whether the rays or the bins are added).
// n in the bound is BinParams::n_scale: the rays of this call, or of all shards
// of a sharded binning (rt_bin_part_*), whose int64 sums add exactly.
//
// What bounds it: the rays' 64 B each come from HBM or L2 in ~10 us for 2^20
// rays; FP64 arithmetic would take longer (acos, atan2, two roots and four
// divisions are ~200 FP64 instructions of 64 cycles a warp).  A ray's bin is
// therefore found in FP32, and in FP64 only where an FP32 value lies within
// its error of a bin's edge (below 1 ray in 1000), so that every ray lands in
// the bin that the FP64 values choose.  2^20 rays, 42 % escaped, 64 x 32 x 128
// bins with sky map and spectrum: 53 us, where FP64 for every ray, 64-bit shared
// atomics and six divisions in each thread took 393 us.
#include <cuda_runtime.h>
#include <stdint.h>
#include <stdio.h>

#include <cmath>
#include <mutex>

#include "rt.h"
#include "rt_device.cuh"
#include "rt_internal.h"

namespace rtk {

namespace {

constexpr int SMEM_SPEC_MAX = 1024;   // int64 entries of the shared spectrum

// 2^e of the fixed point and its inverse, from the exponent's bits (ldexp and
// ilogb where a factor would not be a normal number).
__device__ __forceinline__ int fixed_exponent(long long wmax_bits, int64_t n) {
  const double bound = __longlong_as_double(wmax_bits) * (double)(n > 0 ? n : 1);
  const int b = (__double2hiint(bound) >> 20) & 0x7ff;
  return 61 - ((b > 0 && b < 0x7ff) ? b - 1023 : ilogb(bound));
}
__device__ __forceinline__ double power_of_two(int e) {
  return (e >= -1022 && e <= 1023) ? __hiloint2double((e + 1023) << 20, 0) : ldexp(1.0, e);
}
__device__ __forceinline__ double fixed_scale(long long wmax_bits, int64_t n) {
  return wmax_bits > 0 ? power_of_two(fixed_exponent(wmax_bits, n)) : 1.0;
}
__device__ __forceinline__ double fixed_unit(long long wmax_bits, int64_t n) {
  if (!(wmax_bits > 0)) return 1.0;
  const int e = fixed_exponent(wmax_bits, n);
  return (e >= -1022 && e <= 1022) ? power_of_two(-e) : 1.0 / power_of_two(e);
}

__global__ void max_kernel(BinParams p) {
  constexpr long long INF = 0x7ff0000000000000ll;
  const int64_t step = (int64_t)gridDim.x * blockDim.x;
  long long best = 0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < p.n; i += 4 * step) {
    // four independent rays a round: the loads' latency is what this pass costs
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int64_t j = i + k * step;
      if (j >= p.n) break;
      const long long b = ((const long long*)p.weight)[j];
      if (p.status[j] == RAY_ESCAPED && b > best && b <= INF) best = b;   // no NaN
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const long long v = __shfl_down_sync(0xffffffffu, best, o);
    best = v > best ? v : best;
  }
  if ((threadIdx.x & 31) == 0 && best > 0) atomicMax(&p.acc[0], best);
}

// A double's leading 24 bits as a float by its bits (a conversion instruction
// would issue on the FP64 pipe); below the normal floats 0; *ok cleared for
// values beyond 2^126 and non-finite ones.
__device__ __forceinline__ float lead_float(double v, bool* ok) {
  const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
  const unsigned e = (hi >> 20) & 0x7ffu;
  if (e > 1149u) *ok = false;
  if (e < 898u) return 0.0f;
  return __uint_as_float((hi & 0x80000000u) | (((hi & 0x7fffffffu) - (896u << 20)) << 3) |
                         (lo >> 29));
}

// Bin of an FP32 position f (in bins) that is off by at most m bins: -1 below
// the range, nbin above it, -2 where an edge is within m.
__device__ __forceinline__ int sure_bin(float f, float m, int nbin) {
  const float g = floorf(f), r = f - g;
  if (!(r >= m && r <= 1.0f - m)) return -2;       // also NaN
  if (g < 0.0f) return -1;
  return g >= (float)nbin ? nbin : (int)g;
}

struct Bins {
  double dth, dph, dnu, y_unit, iR;
  float ith32, iph32, inu32, iy32, lo32, rs32;     // inverse widths, in FP32
  float mth, mph, mnu;                             // FP32 errors in bins
};

// Bounds on the FP32 errors: the angles carry a dozen roundings of 2^-23
// (truncated inputs included), below 2e-6 rad -- for phi of the transverse
// part of the direction -- and the frequency four, below 5e-7 of |y| and
// |nu_lo|; the margins are four times that.
constexpr float ANGLE_MARGIN = 8e-6f, FREQ_MARGIN = 2e-6f;

// (on the host: six FP64 divisions in every thread took longer than the rays)
Bins bins_of(const BinParams& p) {
  Bins b;
  b.dth = PI / p.nth;
  b.dph = 2.0 * PI / p.nph;
  b.dnu = (p.nu_hi - p.nu_lo) / p.nnu;
  b.y_unit = 0.5 * p.v0 * p.v0;
  b.iR = 1.0 / p.R_km;
  b.ith32 = (float)p.nth * (float)(1.0 / PI);
  b.iph32 = (float)p.nph * (float)(0.5 / PI);
  b.inu32 = (float)(1.0 / b.dnu);
  b.iy32 = (float)(1.0 / b.y_unit);
  b.lo32 = (float)p.nu_lo;
  b.rs32 = (float)(p.rs_prop * p.R_km);
  b.mth = ANGLE_MARGIN * b.ith32;
  b.mph = ANGLE_MARGIN * b.iph32;
  b.mnu = FREQ_MARGIN * b.inu32;
  return b;
}

// The ray's bin from its FP64 state: frequency bin (-1: out of range) and sky cell.
__device__ __forceinline__ int exact_frequency(const BinParams& p, const Bins& b, int64_t i) {
  const double y = p.state[6 * p.ld + i] / b.y_unit;
  if (!(y >= p.nu_lo && y < p.nu_hi)) return -1;
  const int inu = (int)floor((y - p.nu_lo) / b.dnu);
  return inu >= p.nnu ? p.nnu - 1 : inu;
}
__device__ __forceinline__ int exact_sky(const BinParams& p, const Bins& b, int64_t i) {
  // direction of the orthonormal-frame momentum at the end point
  const int64_t ld = p.ld;
  const double x0 = p.state[i] * b.iR, x1 = p.state[ld + i] * b.iR;
  const double x2 = p.state[2 * ld + i] * b.iR;
  const double k0 = p.state[3 * ld + i], k1 = p.state[4 * ld + i], k2 = p.state[5 * ld + i];
  const double ir = rsqrt(x0 * x0 + x1 * x1 + x2 * x2);
  const double n0 = x0 * ir, n1 = x1 * ir, n2 = x2 * ir;
  const double A = 1.0 - p.rs_prop * ir;
  const double cr = (sqrt(A) - 1.0) * (n0 * k0 + n1 * k1 + n2 * k2);
  const double o0 = k0 + cr * n0, o1 = k1 + cr * n1, o2 = k2 + cr * n2;
  const double kmag = sqrt(o0 * o0 + o1 * o1 + o2 * o2);
  const double th = acos(fmax(-1.0, fmin(1.0, o2 / kmag)));
  double ph = atan2(o1, o0);
  if (ph < 0.0) ph += 2.0 * PI;
  int ith = (int)floor(th / b.dth);
  if (ith >= p.nth) ith = p.nth - 1;
  int iph = (int)floor(ph / b.dph);
  if (iph >= p.nph) iph -= p.nph;
  return ith * p.nph + iph;
}

// Sky cell in FP32, or -2 where an edge is too near or a value out of FP32's range.
__device__ __forceinline__ int sky32(const BinParams& p, const Bins& b, int64_t i) {
  bool ok = true;
  float x[3], k[3];
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    x[j] = lead_float(p.state[j * p.ld + i], &ok);
    k[j] = lead_float(p.state[(3 + j) * p.ld + i], &ok);
  }
  // momenta scaled by a power of two into FP32's middle: eV values can be tiny
  const float km = fmaxf(fabsf(k[0]), fmaxf(fabsf(k[1]), fabsf(k[2])));
  if (!(km > 0x1p-90f)) return -2;
  const float ks = __uint_as_float((254u << 23) - (__float_as_uint(km) & 0x7f800000u));
#pragma unroll
  for (int j = 0; j < 3; ++j) k[j] *= ks;
  const float r2 = x[0] * x[0] + x[1] * x[1] + x[2] * x[2];
  const float ir = rsqrtf(r2);
  const float A = 1.0f - b.rs32 * ir;
  if (!(ok && r2 > 0x1p-60f && r2 < 0x1p100f && A > 0x1p-4f)) return -2;
  const float n0 = x[0] * ir, n1 = x[1] * ir, n2 = x[2] * ir;
  const float cr = (sqrtf(A) - 1.0f) * (n0 * k[0] + n1 * k[1] + n2 * k[2]);
  const float o0 = k[0] + cr * n0, o1 = k[1] + cr * n1, o2 = k[2] + cr * n2;
  const float t2 = o0 * o0 + o1 * o1;
  const float it = rsqrtf(t2);                     // 1 / transverse part (k is O(1))
  const float rho = t2 * it;
  if (!(t2 > 1e-6f * (t2 + o2 * o2))) return -2;   // near a pole
  const int ith = sure_bin(atan2f(rho, o2) * b.ith32, b.mth, p.nth);
  float ph = atan2f(o1, o0);
  if (ph < 0.0f) ph += 6.2831853f;
  const int iph = sure_bin(ph * b.iph32, b.mph * sqrtf(t2 + o2 * o2) * it, p.nph);
  // a position outside the range is an edge's neighbour: FP64 decides
  if (ith < 0 || iph < 0 || ith >= p.nth || iph >= p.nph) return -2;
  return ith * p.nph + iph;
}

__device__ __forceinline__ int frequency32(const BinParams& p, const Bins& b, int64_t i) {
  bool ok = true;
  const float y = lead_float(p.state[6 * p.ld + i], &ok) * b.iy32;
  const int inu = sure_bin((y - b.lo32) * b.inu32,
                           b.mnu * (fabsf(y) + fabsf(b.lo32)) + 1e-6f * (float)p.nnu, p.nnu);
  if (!ok || inu == -2) return -2;
  return inu >= p.nnu ? -1 : inu;
}

// MARG: the sums of the sky map and the spectrum, too (a caller that reads them
// from p.acc); SPEC: the spectrum alone.
template <bool MARG, bool SPEC>
__global__ void __launch_bounds__(256) accum_kernel(BinParams p, Bins b) {
  // each entry in two 32-bit halves: a 64-bit add in shared memory is a
  // compare-and-swap loop, a 32-bit one an instruction
  __shared__ unsigned s_lo[SPEC ? SMEM_SPEC_MAX : 1], s_hi[SPEC ? SMEM_SPEC_MAX : 1];
  const int nsky = p.nth * p.nph;
  const bool spec_smem = SPEC && p.nnu <= SMEM_SPEC_MAX;
  if (spec_smem) {
    for (int j = threadIdx.x; j < p.nnu; j += blockDim.x) s_lo[j] = s_hi[j] = 0u;
    __syncthreads();
  }
  const double scale = fixed_scale(p.acc[0], p.n_scale);
  unsigned long long* g_hist = (unsigned long long*)p.acc + 2;
  unsigned long long* g_sky = g_hist + (size_t)nsky * p.nnu;
  unsigned long long* g_spec = g_sky + nsky;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < p.n;
       i += (int64_t)gridDim.x * blockDim.x) {
    if (p.status[i] != RAY_ESCAPED) continue;
    const unsigned long long q = (unsigned long long)llrint(p.weight[i] * scale);
    int isky = sky32(p, b, i);
    int inu = frequency32(p, b, i);
    if (inu == -2) inu = exact_frequency(p, b, i);
    if (inu < 0) {
      atomicAdd((unsigned long long*)&p.acc[1], q);
      continue;
    }
    if (isky == -2) isky = exact_sky(p, b, i);
    atomicAdd(&g_hist[(size_t)isky * p.nnu + inu], q);
    if (MARG) atomicAdd(&g_sky[isky], q);
    if (spec_smem) {
      const unsigned ql = (unsigned)q;
      const unsigned old = atomicAdd(&s_lo[inu], ql);
      const unsigned h = (unsigned)(q >> 32) + (old + ql < old ? 1u : 0u);
      if (h) atomicAdd(&s_hi[inu], h);
    } else if (SPEC) {
      atomicAdd(&g_spec[inu], q);
    }
  }
  if (spec_smem) {
    __syncthreads();
    for (int j = threadIdx.x; j < p.nnu; j += blockDim.x) {
      const unsigned long long v = ((unsigned long long)s_hi[j] << 32) | s_lo[j];
      if (v) atomicAdd(&g_spec[j], v);
    }
  }
}

// One warp per sky cell's row, whose sum is the sky map's entry, or, with SEG, per
// segment of it (segs segments of len bins): the parts' sums are then added to those
// behind the cube, for sky_kernel, unless the rays were (sum false).
template <bool SEG>
__global__ void __launch_bounds__(256) finalize_kernel(BinParams p, int segs, int len, bool sum) {
  const double inv = fixed_unit(p.acc[0], p.n_scale);
  const int nsky = p.nth * p.nph, nnu = p.nnu;
  const long long* g_hist = p.acc + 2;
  unsigned long long* g_sky = (unsigned long long*)p.acc + 2 + (int64_t)nsky * nnu;
  const long long* g_spec = (const long long*)g_sky + nsky;
  const int lane = threadIdx.x & 31;
  const int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t threads = (int64_t)gridDim.x * blockDim.x;
  const int64_t parts = SEG ? (int64_t)nsky * segs : nsky;
  for (int64_t g = tid >> 5; g < parts; g += threads >> 5) {
    const int64_t s = SEG ? g / segs : g;
    const int lo = SEG ? (int)(g - s * segs) * len : 0, hi = SEG ? min(lo + len, nnu) : nnu;
    const long long* row = g_hist + s * nnu;
    double* out = p.hist + s * nnu;
    long long q_sum = 0;
    for (int j = lo + lane; j < hi; j += 32) {
      const long long q = row[j];
      out[j] = (double)q * inv;
      q_sum += q;
    }
    if (p.sky && (!SEG || sum)) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) q_sum += __shfl_down_sync(0xffffffffu, q_sum, o);
      if (lane == 0 && !SEG) p.sky[s] = (double)q_sum * inv;
      if (lane == 0 && SEG) atomicAdd(g_sky + s, (unsigned long long)q_sum);
    }
  }
  if (p.spec)
    for (int64_t j = tid; j < nnu; j += threads) p.spec[j] = (double)g_spec[j] * inv;
  if (tid == 0) *p.oor = (double)p.acc[1] * inv;
}

__global__ void __launch_bounds__(256) sky_kernel(BinParams p) {
  const double inv = fixed_unit(p.acc[0], p.n_scale);
  const int64_t nsky = (int64_t)p.nth * p.nph;
  const long long* g_sky = p.acc + 2 + nsky * p.nnu;
  const int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (s < nsky) p.sky[s] = (double)g_sky[s] * inv;
}

}  // namespace

namespace {

cudaError_t sm_count(int* nsm) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  return cudaDeviceGetAttribute(nsm, cudaDevAttrMultiProcessorCount, dev);
}

constexpr int BIN_BLOCK = 256;

// Grid of the per-ray kernels: one thread per ray up to 8 blocks per SM.
unsigned ray_grid(int64_t n, int nsm) {
  int64_t grid = (n + BIN_BLOCK - 1) / BIN_BLOCK;
  if (grid > (int64_t)nsm * 8) grid = (int64_t)nsm * 8;
  return (unsigned)(grid < 1 ? 1 : grid);
}

template <bool MARG, bool SPEC>
cudaError_t launch_accum(const BinParams& p, cudaStream_t stream) {
  int nsm = 0;
  cudaError_t e = sm_count(&nsm);
  if (e != cudaSuccess) return e;
  accum_kernel<MARG, SPEC><<<ray_grid(p.n, nsm), BIN_BLOCK, 0, stream>>>(p, bins_of(p));
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_bin_max(const BinParams& p, cudaStream_t stream) {
  int nsm = 0;
  cudaError_t e = sm_count(&nsm);
  if (e != cudaSuccess) return e;
  const size_t entries = bin_scratch_entries(p.nth, p.nph, p.nnu);
  e = cudaMemsetAsync(p.acc, 0, entries * sizeof(long long), stream);
  if (e != cudaSuccess) return e;
  max_kernel<<<ray_grid((p.n + 3) / 4, nsm), BIN_BLOCK, 0, stream>>>(p);
  return cudaGetLastError();
}

cudaError_t launch_bin_accum(const BinParams& p, cudaStream_t stream) {
  return launch_accum<true, true>(p, stream);
}

namespace {

// marg: p.acc holds the sky map's sums already.
cudaError_t launch_finalize(const BinParams& p, bool marg, cudaStream_t stream) {
  int nsm = 0;
  cudaError_t e = sm_count(&nsm);
  if (e != cudaSuccess) return e;
  // One warp per row, or, with fewer rows than warps that the GPU holds, per segment of
  // at least 256 bins (a spectrum alone is one row: 2^22 bins in one warp took 60 ms,
  // shared out the whole call takes 87 us); at least enough threads for the spectrum's entries.
  const int64_t nsky = (int64_t)p.nth * p.nph, warps_held = (int64_t)nsm * 64;
  int64_t segs = nsky < warps_held ? warps_held / nsky : 1;
  if (segs > (p.nnu + 255) / 256) segs = (p.nnu + 255) / 256;
  const int len = (int)(((p.nnu + segs - 1) / segs + 31) / 32 * 32);
  segs = (p.nnu + len - 1) / len;
  int64_t warps = nsky * segs;
  if (p.spec && warps < (p.nnu + 31) / 32) warps = (p.nnu + 31) / 32;
  int64_t gf = (warps + BIN_BLOCK / 32 - 1) / (BIN_BLOCK / 32);
  if (gf > (int64_t)nsm * 8) gf = (int64_t)nsm * 8;
  if (segs == 1)
    finalize_kernel<false><<<(unsigned)gf, BIN_BLOCK, 0, stream>>>(p, 1, p.nnu, true);
  else
    finalize_kernel<true><<<(unsigned)gf, BIN_BLOCK, 0, stream>>>(p, (int)segs, len, !marg);
  e = cudaGetLastError();
  if (e != cudaSuccess || segs == 1 || !p.sky) return e;
  sky_kernel<<<(unsigned)((nsky + BIN_BLOCK - 1) / BIN_BLOCK), BIN_BLOCK, 0, stream>>>(p);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_bin_finalize(const BinParams& p, cudaStream_t stream) {
  return launch_finalize(p, true, stream);
}

cudaError_t launch_bin(const BinParams& p, cudaStream_t stream) {
  cudaError_t e = launch_bin_max(p, stream);
  if (e == cudaSuccess)
    e = p.spec ? launch_accum<false, true>(p, stream) : launch_accum<false, false>(p, stream);
  if (e == cudaSuccess) e = launch_finalize(p, false, stream);
  return e;
}

}  // namespace rtk

// ---------------------------------------------------------------------------
// Allocation-free variant of the binning entry point.
//
// Some callers may not allocate device memory from inside the library: code
// that runs under a device-memory budget managed by someone else (a
// framework's caching allocator, a fixed memory pool shared through MPS), or a
// real-time pipeline that cannot afford the device synchronisation that
// cudaMalloc / cudaFree may imply.  rt_bin_spectrum_noalloc serves them: its
// fixed-point accumulator is a file-scope __device__ array of a fixed maximum
// size that every GPU loading this library holds until exit, instead of the
// handle-owned scratch that rt_bin_spectrum allocates on first use.  It takes
// the star parameters by value (the three numbers binning needs), so it does
// not need an rt_star handle either; the kernels are those of rt_bin_spectrum.

namespace rtk {
namespace {

constexpr size_t NOALLOC_ENTRIES = (size_t)RT_BIN_NOALLOC_MAX_ENTRIES;  // 4 MiB of int64
static __device__ __align__(256) long long g_noalloc_acc[NOALLOC_ENTRIES];

// Device address of g_noalloc_acc, looked up once per device (with that
// device current) by the first call on it.  cudaDeviceReset destroys the
// context that this address belongs to (documented in rt.h).
constexpr int NOALLOC_MAX_DEVICES = 64;
std::mutex g_noalloc_mu;
long long* g_noalloc_ptr[NOALLOC_MAX_DEVICES] = {nullptr};

rt_status bin_fail(rt_status s, const char* msg) {
  set_last_error(msg);   // readable through rt_last_error()
  return s;
}

rt_status bin_cuda_fail(cudaError_t e) {
  cudaGetLastError();    // clear a sticky launch error so that later calls do not see it
  return bin_fail(RT_ECUDA, cudaGetErrorString(e));
}

// Checks shared by the entry points of this file.
rt_status check_bins(int32_t nth, int32_t nph, int32_t nnu) {
  if (nth < 1 || nph < 1 || nnu < 1) return bin_fail(RT_EINVAL, "bin counts must be >= 1");
  if ((int64_t)nth * nph * nnu > (int64_t)1 << 28) return bin_fail(RT_EINVAL, "too many bins");
  return RT_OK;
}

rt_status check_rays(int64_t n, const double* d_state, const double* d_weight,
                     const uint8_t* d_status) {
  if (n <= 0) return RT_OK;
  rt_status st;
  if (d_state && (st = check_device_array(d_state, "d_state")) != RT_OK) return st;
  if ((st = check_device_array(d_weight, "d_weight")) != RT_OK) return st;
  if ((st = check_device_array(d_status, "d_status")) != RT_OK) return st;
  return RT_OK;
}

rt_status check_outputs(const double* d_hist, const double* d_sky, const double* d_spec,
                        const double* d_oor) {
  rt_status st;
  if ((st = check_device_array(d_hist, "d_hist")) != RT_OK) return st;
  if ((st = check_device_array(d_oor, "d_out_of_range")) != RT_OK) return st;
  if (d_sky && (st = check_device_array(d_sky, "d_sky")) != RT_OK) return st;
  if (d_spec && (st = check_device_array(d_spec, "d_spec")) != RT_OK) return st;
  return RT_OK;
}

}  // namespace
}  // namespace rtk

extern "C" rt_status rt_bin_spectrum_noalloc(const rt_star_params* params, int64_t n,
                                             const double* d_state, const double* d_weight,
                                             const uint8_t* d_status, int32_t nth, int32_t nph,
                                             int32_t nnu, double nu_lo, double nu_hi,
                                             double* d_hist, double* d_sky, double* d_spec,
                                             double* d_out_of_range, void* stream) {
  rtk::NvtxRange nvtx_range("rt_bin_spectrum_noalloc");
  using namespace rtk;
  rt_status st;
  if ((st = check_star_params(params)) != RT_OK) return st;
  if (n < 0) return bin_fail(RT_EINVAL, "n must be >= 0");
  if ((st = check_bins(nth, nph, nnu)) != RT_OK) return st;
  if (!(nu_hi > nu_lo) || !std::isfinite(nu_lo) || !std::isfinite(nu_hi))
    return bin_fail(RT_EINVAL, "need finite nu_lo < nu_hi");
  const size_t need = bin_scratch_entries(nth, nph, nnu);
  if (need > NOALLOC_ENTRIES)
    return bin_fail(RT_EINVAL,
                    "histogram too large for the static accumulator: need 2 + nth*nph*nnu + "
                    "nth*nph + nnu <= RT_BIN_NOALLOC_MAX_ENTRIES (524288)");
  if (n > 0 && !d_state) return bin_fail(RT_EINVAL, "d_state is NULL");
  if ((st = check_rays(n, d_state, d_weight, d_status)) != RT_OK) return st;
  if ((st = check_outputs(d_hist, d_sky, d_spec, d_out_of_range)) != RT_OK) return st;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return bin_cuda_fail(e);
  if (dev < 0 || dev >= NOALLOC_MAX_DEVICES) return bin_fail(RT_EINVAL, "device index too large");
  long long* acc;
  {
    std::lock_guard<std::mutex> lock(g_noalloc_mu);
    if (!g_noalloc_ptr[dev]) {
      void* ptr = nullptr;
      e = cudaGetSymbolAddress(&ptr, g_noalloc_acc);
      if (e != cudaSuccess || ptr == nullptr) {
        cudaGetLastError();
        return bin_fail(RT_ECUDA, "cudaGetSymbolAddress of the static accumulator failed");
      }
      g_noalloc_ptr[dev] = (long long*)ptr;
    }
    acc = g_noalloc_ptr[dev];
  }
  BinParams p;
  p.R_km = params->R_km;
  const double rs = 2.0 * params->M_sun * 1.4766250 / params->R_km;
  p.rs_prop = (params->prop_metric == RT_METRIC_FLAT) ? 0.0 : rs;
  p.v0 = params->v0_kms / 299792.458;
  p.n = n;
  p.ld = n;
  p.n_scale = n;
  p.state = d_state;
  p.weight = d_weight;
  p.status = d_status;
  p.nth = nth;
  p.nph = nph;
  p.nnu = nnu;
  p.nu_lo = nu_lo;
  p.nu_hi = nu_hi;
  p.acc = acc;        // launch_bin clears the part of it this call uses
  p.hist = d_hist;
  p.sky = d_sky;
  p.spec = d_spec;
  p.oor = d_out_of_range;
  e = launch_bin(p, (cudaStream_t)stream);
  if (e != cudaSuccess) return bin_cuda_fail(e);
  return RT_OK;
}

// ---------------------------------------------------------------------------
// Sharded binning: the three phases of rt_bin_spectrum around caller-owned
// int64 sums, reduced exactly between the phases by the caller (one process
// per GPU, each with a contiguous range of one workload's rays).

namespace {

rtk::BinParams part_params(int64_t n, int64_t n_total, const double* d_state,
                           const double* d_weight, const uint8_t* d_status, int32_t nth,
                           int32_t nph, int32_t nnu, double nu_lo, double nu_hi, int64_t* d_acc) {
  rtk::BinParams p;
  p.R_km = 1.0;
  p.rs_prop = 0.0;
  p.v0 = 1.0;
  p.n = n;
  p.ld = n;
  p.n_scale = n_total;
  p.state = d_state;
  p.weight = d_weight;
  p.status = d_status;
  p.nth = nth;
  p.nph = nph;
  p.nnu = nnu;
  p.nu_lo = nu_lo;
  p.nu_hi = nu_hi;
  p.acc = (long long*)d_acc;
  p.hist = p.sky = p.spec = p.oor = nullptr;
  return p;
}

}  // namespace

extern "C" rt_status rt_bin_part_max(int64_t n, const double* d_weight, const uint8_t* d_status,
                                     int32_t nth, int32_t nph, int32_t nnu, int64_t* d_acc,
                                     void* stream) {
  rtk::NvtxRange nvtx_range("rt_bin_part_max");
  using namespace rtk;
  rt_status st;
  if (n < 0) return bin_fail(RT_EINVAL, "n must be >= 0");
  if ((st = check_bins(nth, nph, nnu)) != RT_OK) return st;
  if ((st = check_rays(n, nullptr, d_weight, d_status)) != RT_OK) return st;
  if ((st = check_device_array(d_acc, "d_acc")) != RT_OK) return st;
  const BinParams p =
      part_params(n, n, nullptr, d_weight, d_status, nth, nph, nnu, 0.0, 1.0, d_acc);
  const cudaError_t e = launch_bin_max(p, (cudaStream_t)stream);
  if (e != cudaSuccess) return bin_cuda_fail(e);
  return RT_OK;
}

extern "C" rt_status rt_bin_part_accumulate(const rt_star* star, int64_t n, int64_t ld,
                                            int64_t n_total, const double* d_state,
                                            const double* d_weight,
                                            const uint8_t* d_status, int32_t nth, int32_t nph,
                                            int32_t nnu, double nu_lo, double nu_hi,
                                            int64_t* d_acc, void* stream) {
  rtk::NvtxRange nvtx_range("rt_bin_part_accumulate");
  using namespace rtk;
  rt_status st;
  if (!star) return bin_fail(RT_EINVAL, "star is NULL");
  if (n < 0 || n_total < n) return bin_fail(RT_EINVAL, "need 0 <= n <= n_total");
  if (ld < n) return bin_fail(RT_EINVAL, "need ld >= n");
  if ((st = check_bins(nth, nph, nnu)) != RT_OK) return st;
  if (!(nu_hi > nu_lo) || !std::isfinite(nu_lo) || !std::isfinite(nu_hi))
    return bin_fail(RT_EINVAL, "need finite nu_lo < nu_hi");
  if (n > 0 && !d_state) return bin_fail(RT_EINVAL, "d_state is NULL");
  if ((st = check_rays(n, d_state, d_weight, d_status)) != RT_OK) return st;
  if ((st = check_device_array(d_acc, "d_acc")) != RT_OK) return st;
  BinParams p =
      part_params(n, n_total, d_state, d_weight, d_status, nth, nph, nnu, nu_lo, nu_hi, d_acc);
  const StarDev& h = star_host_desc(star);
  p.ld = ld;
  p.R_km = h.R_km;
  p.rs_prop = h.rs_prop;
  p.v0 = h.v0;
  const cudaError_t e = launch_bin_accum(p, (cudaStream_t)stream);
  if (e != cudaSuccess) return bin_cuda_fail(e);
  return RT_OK;
}

extern "C" rt_status rt_bin_part_finalize(int32_t nth, int32_t nph, int32_t nnu, int64_t n_total,
                                          const int64_t* d_acc, double* d_hist, double* d_sky,
                                          double* d_spec, double* d_out_of_range, void* stream) {
  rtk::NvtxRange nvtx_range("rt_bin_part_finalize");
  using namespace rtk;
  rt_status st;
  if (n_total < 0) return bin_fail(RT_EINVAL, "n_total must be >= 0");
  if ((st = check_bins(nth, nph, nnu)) != RT_OK) return st;
  if ((st = check_device_array(d_acc, "d_acc")) != RT_OK) return st;
  if ((st = check_outputs(d_hist, d_sky, d_spec, d_out_of_range)) != RT_OK) return st;
  BinParams p = part_params(0, n_total, nullptr, nullptr, nullptr, nth, nph, nnu, 0.0, 1.0,
                            const_cast<int64_t*>(d_acc));
  p.hist = d_hist;
  p.sky = d_sky;
  p.spec = d_spec;
  p.oor = d_out_of_range;
  const cudaError_t e = launch_bin_finalize(p, (cudaStream_t)stream);
  if (e != cudaSuccess) return bin_cuda_fail(e);
  return RT_OK;
}
