// Guided rays first, in warps of their own (the kernels of the double-float path
// and of the rotating magnetosphere).
//
// A ray that starts within 1e-3 rad of the null cone can cross it for 10^4 - 10^5
// attempts, and a launch lasts as long as its longest ray.  Among 31 other lanes
// every attempt of that ray also costs their crossings, escapes and refills.  So
// these rays leave the plain queue before the launch (launch_guided: status
// RAY_EXPRESS within 1e-4 rad, RAY_GUIDED beyond, their number beside the queue's
// counter), and a quarter of the launch's warps, the first of each block, look for
// them in the statuses, the nearest first, and trace nothing else until none is left
// (half of the warps, or a warp to itself for each of the nearest, changed nothing
// beyond noise).  A ray is marked for where it starts and for nothing else, so the
// rays beside it, the launch's shape and their number do not change a result: the
// rotating kernel's are those of the plain queue, bit for bit, and the double-float
// kernel traces every marked ray in FP64 groups.
//
// Not in the mixed kernel: there a second place that loads a ray made the compiler
// contract other multiply-adds of the FP32 start (5 % of the rays took another step
// sequence), for 117 ms against 125 on 16 x 65536 rays.
#pragma once
#include "rt_internal.h"

namespace rtk {
namespace {

// Guided rays that the calling warp traces at a time; 0: it takes none.
__device__ __forceinline__ int guided_quota(const TraceParams& p) {
  const unsigned long long K = p.queue[QUEUE_GUIDED];
  if (K == 0) return 0;
  const unsigned long long warps = (unsigned long long)gridDim.x * (blockDim.x >> 5);
  const unsigned long long most = warps / 4 > 0 ? warps / 4 : 1, takers = K < most ? K : most;
  // the first warp of each block, then the second ones
  if ((unsigned long long)(threadIdx.x >> 5) * gridDim.x + blockIdx.x >= takers) return 0;
  const unsigned long long q = (K + takers - 1) / takers;
  return q < 32 ? (int)q : 32;
}

// A warp's search for marked rays: the statuses in chunks of 32, claimed from the
// counter beside the queue's, once for each mark.  Every lane of the warp calls the
// members together.
struct GuidedScan {
  int64_t base = 0;        // the chunk
  unsigned found = 0;      // its marked rays not yet taken
  bool open = true;        // chunks are left

  // Claims chunks until one has a marked ray or, with `once`, one chunk.  false:
  // none found.
  __device__ __forceinline__ bool more(const TraceParams& p, bool once) {
    const int lane = threadIdx.x & 31;
    while (found == 0 && open) {
      unsigned long long b = 0;
      if (lane == 0) b = atomicAdd(p.queue + QUEUE_SCAN, 32ull);
      const int64_t at = (int64_t)__shfl_sync(0xffffffffu, b, 0), pass = (p.n + 31) & ~31ll;
      open = at < 2 * pass;
      base = at < pass ? at : at - pass;
      const int want = at < pass ? RAY_EXPRESS : RAY_GUIDED;
      const bool hit = open && base + lane < p.n && p.status[base + lane] == want;
      found = __ballot_sync(0xffffffffu, hit);
      if (once) break;
    }
    return found != 0;
  }
  // The chunk's k-th marked ray, or -1.
  __device__ __forceinline__ int64_t nth(int k) const {
    return k < __popc(found) ? base + (int)__fns(found, 0, k + 1) : -1;
  }
  // The first k of them are taken.
  __device__ __forceinline__ void drop(int k) {
    for (; k > 0 && found; --k) found &= found - 1u;
  }
};

}  // namespace
}  // namespace rtk
