// Guided rays first, in warps of their own (the kernels of the double-float path
// and of the rotating magnetosphere).
//
// A ray that starts within 1e-3 rad of the null cone can cross it for 10^4 - 10^5
// attempts, and a launch lasts as long as its longest ray.  Among 31 other lanes
// every attempt of that ray also costs their crossings, escapes and refills.  So
// the rays that start nearest the cone are listed before the launch
// (launch_guided), nearest first, and the first warp of every block starts with
// its share of the list and claims nothing else until those rays have ended.  A
// ray's arithmetic does not depend on the lanes beside it: the rotating results are
// those of the plain queue, bit for bit; the double-float kernel hands its share to
// FP64 groups, which agree to its rounding.
//
// Not in the mixed kernel: there a second place that loads a ray made the compiler
// contract other multiply-adds of the FP32 start (5 % of the rays took another step
// sequence), for 117 ms against 125 on 16 x 65536 rays.
#pragma once
#include "rt_internal.h"

namespace rtk {
namespace {

// The calling warp's share of the guided rays: `mine` rays, the lane's being
// list entry first + lane * stride.
struct GuidedShare {
  const unsigned long long* list;
  unsigned long long first, stride;
  int mine;
};

__device__ __forceinline__ GuidedShare guided_share(const TraceParams& p) {
  GuidedShare g = {nullptr, 0, 1, 0};
  if (!p.guided) return g;
  unsigned long long K = *p.guided;
  if (K > (unsigned long long)GUIDED_CAP) K = (unsigned long long)GUIDED_CAP;
  if (K > (unsigned long long)p.guided_max) K = (unsigned long long)p.guided_max;
  if (K == 0) return g;
  g.list = p.guided + 32 + 2 * GUIDED_CAP;
  // a quarter of the launch's warps at most (guided_max is 32 rays for each): the
  // first warp of each block, then the second ones
  const unsigned long long most = (unsigned long long)p.guided_max / 32;
  g.stride = K < most ? K : most;
  g.first = (unsigned long long)(threadIdx.x >> 5) * gridDim.x + blockIdx.x;
  if (g.first >= g.stride) return g;
  g.mine = (int)((K - g.first + g.stride - 1) / g.stride);   // at most 32
  return g;
}

}  // namespace
}  // namespace rtk
