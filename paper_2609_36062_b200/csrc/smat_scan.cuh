// Exclusive prefix (or suffix) sums of chunk states, in place: the body of the scan kernel, and of the CTAs of a routed read
// that scan beside it.
#pragma once
#include "smat_internal.h"

// A thread owns four consecutive state entries (number e4) of head bh and walks the chunks of its range in order; which: job
// and range.  Loads are issued sixteen chunks ahead of the dependent additions.
__device__ __forceinline__ void smat_scan_entries(const SmatScanArgs& a, int64_t state_elems, int64_t NC, int64_t e4, int64_t bh,
                                                  int which) {
  if (e4 * 4 >= state_elems) return;
  const SmatScanJob& job = a.job[which >> 1];
  const int range = which & 1, reverse = job.reverse;
  const int64_t lo = range ? job.lo1 : job.lo0, hi = range ? job.hi1 : job.hi0;
  float4* base = reinterpret_cast<float4*>(job.S + bh * NC * state_elems) + e4;
  const int64_t stride4 = state_elems / 4;
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
  constexpr int AHEAD = 16;
  for (int64_t s = 0; s < hi - lo; s += AHEAD) {
    float4 v[AHEAD];
#pragma unroll
    for (int u = 0; u < AHEAD; ++u) {
      const int64_t k = s + u;
      if (k < hi - lo) v[u] = base[(reverse ? hi - 1 - k : lo + k) * stride4];
    }
#pragma unroll
    for (int u = 0; u < AHEAD; ++u) {
      const int64_t k = s + u;
      if (k < hi - lo) {
        base[(reverse ? hi - 1 - k : lo + k) * stride4] = acc;
        acc.x += v[u].x; acc.y += v[u].y; acc.z += v[u].z; acc.w += v[u].w;
      }
    }
  }
}
