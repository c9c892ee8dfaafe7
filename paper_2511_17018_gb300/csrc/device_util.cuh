// Small device helpers shared by the kernel modules.
#pragma once

#ifndef __CUDACC_RTC__
#include <cuda_runtime.h>
#include <stdint.h>
#endif

namespace tpcfit {

// Cluster range [b, e) of track t; false, and an empty range, if its offsets are
// out of order or leave the cluster arrays.
__device__ __forceinline__ bool track_range(const int32_t* off, int64_t t, int64_t n_hits, int32_t& b, int32_t& e) {
  b = off[t];
  e = off[t + 1];
  if (b >= 0 && e >= b && (int64_t)e <= n_hits) return true;
  b = e = 0;
  return false;
}

// A recorded track's clusters and the steps of a pass over it, 0 if it has no fit.  The
// recording has the last word: of a track without a fit it holds no state and no
// cluster, whatever the caller's ndf (another fit's, say) makes of it.  The range is
// empty for the offsets that the fit refuses, so no cluster outside the arrays is
// touched.
struct RecordedTrack {
  int32_t begin = 0, end = 0, steps = 0;
};
__device__ __forceinline__ RecordedTrack recorded_track(const int32_t* off, int64_t n_hits, const int32_t* ndf,
                                                        const int32_t* ck_last, int64_t t) {
  RecordedTrack r;
  track_range(off, t, n_hits, r.begin, r.end);
  r.steps = ndf[t] > 0 ? min(ck_last[t] + 1, r.end - r.begin) : 0;
  return r;
}

// Frame of track `trk`: f with base[f] <= trk < base[f + 1] (base[0] = 0,
// base[n_frames] = total tracks); -1 if trk lies outside the table.
__device__ __forceinline__ int frame_of(const int64_t* base, int n_frames, int64_t trk) {
  if (trk < __ldg(base) || trk >= __ldg(base + n_frames)) return -1;
  int lo = 0, hi = n_frames;  // invariant: base[lo] <= trk < base[hi]
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (__ldg(base + mid) <= trk) lo = mid;
    else hi = mid;
  }
  return lo;
}

// A cluster's row and sector by an ordinary load.  Not __ldg: the read-only path is
// for memory that nobody writes during the launch, and another stream may still be
// copying a frame in, next to the clusters read or, before its flag, the very ones.
__device__ __forceinline__ uint16_t load_rowsec(const uint16_t* p) {
  uint16_t v;
  asm volatile("ld.global.u16 %0, [%1];" : "=h"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ uint64_t global_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Wait until *flag != 0 (acquire), for at most timeout_ns of device time and at
// most 2^23 polls.  Returns false if the wait ran out.
__device__ __forceinline__ bool wait_flag(const int32_t* flag, int64_t timeout_ns) {
  const uint64_t t0 = global_ns();
#pragma unroll 1
  for (int it = 0; it < (1 << 23); ++it) {
    int v;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(flag) : "memory");
    if (v != 0) return true;
    if ((int64_t)(global_ns() - t0) > timeout_ns) return false;
    __nanosleep(256);
  }
  return false;
}

}  // namespace tpcfit
