// Outlier rejection after the smoother: every cluster whose leave-one-out
// chi2 exceeds a cut is dropped from its track, the others are copied in
// their order.  A warp counts four tracks at once and copies one at a time; the
// kept clusters of 32 consecutive ones are placed with a ballot and a population
// count, so the output order is the input order (the cluster-to-track relation the
// deterministic mode keeps, Sec. 2) and the results do not depend on scheduling.
//
// Three kernels: the kept clusters counted; the counts of the blocks' tracks
// summed up; the clusters copied to where the sums say.  Bound by memory: chi2 is
// read twice, the clusters are read and written once (28 bytes a cluster).  (Kept
// ballots would spare the second read of chi2, but their 3 MB cost a new handle's
// first call 100 us of allocation.)  A warp loads four times 32 clusters at once,
// before it knows which are kept: one latency per 128 clusters instead of two per
// 32.  200,000 tracks, 16.1 million clusters: 188 us of kernels before.
#include <cuda_runtime.h>
#include <stdint.h>

#include "device_util.cuh"
#include "internal.h"

namespace tpcfit {
namespace {

constexpr int kWarpsPerBlock = 8;
constexpr int kTracksPerBlock = 32;
constexpr int kUnroll = 4;  // times 32 clusters in flight

// The ranges of the block's tracks (empty beyond the last one).
__device__ __forceinline__ void block_ranges(const int32_t* off, int32_t n_tracks, int64_t n_hits, int32_t (&rb)[kTracksPerBlock],
                                             int32_t (&re)[kTracksPerBlock]) {
  if (threadIdx.x < kTracksPerBlock) {
    const int64_t t = (int64_t)blockIdx.x * kTracksPerBlock + threadIdx.x;
    int32_t b = 0, e = 0;
    if (t < n_tracks) track_range(off, t, n_hits, b, e);
    rb[threadIdx.x] = b;
    re[threadIdx.x] = e;
  }
  __syncthreads();
}

// kept[t] = number of clusters track t keeps, sums[block] = that of the block's
// tracks.
__global__ void __launch_bounds__(kWarpsPerBlock * 32) reject_count(const int32_t* off, int32_t n_tracks,
                                                                      int64_t n_hits, const float* chi2, float cut,
                                                                      int32_t* kept, int32_t* sums) {
  __shared__ int warp_sum[kWarpsPerBlock];
  __shared__ int32_t rb[kTracksPerBlock], re[kTracksPerBlock];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  block_ranges(off, n_tracks, n_hits, rb, re);
  constexpr int kPer = kTracksPerBlock / kWarpsPerBlock;  // tracks of a warp, the first 128 clusters of all in flight
  float x[kPer][kUnroll];
#pragma unroll
  for (int k = 0; k < kPer; ++k)
#pragma unroll
    for (int j = 0; j < kUnroll; ++j) {
      const int64_t c = (int64_t)rb[warp + k * kWarpsPerBlock] + 32 * j + lane;
      x[k][j] = c < re[warp + k * kWarpsPerBlock] ? __ldcs(chi2 + c) : 0.0f;
    }
  int sum = 0;
#pragma unroll
  for (int k = 0; k < kPer; ++k) {
    const int w = warp + k * kWarpsPerBlock;
    const int32_t b = rb[w], e = re[w];
    int n = 0;
#pragma unroll
    for (int j = 0; j < kUnroll; ++j)  // a NaN chi2 keeps its cluster
      n += __popc(__ballot_sync(0xffffffffu, (int64_t)b + 32 * j + lane < e && !(x[k][j] > cut)));
    for (int64_t base = (int64_t)b + 32 * kUnroll; base < e; base += 32) {
      const int64_t c = base + lane;
      n += __popc(__ballot_sync(0xffffffffu, c < e && !(__ldcs(chi2 + (c < e ? c : b)) > cut)));
    }
    const int64_t t = (int64_t)blockIdx.x * kTracksPerBlock + w;
    if (lane == 0 && t < n_tracks) kept[t] = n;
    sum += n;
  }
  if (lane == 0) warp_sum[warp] = sum;
  __syncthreads();
  if (threadIdx.x == 0) {
    int s = 0;
    for (int k = 0; k < kWarpsPerBlock; ++k) s += warp_sum[k];
    sums[blockIdx.x] = s;
  }
}

// Copy the kept clusters of each track to its place, in order, and turn the
// tracks' counts into the new offsets; nothing is written at or beyond n_hits (the
// outputs' length).
__global__ void __launch_bounds__(kWarpsPerBlock * 32) reject_compact(
    const int32_t* off, int32_t n_tracks, int64_t n_hits, const float* chi2, float cut, const int32_t* sums,
    const float* y, const float* z, const uint16_t* rowsec, int32_t* new_off, float* y_out, float* z_out,
    uint16_t* rowsec_out) {
  __shared__ int32_t place[kTracksPerBlock];
  __shared__ int32_t rb[kTracksPerBlock], re[kTracksPerBlock];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  static_assert(kTracksPerBlock == 32, "one warp places the block's tracks");
  if (warp == 0) {
    const int64_t t = (int64_t)blockIdx.x * kTracksPerBlock + lane;
    const int n = t < n_tracks ? new_off[t] : 0;
    int incl = n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int u = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += u;
    }
    const int at = sums[blockIdx.x] + incl - n;
    place[lane] = at;
    if (t < n_tracks) new_off[t] = at;
  }
  block_ranges(off, n_tracks, n_hits, rb, re);
  const unsigned below = (1u << lane) - 1u;
  for (int k = warp; k < kTracksPerBlock; k += kWarpsPerBlock) {
    const int32_t b = rb[k], e = re[k];
    int64_t pos = place[k];
    for (int64_t base = b; base < e; base += 32 * kUnroll) {
      float x[kUnroll], cy[kUnroll], cz[kUnroll];
      uint16_t rs[kUnroll];
#pragma unroll
      for (int j = 0; j < kUnroll; ++j) {
        const int64_t c = base + 32 * j + lane;
        if (c < e) {
          x[j] = __ldcs(chi2 + c);
          cy[j] = __ldcs(y + c);
          cz[j] = __ldcs(z + c);
          rs[j] = __ldcs(rowsec + c);
        }
      }
#pragma unroll
      for (int j = 0; j < kUnroll; ++j) {
        const bool keep = base + 32 * j + lane < e && !(x[j] > cut);
        const unsigned m = __ballot_sync(0xffffffffu, keep);
        const int64_t o = pos + __popc(m & below);
        if (keep && o >= 0 && o < n_hits) {  // overlapping ranges must not write outside the outputs
          y_out[o] = cy[j];
          z_out[o] = cz[j];
          rowsec_out[o] = rs[j];
        }
        pos += __popc(m);
      }
    }
  }
}

}  // namespace

int64_t reject_scratch_ints(int32_t n_tracks) { return ((int64_t)n_tracks + kTracksPerBlock - 1) / kTracksPerBlock + 1; }

cudaError_t launch_reject(const int32_t* off, int32_t n_tracks, const float* y, const float* z, const uint16_t* rowsec,
                          int64_t n_hits, const float* chi2, float cut, float* y_out, float* z_out,
                          uint16_t* rowsec_out, int32_t* off_out, int32_t* scratch, cudaStream_t s) {
  if (n_tracks <= 0) return cudaMemsetAsync(off_out, 0, sizeof(int32_t), s);
  const int blocks = (int)(((int64_t)n_tracks + kTracksPerBlock - 1) / kTracksPerBlock);
  reject_count<<<blocks, kWarpsPerBlock * 32, 0, s>>>(off, n_tracks, n_hits, chi2, cut, off_out, scratch);
  const cudaError_t e = launch_scan_exclusive(scratch, blocks, off_out + n_tracks, nullptr, s);
  if (e != cudaSuccess) return e;
  reject_compact<<<blocks, kWarpsPerBlock * 32, 0, s>>>(off, n_tracks, n_hits, chi2, cut, scratch, y, z, rowsec,
                                                        off_out, y_out, z_out, rowsec_out);
  return cudaGetLastError();
}

}  // namespace tpcfit
