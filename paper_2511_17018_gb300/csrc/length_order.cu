// Track ordering by length: a counting sort over the number of clusters per
// track, longest first, so that the 32 tracks of a warp have equal lengths and
// its lanes finish together.  Positions within one length are assigned with
// atomics; the fit writes every output at the track's own index, so the
// results do not depend on that order.
#include <cuda_runtime.h>
#include <stdint.h>

#include "internal.h"
#include "device_util.cuh"

namespace tpcfit {
namespace {

constexpr int kBins = 256;
constexpr int kThreads = 256;
constexpr int kItems = 4;

__device__ __forceinline__ int length_bin(const int32_t* off, int64_t i) {
  int len = off[i + 1] - off[i];
  return len < 0 ? 0 : (len > kBins - 1 ? kBins - 1 : len);
}

__global__ void __launch_bounds__(kThreads) length_hist(const int32_t* off, int32_t n, int32_t* hist) {
  __shared__ int sh[kBins];
  for (int i = threadIdx.x; i < kBins; i += blockDim.x) sh[i] = 0;
  __syncthreads();
  const int64_t base = (int64_t)blockIdx.x * kThreads * kItems;
#pragma unroll
  for (int it = 0; it < kItems; ++it) {
    const int64_t i = base + (int64_t)it * kThreads + threadIdx.x;
    if (i < n) atomicAdd(&sh[length_bin(off, i)], 1);
  }
  __syncthreads();
  for (int b = threadIdx.x; b < kBins; b += blockDim.x)
    if (sh[b]) atomicAdd(&hist[b], sh[b]);
}

// start[b] = number of tracks longer than b (longest first), from the histogram
// of 256 bins, by the first 256 threads of a block (all its threads call it).
__device__ __forceinline__ void longest_first(const int* hist, int* start) {
  __shared__ int warp_sum[kBins / 32];
  const int t = threadIdx.x, lane = t & 31;
  const int b = kBins - 1 - t;  // thread t owns bin 255 - t: an exclusive prefix sum from the longest bin
  const int v = t < kBins ? hist[b] : 0;
  int incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int u = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += u;
  }
  if (t < kBins && lane == 31) warp_sum[t >> 5] = incl;
  __syncthreads();
  if (t < kBins) {
    int before = incl - v;
    for (int w = 0; w < (t >> 5); ++w) before += warp_sum[w];
    start[b] = before;
  }
}

// The whole ordering of a small batch in one block: histogram, prefix sum and
// scatter, with nothing to clear beforehand.  Bound by its launch and two passes
// of dependent loads.  For up to kSmallOrder tracks it replaces a memset and two
// kernels (1,000 tracks: 14 us of kernels and two launch gaps).
constexpr int kSmallThreads = 1024;
constexpr int kSmallItems = 16;
constexpr int kSmallOrder = kSmallThreads * kSmallItems;

__global__ void __launch_bounds__(kSmallThreads) length_order_small(const int32_t* off, int32_t n, int32_t* perm) {
  __shared__ int hist[kBins];
  __shared__ int cursor[kBins];
  if (threadIdx.x < kBins) hist[threadIdx.x] = 0;
  __syncthreads();
  int bin[kSmallItems];
#pragma unroll
  for (int it = 0; it < kSmallItems; ++it) {
    const int i = it * kSmallThreads + threadIdx.x;
    bin[it] = i < n ? length_bin(off, i) : -1;
  }
#pragma unroll
  for (int it = 0; it < kSmallItems; ++it)
    if (bin[it] >= 0) atomicAdd(&hist[bin[it]], 1);
  __syncthreads();
  longest_first(hist, cursor);
  __syncthreads();
#pragma unroll
  for (int it = 0; it < kSmallItems; ++it)
    if (bin[it] >= 0) perm[atomicAdd(&cursor[bin[it]], 1)] = it * kSmallThreads + threadIdx.x;
}

__global__ void __launch_bounds__(kThreads) length_scatter(const int32_t* off, int32_t n, const int32_t* hist,
                                                           int32_t* cursor, int32_t* perm) {
  __shared__ int start[kBins];
  __shared__ int local[kBins];
  __shared__ int base[kBins];
  longest_first(hist, start);
  local[threadIdx.x] = 0;
  __syncthreads();
  const int64_t first = (int64_t)blockIdx.x * kThreads * kItems;
  int bin[kItems], rank[kItems];
#pragma unroll
  for (int it = 0; it < kItems; ++it) {
    const int64_t i = first + (int64_t)it * kThreads + threadIdx.x;
    bin[it] = -1;
    if (i < n) {
      bin[it] = length_bin(off, i);
      rank[it] = atomicAdd(&local[bin[it]], 1);
    }
  }
  __syncthreads();
  {
    const int b = threadIdx.x;
    base[b] = local[b] ? atomicAdd(&cursor[b], local[b]) : 0;
  }
  __syncthreads();
#pragma unroll
  for (int it = 0; it < kItems; ++it) {
    const int64_t i = first + (int64_t)it * kThreads + threadIdx.x;
    if (bin[it] >= 0) perm[start[bin[it]] + base[bin[it]] + rank[it]] = (int32_t)i;
  }
}

// Batched frames: key = frame * 256 + (255 - length) orders by frame, then by
// decreasing length.  A block's tracks are consecutive, so nearly all of them are
// in the frame of its first one (a second one at a boundary): those are counted in
// shared memory and the block adds one count per length to the frame's, instead of
// one global atomic per track on a few hundred addresses (40 frames, 576,000
// tracks: histogram and scatter 18 + 23 us before).
__device__ __forceinline__ int frame_clamped(const int64_t* fb, int n_frames, int64_t i) {
  const int f = frame_of(fb, n_frames, i);
  return f < 0 ? n_frames - 1 : f;  // out-of-table tracks are rejected by the fit; keep them in range here
}

// Frame of track i, given that of a track before it in the block.
__device__ __forceinline__ int frame_near(const int64_t* fb, int n_frames, int64_t i, int f0, int64_t end0) {
  return i < end0 ? f0 : frame_clamped(fb, n_frames, i);
}

__global__ void __launch_bounds__(kThreads) frame_hist(const int32_t* off, int32_t n, const int64_t* fb, int n_frames,
                                                       int32_t* hist) {
  __shared__ int sh[kBins];
  sh[threadIdx.x] = 0;
  const int64_t first = (int64_t)blockIdx.x * kThreads * kItems;
  const int f0 = frame_clamped(fb, n_frames, first);
  const int64_t end0 = fb[f0 + 1];
  __syncthreads();
#pragma unroll
  for (int it = 0; it < kItems; ++it) {
    const int64_t i = first + (int64_t)it * kThreads + threadIdx.x;
    if (i >= n) continue;
    const int f = frame_near(fb, n_frames, i, f0, end0);
    const int bin = kBins - 1 - length_bin(off, i);
    if (f == f0) atomicAdd(&sh[bin], 1);
    else atomicAdd(&hist[f * kBins + bin], 1);
  }
  __syncthreads();
  if (sh[threadIdx.x]) atomicAdd(&hist[f0 * kBins + threadIdx.x], sh[threadIdx.x]);
}

__global__ void __launch_bounds__(kThreads) frame_scatter(const int32_t* off, int32_t n, const int64_t* fb,
                                                          int n_frames, const int32_t* start, int32_t* cursor,
                                                          int32_t* perm) {
  __shared__ int local[kBins];
  __shared__ int base[kBins];
  local[threadIdx.x] = 0;
  const int64_t first = (int64_t)blockIdx.x * kThreads * kItems;
  const int f0 = frame_clamped(fb, n_frames, first);
  const int64_t end0 = fb[f0 + 1];
  __syncthreads();
  int bin[kItems], rank[kItems];
#pragma unroll
  for (int it = 0; it < kItems; ++it) {
    const int64_t i = first + (int64_t)it * kThreads + threadIdx.x;
    bin[it] = -1;
    if (i >= n) continue;
    const int f = frame_near(fb, n_frames, i, f0, end0);
    const int k = kBins - 1 - length_bin(off, i);
    if (f == f0) {
      bin[it] = k;
      rank[it] = atomicAdd(&local[k], 1);
    } else {
      const int key = f * kBins + k;
      perm[start[key] + atomicAdd(&cursor[key], 1)] = (int32_t)i;
    }
  }
  __syncthreads();
  {
    const int k = threadIdx.x;
    base[k] = local[k] ? start[f0 * kBins + k] + atomicAdd(&cursor[f0 * kBins + k], local[k]) : 0;
  }
  __syncthreads();
#pragma unroll
  for (int it = 0; it < kItems; ++it) {
    const int64_t i = first + (int64_t)it * kThreads + threadIdx.x;
    if (bin[it] >= 0) perm[base[bin[it]] + rank[it]] = (int32_t)i;
  }
}

}  // namespace

int64_t frame_order_scratch_ints(int32_t n_frames) {
  const int64_t bins = (int64_t)n_frames * kBins;
  return 2 * bins + scan_tmp_ints(bins);
}

cudaError_t launch_frame_length_order(const int32_t* off, int32_t n_tracks, const int64_t* frame_base,
                                      int32_t n_frames, int32_t* perm, int32_t* scratch, cudaStream_t s) {
  if (n_tracks <= 0) return cudaSuccess;
  const int64_t bins = (int64_t)n_frames * kBins;
  int32_t* start = scratch;
  int32_t* cursor = scratch + bins;
  int32_t* tmp = scratch + 2 * bins;
  cudaError_t e = cudaMemsetAsync(scratch, 0, sizeof(int32_t) * 2 * bins, s);
  if (e != cudaSuccess) return e;
  const int64_t blocks = ((int64_t)n_tracks + kThreads * kItems - 1) / (kThreads * kItems);
  frame_hist<<<(unsigned)blocks, kThreads, 0, s>>>(off, n_tracks, frame_base, n_frames, start);
  e = launch_scan_exclusive(start, (int)bins, nullptr, tmp, s);
  if (e != cudaSuccess) return e;
  frame_scatter<<<(unsigned)blocks, kThreads, 0, s>>>(off, n_tracks, frame_base, n_frames, start, cursor, perm);
  return cudaGetLastError();
}

cudaError_t launch_length_order(const int32_t* off, int32_t n_tracks, int32_t* perm, int32_t* scratch,
                                cudaStream_t s) {
  if (n_tracks <= 0) return cudaSuccess;
  if (n_tracks <= kSmallOrder) {
    length_order_small<<<1, kSmallThreads, 0, s>>>(off, n_tracks, perm);
    return cudaGetLastError();
  }
  cudaError_t e = cudaMemsetAsync(scratch, 0, sizeof(int32_t) * 2 * kBins, s);
  if (e != cudaSuccess) return e;
  const int64_t blocks = ((int64_t)n_tracks + kThreads * kItems - 1) / (kThreads * kItems);
  length_hist<<<(unsigned)blocks, kThreads, 0, s>>>(off, n_tracks, scratch);
  length_scatter<<<(unsigned)blocks, kThreads, 0, s>>>(off, n_tracks, scratch, scratch + kBins, perm);
  return cudaGetLastError();
}

}  // namespace tpcfit
