// Internal declarations shared by the host part of libtpcfit and its kernel
// modules.  Not part of the public C ABI (include/tpcfit.h).
#pragma once

#include <cstdint>
#include <string>
#include <cuda_runtime.h>

#include "kernel_abi.h"
#include "tpcfit.h"

namespace tpcfit {

// Geometry and field -> per-time-frame constants (host, FP64 rounded to FP32);
// false for an invalid geometry.
bool build_geo(const tpcfit_geometry* g, double bz, GeoConst& out);

// Blocks of a kernel resident at once over all SMs, and the SMs (cached per
// kernel by its launcher).
struct Resident {
  int blocks = 0;
  int sms = 0;
};
template <class K>
cudaError_t resident_blocks(K kernel, int threads, size_t smem, Resident& r) {
  // (several threads may come here at once: blocks is the last to be written)
  if (__atomic_load_n(&r.blocks, __ATOMIC_ACQUIRE) != 0) return cudaSuccess;
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  int dev = 0, sms = 0, per_sm = 0;
  e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  r.sms = sms;
  __atomic_store_n(&r.blocks, sms * per_sm, __ATOMIC_RELEASE);
  return cudaSuccess;
}

// How a persistent kernel's work items (up to 32 tracks, one per lane) are laid
// over the GPU.  `resident`: blocks of `max_warps` warps resident at once,
// `sms`: SMs.
//   - A batch with fewer than 32 tracks per warp scheduler (19,456 on 152 SMs)
//     gets smaller items, one per scheduler: a lone warp's time per step does not
//     depend on how many of its lanes work, and fewer lanes diverge less.
//   - A batch with fewer items than resident warps runs on every SM with fewer
//     warps per block, instead of on few SMs with full blocks.
// Warp w of block b starts with item w * blocks + b, so that the items, which
// are sorted by length, spread evenly over the SMs; later items come from the
// work counter, which is not touched (nor cleared) when there are none.
// Measured (whole calls, us; full blocks of 32-track items before): fit of 1,000
// tracks of 152 clusters 365 -> 179, of 20,000 tracks 395 -> 204; fit + adjoint of
// 1,000 tracks 1,719 -> 704, deterministic of 50,000 tracks 2,301 -> 1,775.
struct WorkShape {
  int32_t tracks;  // per item
  int32_t items;
  int32_t blocks;
  int32_t warps;   // per block
};
inline WorkShape work_shape(int64_t n_tracks, int resident, int max_warps, int sms) {
  WorkShape w;
  const int64_t schedulers = 4 * (int64_t)sms;
  const int64_t t = (n_tracks + schedulers - 1) / schedulers;
  w.tracks = (int32_t)(t < 1 ? 1 : (t < kWarp ? t : kWarp));
  const int64_t items = (n_tracks + w.tracks - 1) / w.tracks;
  w.items = (int32_t)items;
  w.blocks = (int32_t)(items < resident ? items : resident);
  const int64_t per_block = (items + w.blocks - 1) / w.blocks;
  w.warps = (int32_t)(per_block < max_warps ? per_block : max_warps);
  return w;
}
inline bool needs_work_counter(const WorkShape& w) { return w.items > w.blocks * w.warps; }

// The windows in which the fit stages clusters (WarpStage in fit_core.cuh): four
// clusters that are aligned in y, wherever in a window the array begins.  Arrays taken
// from larger ones at one offset begin at the same place, so that z and rowsec share
// the windows; where they do not (mixed), only a kernel made for it copies windows.
// mixed_kernel, shifted: what the kernel is made for; it copies cluster by cluster what
// it is not made for.
inline int window_place(const void* p, size_t element) { return (int)((uintptr_t)p / element) & 3; }
inline bool mixed_windows(const FitArgs& a) {
  const int y = window_place(a.y, sizeof(float));
  return y != window_place(a.z, sizeof(float)) || y != window_place(a.rowsec, sizeof(uint16_t));
}
inline void set_windows(FitArgs& a, bool mixed_kernel, bool shifted) {
  const int place = window_place(a.y, sizeof(float));
  const bool fits = a.n_hits >= 4 && (place == 0 || (shifted && a.n_hits <= INT32_MAX - 4));  // (hits plus 3 in 32 bits)
  a.win_shift = fits ? place : 0;
  a.win_whole = fits && (mixed_kernel || !mixed_windows(a)) ? (uint32_t)(a.n_hits - 3) : 0;
}

// Tracks per work item alone (what the tape's layout depends on).
inline int32_t item_tracks(int64_t n_tracks, int sms) { return work_shape(n_tracks, 1, 1, sms).tracks; }
// Clear a launch's counters: the tape's (with the work item counter), the work
// item counter alone, or nothing.
inline cudaError_t clear_work(unsigned int* work, bool tape, bool counter, cudaStream_t s) {
  if (tape) return cudaMemsetAsync(work, 0, 4 * sizeof(unsigned int), s);
  if (counter) return cudaMemsetAsync(work, 0, sizeof(unsigned int), s);
  return cudaSuccess;
}

// ---- kernel launchers, one per module
cudaError_t launch_fit_fast(const FitArgs& a, int lanes_per_track, int rows_per_stage, int warps, cudaStream_t s);
cudaError_t launch_fit_det(const FitArgs& a, int lanes_per_track, int rows_per_stage, int warps, cudaStream_t s);
cudaError_t launch_backward_fast(const BwdArgs& a, int warps, cudaStream_t s);
cudaError_t launch_backward_det(const BwdArgs& a, int warps, cudaStream_t s);
// float4 elements of the segment store a backward launch needs (`warps`: of the
// reverse from checkpoints; the physics bits phys; the factor form, 0 square root,
// 1 U-D)
cudaError_t backward_store_fast(int warps, int phys, int form, int64_t& float4s);
cudaError_t backward_store_det(int warps, int phys, int form, int64_t& float4s);
// the two-filter smoother of a recorded fit, and its segment store (float4s)
cudaError_t launch_smooth_fast(const SmoothArgs& a, cudaStream_t s);
cudaError_t launch_smooth_det(const SmoothArgs& a, cudaStream_t s);
cudaError_t smooth_store_fast(int64_t& float4s);
cudaError_t smooth_store_det(int64_t& float4s);
// true if `warps` is a compiled backward block shape
bool backward_shape_supported(int warps);

// Zero the gradients gm [n_hits][2] (8-byte aligned) of the clusters that the adjoint of
// a recorded fit does not reach (key_reduce.cu), and the alignment gradient
// [kAlignFloats] if not null.
cudaError_t launch_clear_gradients(const int32_t* off, int32_t n_tracks, int64_t n_hits, const int32_t* ndf,
                                   const int32_t* ck_last, float* gm, float* grad_align, cudaStream_t s);
// Deterministic per-key reduction of cluster gradients (key_reduce.cu).
size_t key_sort_scratch_bytes(int64_t n_hits);
cudaError_t launch_key_sort(const uint16_t* rowsec, int64_t n_hits, int n_rows, void* scratch, int** sorted_out,
                            int** key_start_out, cudaStream_t s);
cudaError_t launch_key_reduce(const float* grad_meas, const int* sorted, const int* key_start, float* grad_align,
                              cudaStream_t s);
// The order-independent alternative: fixed-point integer sums per key (the
// deterministic mode's default); scratch of key_fixed_scratch_bytes().
size_t key_fixed_scratch_bytes();
cudaError_t launch_key_fixed_reduce(const float* grad_meas, const uint16_t* rowsec, int64_t n_hits, int n_rows,
                                    void* scratch, float* grad_align, cudaStream_t s);
// true if (lanes_per_track, rows_per_stage, warps) is a compiled launch shape
bool fit_shape_supported(int lanes_per_track, int rows_per_stage, int warps);

// ---- run-time compilation of the fit (rtc.cpp, Sec. 5)
bool rtc_available();
long long rtc_compile_count();
const char* rtc_log();
// The NVRTC source of the fit for these constants and mode.
std::string rtc_fit_source(const GeoConst& g, bool det);
// NVRTC only (no device needed): the CUBIN of a variant, stored in cache_dir
// when given.
// record: 0 nothing, 1 checkpoints, 2 the tape.
tpcfit_status rtc_build(const GeoConst& g, bool det, int rps, int warps, int record, bool frames,
                        const char* cache_dir);
// Compile (once per source and variant) and launch the fit specialised for g.
tpcfit_status rtc_launch_fit(const GeoConst& g, bool det, int rps, int warps, const FitArgs& a, const char* cache_dir,
                             cudaStream_t s);

// Ordering by (frame ascending, length descending) for batched frames.
// scratch: int32 [2 * n_frames * 256 + scan_tmp_ints(n_frames * 256)].
int64_t frame_order_scratch_ints(int32_t n_frames);
cudaError_t launch_frame_length_order(const int32_t* off, int32_t n_tracks, const int64_t* frame_base,
                                      int32_t n_frames, int32_t* perm, int32_t* scratch, cudaStream_t s);
// Outlier rejection (reject.cu): the clusters with chi2 > cut dropped, the
// others copied in order; off_out [n_tracks + 1] receives the new offsets.
// scratch: reject_scratch_ints(n_tracks) ints.
int64_t reject_scratch_ints(int32_t n_tracks);
cudaError_t launch_reject(const int32_t* off, int32_t n_tracks, const float* y, const float* z, const uint16_t* rowsec,
                          int64_t n_hits, const float* chi2, float cut, float* y_out, float* z_out,
                          uint16_t* rowsec_out, int32_t* off_out, int32_t* scratch, cudaStream_t s);
// Exclusive prefix sum of n ints in place (key_reduce.cu); tmp: scan_tmp_ints(n)
// ints, or null (one block does it whatever n; total, if not null, then receives
// the sum of all).
int64_t scan_tmp_ints(int64_t n);
cudaError_t launch_scan_exclusive(int* v, int n, int* total, int* tmp, cudaStream_t s);

// Length-ordering permutation: perm[k] = track processed k-th, longest first.
// scratch: int32[2 * 256] (zeroed by the launcher).
cudaError_t launch_length_order(const int32_t* off, int32_t n_tracks, int32_t* perm, int32_t* scratch,
                                cudaStream_t s);

}  // namespace tpcfit
