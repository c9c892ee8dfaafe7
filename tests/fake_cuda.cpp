// A CUDA runtime and kernel launchers that do nothing, for testing the library's host
// side (tpcfit_host.cpp) without a GPU: allocations are counted against a limit and
// remembered, launches note the device pointers that they were given.
#include <cuda_runtime.h>

#include <cstdlib>
#include <map>
#include <set>
#include <string>

#include "internal.h"

namespace {
std::map<void*, size_t> g_live;
size_t g_bytes = 0, g_limit = 0;
int g_capturing = 0;
cudaError_t g_last = cudaSuccess;
std::set<void*> g_used;  // by the launches since the last fake_forget
int g_taped = 0;         // the last fit wrote the tape

void use(const void* p) {
  if (p) g_used.insert(const_cast<void*>(p));
}
cudaError_t fail(cudaError_t e) { return g_last = e; }
}  // namespace

extern "C" {
void fake_limit(long long bytes) { g_limit = (size_t)bytes; }
void fake_capture(int on) { g_capturing = on; }
long long fake_bytes() { return (long long)g_bytes; }
void fake_forget() { g_used.clear(); }
int fake_taped() { return g_taped; }
// Buffers that the launches since fake_forget were given, and how many of them are
// allocated.
long long fake_used() { return (long long)g_used.size(); }
long long fake_used_live() {
  long long n = 0;
  for (void* p : g_used) n += (long long)g_live.count(p);
  return n;
}

cudaError_t cudaMalloc(void** p, size_t n) {
  if (g_capturing) return fail(cudaErrorStreamCaptureUnsupported);
  if (n == 0) {
    *p = nullptr;
    return cudaSuccess;
  }
  if (g_bytes + n > g_limit) return fail(cudaErrorMemoryAllocation);
  *p = std::malloc(16);
  g_live[*p] = n;
  g_bytes += n;
  return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
  if (!p) return cudaSuccess;
  auto it = g_live.find(p);
  if (it == g_live.end()) return fail(cudaErrorInvalidValue);
  g_bytes -= it->second;
  g_live.erase(it);  // (the address itself is not given back: it stays unique)
  return cudaSuccess;
}
cudaError_t cudaMemGetInfo(size_t* avail, size_t* total) {
  *avail = g_limit - g_bytes;
  *total = g_limit;
  return cudaSuccess;
}
cudaError_t cudaGetLastError() {
  const cudaError_t e = g_last;
  g_last = cudaSuccess;
  return e;
}
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* s) {
  *s = g_capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
  return cudaSuccess;
}
cudaError_t cudaGetDevice(int* d) { return *d = 0, cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { return *v = 152, cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaMemcpy(void*, const void*, size_t, cudaMemcpyKind) { return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void*, const void*, size_t, cudaMemcpyKind, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaMemcpy2DAsync(void*, size_t, const void*, size_t, size_t, size_t, cudaMemcpyKind, cudaStream_t) {
  return cudaSuccess;
}
cudaError_t cudaMemset(void*, int, size_t) { return cudaSuccess; }
cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { return *s = nullptr, cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return *e = nullptr, cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
}

namespace tpcfit {
namespace {
// (as the real launchers do, these report what is left in the error state)
cudaError_t fit(const FitArgs& a) {
  for (const void* p : {(const void*)a.perm, (const void*)a.ck, (const void*)a.ck_last, (const void*)a.tape,
                        (const void*)a.tape_item, (const void*)a.work, (const void*)a.align})
    use(p);
  g_taped = a.tape != nullptr;
  return cudaGetLastError();
}
template <class A>
cudaError_t follow(const A& a) {
  for (const void* p : {(const void*)a.perm, (const void*)a.ck, (const void*)a.ck_last, (const void*)a.tape,
                        (const void*)a.tape_item, (const void*)a.work, (const void*)a.seg})
    use(p);
  return cudaGetLastError();
}
}  // namespace
cudaError_t launch_fit_fast(const FitArgs& a, int, int, int, cudaStream_t) { return fit(a); }
cudaError_t launch_fit_det(const FitArgs& a, int, int, int, cudaStream_t) { return fit(a); }
cudaError_t launch_backward_fast(const BwdArgs& a, int, cudaStream_t) { return follow(a); }
cudaError_t launch_backward_det(const BwdArgs& a, int, cudaStream_t) {
  use(a.grad_meas);
  return follow(a);
}
cudaError_t launch_smooth_fast(const SmoothArgs& a, cudaStream_t) { return follow(a); }
cudaError_t launch_smooth_det(const SmoothArgs& a, cudaStream_t) { return follow(a); }
cudaError_t backward_store_fast(int, int, int, int64_t& n) { return n = 1 << 20, cudaSuccess; }
cudaError_t backward_store_det(int, int, int, int64_t& n) { return n = 2 << 20, cudaSuccess; }
cudaError_t smooth_store_fast(int64_t& n) { return n = 3 << 20, cudaSuccess; }
cudaError_t smooth_store_det(int64_t& n) { return n = 3 << 20, cudaSuccess; }
cudaError_t launch_clear_gradients(const int32_t*, int32_t, int64_t, const int32_t*, const int32_t*, float* gm, float*,
                                   cudaStream_t) {
  return use(gm), cudaSuccess;
}
size_t key_sort_scratch_bytes(int64_t n) { return 16 * (size_t)n; }
size_t key_fixed_scratch_bytes() { return 131072; }
cudaError_t launch_key_sort(const uint16_t*, int64_t, int, void* scratch, int**, int**, cudaStream_t) {
  return use(scratch), cudaSuccess;
}
cudaError_t launch_key_reduce(const float*, const int*, const int*, float*, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_key_fixed_reduce(const float*, const uint16_t*, int64_t, int, void* scratch, float*, cudaStream_t) {
  return use(scratch), cudaSuccess;
}
cudaError_t launch_length_order(const int32_t*, int32_t, int32_t* perm, int32_t*, cudaStream_t) {
  return use(perm), cudaSuccess;
}
int64_t frame_order_scratch_ints(int32_t n) { return 600 * (int64_t)n; }
cudaError_t launch_frame_length_order(const int32_t*, int32_t, const int64_t*, int32_t, int32_t* perm, int32_t* scratch,
                                      cudaStream_t) {
  return use(perm), use(scratch), cudaSuccess;
}
int64_t reject_scratch_ints(int32_t n) { return n / 32 + 2; }
cudaError_t launch_reject(const int32_t*, int32_t, const float*, const float*, const uint16_t*, int64_t, const float*,
                          float, float*, float*, uint16_t*, int32_t*, int32_t* scratch, cudaStream_t) {
  return use(scratch), cudaSuccess;
}
bool rtc_available() { return false; }
long long rtc_compile_count() { return 0; }
const char* rtc_log() { return ""; }
tpcfit_status rtc_build(const GeoConst&, bool, int, int, int, bool, const char*) { return TPCFIT_ERTC; }
tpcfit_status rtc_launch_fit(const GeoConst&, bool, int, int, const FitArgs&, const char*, cudaStream_t) {
  return TPCFIT_ERTC;
}
}  // namespace tpcfit
