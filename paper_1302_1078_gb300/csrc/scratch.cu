// Stream-ordered memory of the library: the scratch of calls without a plan and what plans own.
//
// The default memory pool gives everything back to the driver whenever the device is waited for, so
// a program that synchronises between calls paid for mapping the same scratch again each time (a
// 64 x 64 grid's SpMV: 25 us among others, 230 us after a wait).  The library keeps one pool per
// device instead, which holds on to at most kKeepBytes; what exceeds it goes back at the next
// wait, and gbs_release_scratch gives back the rest.  The driver orders reuse between streams, and
// the pool is created once under a lock, so any threads and streams may call.
#include <atomic>
#include <mutex>

#include "gbspmv.h"
#include "launch.h"

namespace gbs {
namespace {

constexpr int kMaxDevices = 64;
constexpr unsigned long long kKeepBytes = 256ull << 20;

std::mutex g_mu;
std::atomic<cudaMemPool_t> g_pool[kMaxDevices];

// The current device's pool; NULL where there is none (the caller takes the default pool).
cudaMemPool_t pool_of_device(cudaStream_t s) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return nullptr;
  cudaMemPool_t p = g_pool[dev].load(std::memory_order_acquire);
  if (p) return p;
  // a pool cannot be made while the stream is captured; the first call outside a capture makes it
  cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(s, &st) != cudaSuccess || st != cudaStreamCaptureStatusNone) return nullptr;
  std::lock_guard<std::mutex> lock(g_mu);
  p = g_pool[dev].load(std::memory_order_relaxed);
  if (p) return p;
  cudaMemPoolProps props{};
  props.allocType = cudaMemAllocationTypePinned;
  props.location.type = cudaMemLocationTypeDevice;
  props.location.id = dev;
  unsigned long long keep = kKeepBytes;
  if (cudaMemPoolCreate(&p, &props) != cudaSuccess) {
    cudaGetLastError();
    return nullptr;
  }
  if (cudaMemPoolSetAttribute(p, cudaMemPoolAttrReleaseThreshold, &keep) != cudaSuccess) {
    cudaGetLastError();
    cudaMemPoolDestroy(p);
    return nullptr;
  }
  g_pool[dev].store(p, std::memory_order_release);
  return p;
}

}  // namespace

cudaError_t scratch_alloc(void** p, size_t bytes, cudaStream_t s) {
  *p = nullptr;
  if (bytes == 0) bytes = 1;
  cudaMemPool_t pool = pool_of_device(s);
  return pool ? cudaMallocFromPoolAsync(p, bytes, pool, s) : cudaMallocAsync(p, bytes, s);
}

cudaError_t scratch_free(void* p, cudaStream_t s) { return p ? cudaFreeAsync(p, s) : cudaSuccess; }

}  // namespace gbs

extern "C" int gbs_release_scratch(void) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  cudaMemPool_t p = e == cudaSuccess && dev >= 0 && dev < gbs::kMaxDevices ? gbs::g_pool[dev].load() : nullptr;
  if (e == cudaSuccess && p) e = cudaMemPoolTrimTo(p, 0);
  if (e != cudaSuccess) gbs::set_last_error(cudaGetErrorString(e));
  return e == cudaSuccess ? GBS_OK : GBS_ECUDA;
}
