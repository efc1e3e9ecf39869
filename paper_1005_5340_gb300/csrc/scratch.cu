// Device scratch of the entry points that have no context to keep a workspace
// in (tddft_gemm_f64_emulated, tddft_kernel_apply_centres): a private
// stream-ordered memory pool per device.  Allocations follow the caller's
// stream, so calls from several threads and streams never share a buffer in
// flight.  The pool keeps at most kKeepBytes between calls (a cudaMalloc and
// cudaFree pair costs about 90 us, most of a small product) and gives them
// back when a context is destroyed, or at the process's end.
#include <mutex>

#include "internal.h"

namespace tddft {
namespace {
constexpr unsigned long long kKeepBytes = 256ull << 20;
constexpr int kMaxDevices = 128;
std::mutex g_mutex;
cudaMemPool_t g_pool[kMaxDevices] = {};

cudaError_t device_pool(cudaMemPool_t *pool) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(g_mutex);
  if (!g_pool[dev]) {
    cudaMemPoolProps props = {};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = dev;
    cudaMemPool_t p = nullptr;
    e = cudaMemPoolCreate(&p, &props);
    if (e != cudaSuccess) return e;
    unsigned long long keep = kKeepBytes;
    e = cudaMemPoolSetAttribute(p, cudaMemPoolAttrReleaseThreshold, &keep);
    if (e != cudaSuccess) {
      cudaMemPoolDestroy(p);
      return e;
    }
    g_pool[dev] = p;
  }
  *pool = g_pool[dev];
  return cudaSuccess;
}
}  // namespace

cudaError_t scratch_alloc(void **p, size_t bytes, cudaStream_t st) {
  cudaMemPool_t pool = nullptr;
  const cudaError_t e = device_pool(&pool);
  return e != cudaSuccess ? e : cudaMallocFromPoolAsync(p, bytes, pool, st);
}

int sm_count() {
  static PerDevice n;
  const int v = n.get([] {
    int dev = 0, sms = 0;
    return cudaGetDevice(&dev) == cudaSuccess &&
                   cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess
               ? sms : 0;
  });
  return v > 0 ? v : 1;
}

void scratch_trim() {
  std::lock_guard<std::mutex> lock(g_mutex);
  for (cudaMemPool_t p : g_pool)
    if (p) cudaMemPoolTrimTo(p, 0);
}

}  // namespace tddft
