#include "workspace.hpp"

#include <mutex>

#include "apex_internal.hpp"

namespace apex {

namespace {
std::mutex pool_mutex;
cudaMemPool_t pools[kMaxDevices] = {};

cudaError_t pool_of_device(bool create, cudaMemPool_t* out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(pool_mutex);
  if (!pools[dev] && create) {
    cudaMemPoolProps props = {};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = dev;
    cudaMemPool_t pool = nullptr;
    if ((e = cudaMemPoolCreate(&pool, &props)) != cudaSuccess) return e;
    unsigned long long kept = kWorkspaceKept;
    if ((e = cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &kept)) != cudaSuccess) {
      cudaMemPoolDestroy(pool);
      return e;
    }
    pools[dev] = pool;
  }
  *out = pools[dev];
  return cudaSuccess;
}
}  // namespace

cudaError_t workspace_alloc(void** out, size_t bytes, cudaStream_t s) {
  *out = nullptr;
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  cudaError_t e = cudaStreamIsCapturing(s, &cap);
  if (e != cudaSuccess) return e;
  if (cap != cudaStreamCaptureStatusNone) return cudaErrorStreamCaptureUnsupported;
  cudaMemPool_t pool = nullptr;
  if ((e = pool_of_device(true, &pool)) != cudaSuccess) return e;
  return cudaMallocFromPoolAsync(out, bytes, pool, s);
}

void workspace_free(void* p, cudaStream_t s) {
  if (p) cudaFreeAsync(p, s);
}

cudaError_t workspace_trim() {
  cudaMemPool_t pool = nullptr;
  const cudaError_t e = pool_of_device(false, &pool);
  return e == cudaSuccess && pool ? cudaMemPoolTrimTo(pool, 0) : e;
}

}  // namespace apex

extern "C" int apex_trim_scratch(void) { return apex::workspace_trim() == cudaSuccess ? APEX_OK : APEX_ECUDA; }
