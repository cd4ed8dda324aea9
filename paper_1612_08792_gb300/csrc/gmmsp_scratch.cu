// Device scratch of the calls that have no context to keep it in (the
// accuracy metrics, the context-free connectivity call): a stream-ordered
// memory pool per device, so that a call does not pay an allocation and a
// device-wide free (about 0.4 ms for the metrics of 256 481x321 images).
// The pool keeps at most kKeep bytes between calls, gives them back on
// gmmsp_release_scratch or when an allocation fails, and is safe from several
// threads and streams (an allocation is ordered on the caller's stream, and a
// free makes the memory available to work after it).
#include <cuda_runtime.h>

#include <mutex>

#include "../../include/gmmsp.h"
#include "gmmsp_internal.cuh"

namespace gmmsp {
namespace {

constexpr unsigned long long kKeep = 256ull << 20;
constexpr int kMaxDevices = 64;
std::mutex g_mutex;
cudaMemPool_t g_pool[kMaxDevices] = {};

// The current device's pool (null where the device has none: plain
// allocations then).
cudaMemPool_t pool_of_device(int* device) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return nullptr;
  *device = dev;
  std::lock_guard<std::mutex> lock(g_mutex);
  if (!g_pool[dev]) {
    cudaMemPoolProps props = {};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = dev;
    cudaMemPool_t p = nullptr;
    if (cudaMemPoolCreate(&p, &props) != cudaSuccess) {
      cudaGetLastError();
      return nullptr;
    }
    unsigned long long keep = kKeep;
    if (cudaMemPoolSetAttribute(p, cudaMemPoolAttrReleaseThreshold, &keep) != cudaSuccess) cudaGetLastError();
    g_pool[dev] = p;
  }
  return g_pool[dev];
}

}  // namespace

cudaError_t CallScratch::alloc(size_t bytes, cudaStream_t s) {
  stream = s;
  // These calls synchronise, which a capture does not allow: refused before
  // anything of them is recorded (the pool would allocate inside the graph).
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  cudaError_t e = cudaStreamIsCapturing(s, &cs);
  if (e != cudaSuccess || cs != cudaStreamCaptureStatusNone) {
    cudaGetLastError();
    return cudaErrorStreamCaptureUnsupported;
  }
  int dev = 0;
  cudaMemPool_t pool = pool_of_device(&dev);
  if (pool) {
    pooled = true;
    e = cudaMallocFromPoolAsync(&ptr, bytes, pool, s);
    if (e == cudaErrorMemoryAllocation) {
      cudaGetLastError();
      cudaMemPoolTrimTo(pool, 0);
      e = cudaMallocFromPoolAsync(&ptr, bytes, pool, s);
    }
  } else {
    e = cudaMalloc(&ptr, bytes);
  }
  if (e != cudaSuccess) {
    cudaGetLastError();
    ptr = nullptr;
  }
  return e;
}

CallScratch::~CallScratch() {
  if (!ptr) return;
  if (pooled) cudaFreeAsync(ptr, stream);
  else cudaFree(ptr);
}

}  // namespace gmmsp

extern "C" gmmsp_status gmmsp_release_scratch(void) {
  std::lock_guard<std::mutex> lock(gmmsp::g_mutex);
  for (cudaMemPool_t p : gmmsp::g_pool)
    if (p && cudaMemPoolTrimTo(p, 0) != cudaSuccess) {
      cudaGetLastError();
      return GMMSP_E_CUDA;
    }
  return GMMSP_OK;
}
