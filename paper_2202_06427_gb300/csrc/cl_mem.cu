// cl_mem.cu -- device memory of the library: one stream-ordered memory pool
// per device, shared by every handle and thread (the CUDA pool is safe for
// both). A list's arrays are two blocks of it and the two-set calls' workspace
// one, where each array was a cudaMalloc of its own (about twenty per list,
// 0.5 ms of host time per build and free at 200,000 particles). Freed memory
// beyond kPoolKeep goes back to the device: by the pool itself at the next
// synchronisation, and by mem_settle before a call that freed a lot returns.
#include <mutex>

#include "cl_internal.cuh"

namespace clk {

namespace {

std::mutex pool_mu;
cudaMemPool_t pools[kCacheDevices];

int device_pool(cudaMemPool_t* out) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kCacheDevices) return CL_ERR_CUDA;
  std::lock_guard<std::mutex> g(pool_mu);
  if (!pools[dev]) {
    cudaMemPoolProps props = {};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = dev;
    cudaMemPool_t p = nullptr;
    unsigned long long keep = kPoolKeep;
    if (cudaMemPoolCreate(&p, &props) != cudaSuccess) return CL_ERR_CUDA;
    if (cudaMemPoolSetAttribute(p, cudaMemPoolAttrReleaseThreshold, &keep) != cudaSuccess) {
      cudaMemPoolDestroy(p);
      return CL_ERR_CUDA;
    }
    pools[dev] = p;
  }
  *out = pools[dev];
  return CL_OK;
}

}  // namespace

bool capturing(cudaStream_t s) {
  cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(s, &st) == cudaSuccess) return st != cudaStreamCaptureStatusNone;
  cudaGetLastError();  // the legacy stream, and another one is being captured
  return true;
}

// While a stream is captured, an allocation on it would become a node of the
// graph: memory that does not exist until the graph runs. The calls then allocate
// and free for themselves, which most capture modes refuse.
int mem_alloc(void** p, size_t bytes, cudaStream_t s) {
  *p = nullptr;
  cudaMemPool_t pool;
  int e = CL_OK;
  if (capturing(s)) {
    if (cudaMalloc(p, bytes ? bytes : 1) != cudaSuccess) e = CL_ERR_OOM;
  } else if (!(e = device_pool(&pool)) && cudaMallocFromPoolAsync(p, bytes ? bytes : 1, pool, s) != cudaSuccess) {
    e = CL_ERR_OOM;
  }
  if (e) {
    cudaGetLastError();
    *p = nullptr;
  }
  return e;
}

void mem_free(void* p, cudaStream_t s) {
  if (!p) return;
  if (capturing(s)) cudaFree(p);
  else cudaFreeAsync(p, s);
}

void mem_settle(cudaStream_t s) {
  cudaMemPool_t pool;
  unsigned long long held = 0, used = 0;
  if (capturing(s) || device_pool(&pool) || cudaMemPoolGetAttribute(pool, cudaMemPoolAttrReservedMemCurrent, &held) != cudaSuccess ||
      held <= kPoolKeep || cudaStreamSynchronize(s) != cudaSuccess ||
      cudaMemPoolGetAttribute(pool, cudaMemPoolAttrUsedMemCurrent, &used) != cudaSuccess)
    return;
  cudaMemPoolTrimTo(pool, (size_t)(used + kPoolKeep));
}

}  // namespace clk
