// dev_alloc.cu -- device memory of plans, batches and served jobs.
//
// A small plan is some twenty buffers; with cudaMalloc and cudaFree (35-50 us
// and 25-35 us each when the driver has to map or unmap) its allocations cost
// several times its kernels.  Buffers up to POOL_MAX_BYTES come from a memory
// pool of the library's own (1 us each), larger ones from cudaMalloc, which
// maps large memory faster than a pool does (800 MB: 240 against 630 us).
//
// What the pool keeps once buffers are freed is bounded (POOL_KEEP_BYTES) and
// is given back when an allocation would otherwise fail.  Buffers are allocated
// and freed on one stream of the library that runs nothing else and
// is drained before an allocation is handed out, so a buffer may be used from
// any stream; a buffer is freed only when no queued work uses it (dev_free's
// contract), from any thread.  cudaFree waited for the buffer's own device; with
// a pool the owners do (dev_drain).
//
// Scratch that one stream's work uses waits for that stream alone when it is
// freed (scratch_free): cudaFree waits for the whole device, so that a plan built
// beside a running sweep ended with the sweep.  Scratch from cudaMalloc is freed
// with cudaFreeAsync, and given back when the stream is next synchronised.  (50M
// nonzeros, 1.2 GB of scratch: a build takes 13.7 ms so, as with cudaFree, and
// 15.3 ms with the scratch in the pool.)
#include <mutex>

#include "device_drain.h"
#include "plan.cuh"

namespace spm {
namespace {

constexpr size_t POOL_MAX_BYTES = (size_t)32 << 20;
constexpr size_t POOL_KEEP_BYTES = (size_t)64 << 20;
constexpr int kMaxDevices = 64;

struct DevicePool {
  cudaMemPool_t pool = nullptr;
  cudaStream_t stream = nullptr;
};
std::mutex g_mutex;
DevicePool g_pools[kMaxDevices];

// The pool of the current device, or null (then cudaMalloc serves).
DevicePool* device_pool(int dev) {
  if (dev < 0 || dev >= kMaxDevices) return nullptr;
  std::lock_guard<std::mutex> lock(g_mutex);
  DevicePool& d = g_pools[dev];
  if (d.pool) return &d;
  cudaMemPoolProps props{};
  props.allocType = cudaMemAllocationTypePinned;
  props.location.type = cudaMemLocationTypeDevice;
  props.location.id = dev;
  cudaMemPool_t pool = nullptr;
  cudaStream_t stream = nullptr;
  unsigned long long keep = POOL_KEEP_BYTES;
  if (cudaMemPoolCreate(&pool, &props) != cudaSuccess ||
      cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep) != cudaSuccess ||
      cudaStreamCreateWithFlags(&stream, cudaStreamNonBlocking) != cudaSuccess) {
    (void)cudaGetLastError();
    if (pool) cudaMemPoolDestroy(pool);
    return nullptr;
  }
  d.pool = pool;
  d.stream = stream;
  return &d;
}

// The pool of a device that need not be the current one, or null if it has none.
DevicePool* known_pool(int dev) {
  if (dev < 0 || dev >= kMaxDevices) return nullptr;
  std::lock_guard<std::mutex> lock(g_mutex);
  return g_pools[dev].pool ? &g_pools[dev] : nullptr;
}

bool pooled(size_t bytes) { return bytes <= POOL_MAX_BYTES; }

cudaError_t try_alloc(void** ptr, size_t bytes, DevicePool* d) {
  if (!d || !pooled(bytes)) return cudaMalloc(ptr, bytes);
  cudaError_t e = cudaMallocFromPoolAsync(ptr, bytes, d->pool, d->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(d->stream);
  return e;
}

}  // namespace

spm_status dev_alloc(void** ptr, size_t bytes) {
  *ptr = nullptr;
  int dev = 0;
  SPM_CUDA_TRY(cudaGetDevice(&dev));
  DevicePool* d = device_pool(dev);
  cudaError_t e = try_alloc(ptr, bytes, d);
  if (e == cudaErrorMemoryAllocation && d) {
    (void)cudaGetLastError();
    (void)cudaMemPoolTrimTo(d->pool, 0);  // what the pool keeps goes back first
    e = try_alloc(ptr, bytes, d);
  }
  if (e == cudaSuccess) return SPM_OK;
  (void)cudaGetLastError();
  *ptr = nullptr;
  return e == cudaErrorMemoryAllocation ? SPM_ERR_OOM : SPM_ERR_CUDA;
}

void scratch_free(void* ptr, size_t bytes, cudaStream_t s) {
  if (!ptr) return;
  if (pooled(bytes)) {
    cudaStreamSynchronize(s);
    dev_free(ptr, bytes);
  } else {
    cudaFreeAsync(ptr, s);
  }
  (void)cudaGetLastError();
}

void dev_free(void* ptr, size_t bytes) {
  if (!ptr) return;
  cudaPointerAttributes at{};
  DevicePool* d = nullptr;
  if (pooled(bytes) && cudaPointerGetAttributes(&at, ptr) == cudaSuccess) d = known_pool(at.device);
  if (d) cudaFreeAsync(ptr, d->stream);
  else cudaFree(ptr);
  (void)cudaGetLastError();
}

size_t dev_held(int device) {
  DevicePool* d = known_pool(device);
  if (!d) return 0;
  unsigned long long reserved = 0, used = 0;
  if (cudaStreamSynchronize(d->stream) != cudaSuccess ||  // the frees so far
      cudaMemPoolGetAttribute(d->pool, cudaMemPoolAttrReservedMemCurrent, &reserved) != cudaSuccess ||
      cudaMemPoolGetAttribute(d->pool, cudaMemPoolAttrUsedMemCurrent, &used) != cudaSuccess) {
    (void)cudaGetLastError();
    return 0;
  }
  return reserved > used ? (size_t)(reserved - used) : 0;
}

void dev_trim(int device, size_t keep) {
  DevicePool* d = known_pool(device);
  if (!d || dev_held(device) <= keep) return;
  (void)cudaMemPoolTrimTo(d->pool, 0);
  (void)cudaGetLastError();
}

bool dev_drain(int device) {
  struct Runtime {
    bool get(int* d) { return cudaGetDevice(d) == cudaSuccess; }
    bool set(int d) { return cudaSetDevice(d) == cudaSuccess; }
    bool sync() { return cudaDeviceSynchronize() == cudaSuccess; }
  } rt;
  if (drain_device(rt, device)) return true;
  (void)cudaGetLastError();
  return false;
}

}  // namespace spm
