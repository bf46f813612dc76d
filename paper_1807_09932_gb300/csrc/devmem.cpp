// Device memory of matrices, pair tables and searches: one stream-ordered pool per device.
//
// Opening a data set takes its rank matrix and its pair table (25 MB and 226 MB for 436,444 x 64)
// and a search some fifty buffers; cudaMalloc and cudaFree map and unmap that memory every time
// (0.6 ms to open and close that data set, against 0.2 ms of kernels; 1.7 ms for a table of 1.7
// GB; 0.9 ms per search). The pool keeps up to kPoolKeep bytes of what has been freed mapped for
// the next matrix or search; anything above goes back to the system at the next synchronisation,
// and all of it when an allocation of the library finds no memory. The pool is the driver's, so
// threads and streams may use it side by side; memory is handed from one user to the next only
// after the first one's free is reached by its stream.
#include <mutex>

#include "ebic_internal.h"

namespace ebic {
namespace {

constexpr uint64_t kPoolKeep = 2ull << 30;  // under 1 % of the device's memory
constexpr int kMaxDevices = 64;
std::mutex g_mu;
cudaMemPool_t g_pool[kMaxDevices] = {};

cudaError_t pool_of(int device, cudaMemPool_t* out) {
  if (device < 0 || device >= kMaxDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lk(g_mu);
  if (!g_pool[device]) {
    cudaMemPoolProps props = {};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = device;
    cudaMemPool_t pool = nullptr;
    cudaError_t e = cudaMemPoolCreate(&pool, &props);
    if (e != cudaSuccess) return e;
    uint64_t keep = kPoolKeep;
    e = cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep);
    if (e != cudaSuccess) {
      (void)cudaMemPoolDestroy(pool);
      return e;
    }
    g_pool[device] = pool;
  }
  *out = g_pool[device];
  return cudaSuccess;
}

}  // namespace

cudaError_t device_alloc(void** p, size_t bytes, int device, cudaStream_t s) {
  cudaMemPool_t pool = nullptr;
  cudaError_t e = pool_of(device, &pool);
  if (e != cudaSuccess) return e;
  e = cudaMallocFromPoolAsync(p, bytes ? bytes : 16, pool, s);
  if (e != cudaErrorMemoryAllocation) return e;
  // out of memory: freed memory that the pools still hold goes back first
  (void)cudaGetLastError();
  (void)cudaStreamSynchronize(s);
  (void)cudaMemPoolTrimTo(pool, 0);
  cudaMemPool_t scratch = nullptr;
  if (cudaDeviceGetDefaultMemPool(&scratch, device) == cudaSuccess)
    (void)cudaMemPoolTrimTo(scratch, 0);
  (void)cudaGetLastError();
  return cudaMallocFromPoolAsync(p, bytes ? bytes : 16, pool, s);
}

cudaError_t device_free(void* p, cudaStream_t s) {
  return p ? cudaFreeAsync(p, s) : cudaSuccess;
}

}  // namespace ebic
