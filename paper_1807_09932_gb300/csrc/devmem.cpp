// Device memory. Matrices, pair tables and searches take theirs from one stream-ordered pool per
// device, the pair table of a single call from another; the calls' other scratch comes from the
// device's default pool, and what a captured graph holds the address of from cudaMalloc.
//
// Opening a data set takes its rank matrix and its pair table (25 MB and 226 MB for 436,444 x 64)
// and a search some fifty buffers; cudaMalloc and cudaFree map and unmap that memory every time
// (0.6 ms to open and close that data set, against 0.2 ms of kernels; 1.7 ms for a table of 1.7
// GB; 0.9 ms per search). A pool keeps freed memory mapped for the next user while it holds, used
// and unused, no more than its limit; beyond that, freed memory goes back to the system at the
// next synchronisation. An allocation that finds no memory has all the pools give back what they hold
// unused, and is tried once more (not a call's pair table: the call does without one, and need not
// wait for its stream). The pools are the driver's, so
// threads and streams may use them side by side; memory is handed from one user to the next only
// after the first one's free is reached by its stream.
#include <mutex>
#include <vector>

#include "ebic_internal.h"

namespace ebic {
namespace {

enum Pool { kLasting, kCall, kPools };
// Together under 1 % of the device's memory. The second is what one call takes at most, and a pool of
// its own so that the matrices loaded beside it don't count against its limit.
constexpr uint64_t kPoolKeep[kPools] = {2ull << 30, 512ull << 20};
constexpr int kMaxDevices = 64;
std::mutex g_mu;
cudaMemPool_t g_pool[kMaxDevices][kPools] = {};

// Memory that its owner has given up is freed, once no stream uses it, on a stream of the library's own.
struct Lasting {
  std::mutex mu;
  cudaStream_t stream = nullptr;
  std::vector<void*> waiting;  // to be freed, by the next call that can
  void* neighbour = nullptr;   // see wait_idle
  cudaError_t ready() {        // under mu
    return stream ? cudaSuccess : cudaStreamCreateWithFlags(&stream, cudaStreamNonBlocking);
  }
};
Lasting g_lasting[kMaxDevices];

// Waits until the device, the current one, has run all work given to it. By cudaFree, which waits for
// every stream (CUDA Programming Guide, "Stream Ordered Memory Allocator": cudaMalloc and cudaFree make
// the GPU synchronize across all executing streams; beside a 20 ms kernel on another stream it returned
// when that had ended) and which a thread may call while another one captures in thread-local or relaxed
// mode. cudaDeviceSynchronize fails then, and so does the capture; an operation on the legacy stream does
// that to the capture of any blocking stream. The block that stays allocated beside the freed one
// keeps the two calls at 2.5 us (60 when they map and unmap their page).
cudaError_t wait_idle(Lasting& r) {
  void* block = nullptr;
  cudaError_t e = cudaSuccess;
  {
    std::lock_guard<std::mutex> lk(r.mu);
    if (!r.neighbour) e = cudaMalloc(&r.neighbour, 256);
  }
  if (e == cudaSuccess) e = cudaMalloc(&block, 256);
  if (e == cudaSuccess) return cudaFree(block);
  (void)cudaGetLastError();
  return e == cudaErrorMemoryAllocation ? cudaDeviceSynchronize() : e;
}

cudaError_t pool_of(int device, Pool which, cudaMemPool_t* out) {
  if (device < 0 || device >= kMaxDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lk(g_mu);
  if (!g_pool[device][which]) {
    cudaMemPoolProps props = {};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = device;
    cudaMemPool_t pool = nullptr;
    cudaError_t e = cudaMemPoolCreate(&pool, &props);
    if (e != cudaSuccess) return e;
    uint64_t keep = kPoolKeep[which];
    e = cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep);
    if (e != cudaSuccess) {
      (void)cudaMemPoolDestroy(pool);
      return e;
    }
    g_pool[device][which] = pool;
  }
  *out = g_pool[device][which];
  return cudaSuccess;
}

// What the pools of `device` hold unused goes back to the system.
void trim(int device) {
  if (device >= 0 && device < kMaxDevices) {
    std::lock_guard<std::mutex> lk(g_mu);
    for (cudaMemPool_t pool : g_pool[device])
      if (pool) (void)cudaMemPoolTrimTo(pool, 0);
  }
  cudaMemPool_t scratch = nullptr;
  if (cudaDeviceGetDefaultMemPool(&scratch, device) == cudaSuccess)
    (void)cudaMemPoolTrimTo(scratch, 0);
  (void)cudaGetLastError();
}

// After an allocation on s found no memory: whether to try it again. Memory freed on s is unused
// once s has run; a capture can neither wait for that nor be left with an error, and its
// allocations take no memory before the graph runs.
bool give_back(int device, cudaStream_t s) {
  (void)cudaGetLastError();
  cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(s, &st) != cudaSuccess || st != cudaStreamCaptureStatusNone) {
    (void)cudaGetLastError();
    return false;
  }
  if (cudaStreamSynchronize(s) != cudaSuccess) return false;
  trim(device);
  return true;
}

}  // namespace

cudaError_t device_alloc(void** p, size_t bytes, int device, cudaStream_t s) {
  cudaMemPool_t pool = nullptr;
  cudaError_t e = pool_of(device, kLasting, &pool);
  if (e != cudaSuccess) return e;
  e = cudaMallocFromPoolAsync(p, bytes ? bytes : 16, pool, s);
  if (e == cudaErrorMemoryAllocation && give_back(device, s))
    e = cudaMallocFromPoolAsync(p, bytes ? bytes : 16, pool, s);
  return e;
}

cudaError_t call_table_alloc(void** p, size_t bytes, int device, cudaStream_t s) {
  cudaMemPool_t pool = nullptr;
  const cudaError_t e = pool_of(device, kCall, &pool);
  return e == cudaSuccess ? cudaMallocFromPoolAsync(p, bytes ? bytes : 16, pool, s) : e;
}

cudaError_t device_free(void* p, cudaStream_t s) {
  return p ? cudaFreeAsync(p, s) : cudaSuccess;
}

cudaError_t device_retire(std::vector<void*> ps, int device, bool drained) {
  if (device < 0 || device >= kMaxDevices) return cudaErrorInvalidDevice;
  Lasting& r = g_lasting[device];
  if (!drained) {  // what an earlier call could not free goes with it
    std::lock_guard<std::mutex> lk(r.mu);
    ps.insert(ps.end(), r.waiting.begin(), r.waiting.end());
    r.waiting.clear();
  }
  cudaError_t e = drained ? cudaSuccess : wait_idle(r);
  std::lock_guard<std::mutex> lk(r.mu);
  if (e == cudaSuccess) e = r.ready();
  for (void* p : ps) {
    if (!p) continue;
    if (e == cudaSuccess) e = cudaFreeAsync(p, r.stream);
    if (e != cudaSuccess) r.waiting.push_back(p);
  }
  if (e != cudaSuccess) (void)cudaGetLastError();
  return e;
}

cudaError_t scratch_alloc(void** p, size_t bytes, cudaStream_t s) {
  cudaError_t e = cudaMallocAsync(p, bytes ? bytes : 16, s);
  int device = 0;
  if (e == cudaErrorMemoryAllocation && cudaGetDevice(&device) == cudaSuccess &&
      give_back(device, s))
    e = cudaMallocAsync(p, bytes ? bytes : 16, s);
  return e;
}

cudaError_t release_memory(int device) {
  const cudaError_t e = device_retire({}, device, false);
  if (e == cudaSuccess) trim(device);
  return e;
}

cudaError_t fixed_alloc(void** p, size_t bytes) {
  cudaError_t e = cudaMalloc(p, bytes ? bytes : 16);
  int device = 0;
  if (e == cudaErrorMemoryAllocation && cudaGetDevice(&device) == cudaSuccess &&
      give_back(device, nullptr))
    e = cudaMalloc(p, bytes ? bytes : 16);
  return e;
}

}  // namespace ebic
