// The CUDA runtime calls and kernel launches that the library's host code makes, on host memory: for
// tests of what the host code does when memory runs out or a stream is captured, without a GPU.
// Every trim, synchronisation and launch is written to a log; allocations can be made to fail.
#include <cstdlib>
#include <cstring>
#include <map>
#include <string>

#include "ebic.h"
#include "ebic_internal.h"

namespace {

// the pool of matrices and tables, the default pool, cudaMalloc, the pool of calls' tables
enum Kind { kPool, kAsync, kMalloc, kCallPool, kKinds };

std::string g_log;
int g_seen[kKinds], g_fail_from[kKinds], g_fail_count[kKinds];
bool g_capturing;
// a capture under way in another thread: 0 none, 1 thread-local or relaxed, 2 global; and whether a call
// that may not be made beside it has ended it
int g_other;
bool g_other_broken;
cudaError_t beside(int from) {
  if (g_other < from) return cudaSuccess;
  g_other_broken = true;
  return cudaErrorStreamCaptureUnsupported;
}
struct Block {
  size_t bytes;
  Kind kind;
};
std::map<char*, Block> g_live;

void note(const std::string& what) { g_log += what + "\n"; }

cudaError_t take(void** p, size_t bytes, Kind kind) {
  const int n = g_seen[kind]++;
  if (n >= g_fail_from[kind] && n < g_fail_from[kind] + g_fail_count[kind])
    return cudaErrorMemoryAllocation;
  char* m = static_cast<char*>(std::malloc(bytes));  // (untouched pages cost nothing)
  g_live[m] = {bytes, kind};
  *p = m;
  return cudaSuccess;
}

cudaError_t drop(void* p) {
  auto it = g_live.find(static_cast<char*>(p));
  if (it == g_live.end()) return cudaErrorInvalidValue;
  std::free(p);
  g_live.erase(it);
  return cudaSuccess;
}

// pools by their handles: the library's, told apart by their limits, then the default one
char g_handles[3];
const cudaStream_t kOwnStream = reinterpret_cast<cudaStream_t>(0x100);
const cudaMemPool_t kDefaultPool = reinterpret_cast<cudaMemPool_t>(&g_handles[2]);
int g_pools;
uint64_t g_limit[2];
Kind kind_of(cudaMemPool_t pool) {
  const int i = (int)(reinterpret_cast<char*>(pool) - g_handles);
  return i == 2 ? kAsync : g_limit[i] == (2ull << 30) ? kPool : kCallPool;
}

}  // namespace

extern "C" {

// ---- the test's side -------------------------------------------------------------------------
void fake_reset() {
  g_log.clear();
  for (int k = 0; k < kKinds; ++k) g_seen[k] = g_fail_from[k] = g_fail_count[k] = 0;
  g_capturing = false;
  g_other = 0;
  g_other_broken = false;
}
// allocations `from` .. `from + count` of a kind, counted from the last reset, find no memory
void fake_fail(int kind, int from, int count) {
  g_fail_from[kind] = from;
  g_fail_count[kind] = count;
}
void fake_capture(int on) { g_capturing = on != 0; }
void fake_other_capture(int mode) { g_other = mode; }
int fake_other_broken() { return g_other_broken; }
const char* fake_log() { return g_log.c_str(); }
int fake_seen(int kind) { return g_seen[kind]; }
uint64_t fake_limit(int kind) {
  for (int i = 0; i < g_pools; ++i)
    if (kind_of(reinterpret_cast<cudaMemPool_t>(&g_handles[i])) == kind) return g_limit[i];
  return 0;
}
size_t fake_live(int kind) {
  size_t n = 0;
  for (const auto& b : g_live)
    if (b.second.kind == kind) n += b.second.bytes;
  return n;
}

void* fake_device(size_t bytes) {
  void* p = nullptr;
  (void)take(&p, bytes, kMalloc);
  return p;
}
void fake_device_free(void* p) { (void)drop(p); }

// ---- the runtime's side ------------------------------------------------------------------------
cudaError_t cudaMallocFromPoolAsync(void** p, size_t n, cudaMemPool_t pool, cudaStream_t) {
  return take(p, n, kind_of(pool));
}
cudaError_t cudaMallocAsync(void** p, size_t n, cudaStream_t) { return take(p, n, kAsync); }
cudaError_t cudaMalloc(void** p, size_t n) {
  const cudaError_t e = beside(2);
  return e == cudaSuccess ? take(p, n, kMalloc) : e;
}
cudaError_t cudaFreeAsync(void* p, cudaStream_t s) {
  const cudaError_t e = beside(s ? 2 : 1);
  return e == cudaSuccess ? drop(p) : e;
}
cudaError_t cudaFree(void* p) {  // (waits for the device)
  const cudaError_t e = beside(2);
  if (e != cudaSuccess) return e;
  note("idle");
  return drop(p);
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
  *s = kOwnStream;
  return beside(2);
}
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) {
  *p = std::calloc(1, n);
  return cudaSuccess;
}
cudaError_t cudaFreeHost(void* p) {
  std::free(p);
  return cudaSuccess;
}
cudaError_t cudaHostGetDevicePointer(void** d, void* h, unsigned) {
  *d = h;
  return cudaSuccess;
}
cudaError_t cudaMemPoolCreate(cudaMemPool_t* pool, const cudaMemPoolProps*) {
  if (g_pools == 2) return cudaErrorUnknown;
  *pool = reinterpret_cast<cudaMemPool_t>(&g_handles[g_pools++]);
  return cudaSuccess;
}
cudaError_t cudaMemPoolDestroy(cudaMemPool_t) { return cudaSuccess; }
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t pool, cudaMemPoolAttr, void* v) {
  if (pool != kDefaultPool)
    g_limit[reinterpret_cast<char*>(pool) - g_handles] = *static_cast<uint64_t*>(v);
  return cudaSuccess;
}
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t pool, size_t keep) {
  const Kind k = kind_of(pool);
  note((k == kPool ? "trim library " : k == kAsync ? "trim default " : "trim tables ") +
       std::to_string(keep));
  return cudaSuccess;
}
cudaError_t cudaDeviceGetDefaultMemPool(cudaMemPool_t* pool, int) {
  *pool = kDefaultPool;
  return cudaSuccess;
}
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* st) {
  *st = g_capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
  return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
  if (s == kOwnStream) return beside(2);  // (the library's own, for an allocation)
  note("sync");
  return g_capturing ? cudaErrorStreamCaptureUnsupported : cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() {
  note("device sync");
  const cudaError_t e = beside(1);
  return g_capturing ? cudaErrorStreamCaptureUnsupported : e;
}
cudaError_t cudaGetDevice(int* d) {
  *d = 0;
  return cudaSuccess;
}
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetDeviceCount(int* n) {
  *n = 1;
  return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) {
  *v = 152;
  return cudaSuccess;
}
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "error"; }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* at, const void* p) {
  std::memset(at, 0, sizeof(*at));
  const char* c = static_cast<const char*>(p);
  for (const auto& b : g_live)
    if (c >= b.first && c < b.first + b.second.bytes) at->type = cudaMemoryTypeDevice;
  return cudaSuccess;
}
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) {
  std::memcpy(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
  std::memcpy(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpy2DAsync(void* d, size_t dp, const void* s, size_t sp, size_t w, size_t h,
                              cudaMemcpyKind, cudaStream_t) {
  for (size_t i = 0; i < h; ++i)
    std::memcpy(static_cast<char*>(d) + i * dp, static_cast<const char*>(s) + i * sp, w);
  return cudaSuccess;
}
cudaError_t cudaMemset(void* p, int v, size_t n) {
  std::memset(p, v, n);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t) {
  std::memset(p, v, n);
  return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t*) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float*, cudaEvent_t, cudaEvent_t) { return cudaSuccess; }

}  // extern "C"

// ---- the kernels' side ----------------------------------------------------------------------------
namespace ebic {

cudaError_t launch_rank_transform(const Layout&, const float*, int64_t, int, float, uint32_t*,
                                  uint32_t*, int, cudaStream_t) {
  note("rank");
  return cudaSuccess;
}
cudaError_t launch_prepare(const PrepareArgs&, cudaStream_t) {
  note("prepare");
  return cudaSuccess;
}
cudaError_t launch_eval(const EvalArgs&, bool, int, bool, cudaStream_t) {
  note("evaluate");
  return cudaSuccess;
}
cudaError_t launch_pair_build(const Layout&, const uint32_t*, uint32_t*, uint32_t, int64_t, int,
                              cudaStream_t) {
  note("pair build");
  return cudaSuccess;
}
cudaError_t launch_pair_eval(const PairArgs&, bool, int, bool, cudaStream_t) {
  note("pair evaluate");
  return cudaSuccess;
}
bool pair_score_fits(int64_t, uint32_t, bool, uint32_t, bool, int32_t) { return false; }
cudaError_t launch_pair_score(const PairArgs&, const ScoreArgs&, bool, bool, cudaStream_t) {
  return cudaSuccess;
}
uint32_t fused_prepare_blocks(uint32_t, uint32_t, uint32_t, int) { return 1; }
cudaError_t launch_fused_prepare(const FusedPrepareArgs&, uint32_t, cudaStream_t) {
  return cudaSuccess;
}
cudaError_t launch_fused_finalize(const uint32_t*, uint32_t, const uint32_t*, const uint32_t*,
                                  uint32_t, const uint32_t*, uint32_t, const uint32_t*,
                                  const uint64_t*, uint64_t*, const uint32_t*, uint32_t*,
                                  uint32_t*, bool, cudaStream_t) {
  return cudaSuccess;
}
cudaError_t launch_overlap(const uint32_t*, uint32_t, const uint32_t*, uint32_t, int64_t,
                           uint32_t*, uint32_t*, const uint32_t*, int, bool, cudaStream_t) {
  return cudaSuccess;
}
cudaError_t launch_fitness_finalize(const uint16_t*, const uint32_t*, uint32_t, const uint32_t*,
                                    const uint16_t*, const uint32_t*, uint32_t, const uint32_t*,
                                    const uint32_t*, uint64_t*, const uint32_t*, bool,
                                    cudaStream_t) {
  return cudaSuccess;
}

}  // namespace ebic

// the library's other allocation calls, which no entry point built here makes
extern "C" int fake_scratch(size_t bytes) {
  void* p = nullptr;
  const cudaError_t e = ebic::scratch_alloc(&p, bytes, nullptr);
  if (e == cudaSuccess) (void)cudaFreeAsync(p, nullptr);
  return e;
}
extern "C" int fake_fixed(size_t bytes) {
  void* p = nullptr;
  const cudaError_t e = ebic::fixed_alloc(&p, bytes);
  if (e == cudaSuccess) (void)cudaFree(p);
  return e;
}
