// Scratch memory of the library's calls: stream-ordered, from a pool of the
// library's own that keeps up to 256 MiB between calls.
//
// The device's default pool gives its memory back at every synchronisation,
// after which the first allocation of the next call maps it again: 110 us,
// more than many calls take in all (a phase of one step on a 5 000-node
// graph 150 -> 26 us).  What the pool keeps is bounded, is handed back
// when a device's last graph is destroyed and when an allocation fails, and a pool
// that the caller has made the device's current one is used instead of it.
#include <mutex>

#include "api_util.cuh"
#include "deco_internal.cuh"

namespace deco {
namespace {

constexpr int kMaxDevices = 64;
constexpr uint64_t kKeptBytes = 256ull << 20;

// The pool belongs to the CUDA context in which it was made: it is looked up
// with that context's unique id, so that a teardown and re-creation of the
// context leads to a new pool.
struct PoolSlot {
  unsigned long long ctx_id = 0;
  cudaMemPool_t pool = nullptr;
};
PoolSlot g_slot[kMaxDevices];
std::mutex g_mutex;

// the library's pool on the current device (`make`: made if there is none), or null
cudaMemPool_t kept_pool(bool make) {
  int dev = 0;
  unsigned long long ctx_id = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
    cudaGetLastError();
    return nullptr;
  }
  std::lock_guard<std::mutex> lock(g_mutex);
  if (current_context_id(&ctx_id) != DECO_OK) {
    clear_error();
    return nullptr;
  }
  PoolSlot& slot = g_slot[dev];
  if (slot.pool && slot.ctx_id == ctx_id) return slot.pool;
  if (!make) return nullptr;
  cudaMemPoolProps props{};
  props.allocType = cudaMemAllocationTypePinned;
  props.handleTypes = cudaMemHandleTypeNone;
  props.location.type = cudaMemLocationTypeDevice;
  props.location.id = dev;
  cudaMemPool_t pool = nullptr;
  uint64_t kept = kKeptBytes;
  if (cudaMemPoolCreate(&pool, &props) != cudaSuccess) {
    cudaGetLastError();
    return nullptr;
  }
  if (cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &kept) != cudaSuccess) {
    cudaGetLastError();
    cudaMemPoolDestroy(pool);
    return nullptr;
  }
  slot.pool = pool;
  slot.ctx_id = ctx_id;
  return pool;
}

}  // namespace

cudaError_t scratch_pool(cudaMemPool_t* pool) {
  int dev = 0;
  cudaMemPool_t current = nullptr, standard = nullptr;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetMemPool(&current, dev);
  if (e == cudaSuccess) e = cudaDeviceGetDefaultMemPool(&standard, dev);
  if (e != cudaSuccess) return e;
  *pool = current;
  if (current == standard)
    if (cudaMemPool_t kept = kept_pool(false)) *pool = kept;
  return cudaSuccess;
}

cudaError_t scratch_malloc(void** p, size_t bytes, cudaStream_t st) {
  cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
  cudaError_t e = cudaStreamIsCapturing(st, &capture);
  if (e != cudaSuccess) return e;
  if (capture != cudaStreamCaptureStatusNone) return cudaMallocAsync(p, bytes, st);   // memory of the caller's graph
  cudaMemPool_t pool = nullptr;
  if ((e = scratch_pool(&pool)) != cudaSuccess) return e;
  e = cudaMallocFromPoolAsync(p, bytes, pool, st);
  if (e != cudaErrorMemoryAllocation) return e;
  cudaGetLastError();
  cudaMemPoolTrimTo(pool, 0);
  return cudaMallocAsync(p, bytes, st);
}

void scratch_reserve() { kept_pool(true); }

void scratch_trim() {
  if (cudaMemPool_t pool = kept_pool(false)) {
    if (cudaMemPoolTrimTo(pool, 0) != cudaSuccess) cudaGetLastError();
  }
}

}  // namespace deco
