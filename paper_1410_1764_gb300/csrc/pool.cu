// Device memory that calls take and give back in stream order: derivative
// fields of single BSSN right-hand sides, stages and constraints, the adjoint's
// work space.  One pool per device, shared by all systems, so that a new system
// finds mapped memory (with a pool of its own its first right-hand side of 16^3
// points took 281 us, its second 106).  The pool is never destroyed: a system may
// be destroyed while a call that used the pool is still running, and destroying
// a pool with a free outstanding crashed the process (NVIDIA driver 580.159).
#include <mutex>

#include "internal.h"

namespace chemora {

// Memory kept for later calls while a system exists (the adjoint of 50 steps on
// 128^3, checkpoints every 10, takes 3.4 GB), and when none does (a right-hand
// side of 50,000 points); more than that goes back to the device at the next
// synchronisation.
constexpr uint64_t kPoolKeep = (uint64_t)4 << 30, kPoolIdle = (uint64_t)64 << 20;

constexpr int kPoolDevices = 64;
static std::mutex g_pool_mu;
static cudaMemPool_t g_pool[kPoolDevices];
static int64_t g_pool_systems;

static void set_keep(cudaMemPool_t pool, uint64_t keep) {
  cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep);
}

// The current device's pool, made on first use; NULL: none could be made.
static cudaMemPool_t device_pool(bool create) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kPoolDevices) {
    cudaGetLastError();
    return nullptr;
  }
  const std::lock_guard<std::mutex> lock(g_pool_mu);
  if (g_pool[dev] || !create) return g_pool[dev];
  cudaMemPoolProps props = {};
  props.allocType = cudaMemAllocationTypePinned;
  props.location.type = cudaMemLocationTypeDevice;
  props.location.id = dev;
  cudaMemPool_t pool = nullptr;
  if (cudaMemPoolCreate(&pool, &props) != cudaSuccess) {
    cudaGetLastError();
    return nullptr;
  }
  // a call never waits for one on another stream to give its memory back
  int off = 0;
  cudaMemPoolSetAttribute(pool, cudaMemPoolReuseAllowInternalDependencies, &off);
  set_keep(pool, g_pool_systems > 0 ? kPoolKeep : kPoolIdle);
  return g_pool[dev] = pool;
}

cudaError_t pool_alloc(void** p, size_t bytes, cudaStream_t s) {
  const cudaMemPool_t pool = device_pool(true);
  const cudaError_t e = pool ? cudaMallocFromPoolAsync(p, bytes, pool, s) : cudaMallocAsync(p, bytes, s);
  if (e != cudaSuccess) cudaGetLastError();
  return e;
}

void pool_free(void* p, cudaStream_t s) { cudaFreeAsync(p, s); }

void pool_count_systems(int by) {
  const std::lock_guard<std::mutex> lock(g_pool_mu);
  const bool had = g_pool_systems > 0;
  g_pool_systems += by;
  const bool has = g_pool_systems > 0;
  if (had == has) return;
  for (cudaMemPool_t pool : g_pool)
    if (pool) {
      set_keep(pool, has ? kPoolKeep : kPoolIdle);
      if (!has) cudaMemPoolTrimTo(pool, kPoolIdle);
    }
}

cudaError_t device_alloc(void** p, size_t bytes) {
  cudaError_t e = cudaMalloc(p, bytes);
  const cudaMemPool_t pool = e == cudaErrorMemoryAllocation ? device_pool(false) : nullptr;
  if (!pool) return e;
  cudaGetLastError();
  cudaMemPoolTrimTo(pool, 0);
  return cudaMalloc(p, bytes);
}

}  // namespace chemora
