// Device memory of the library's per-call workspaces.
//
// Every solve, plan and batch run takes its scratch (the working copy of B,
// residues, dependency counters, partial sums) from a stream-ordered
// memory pool owned by the library, one per device and CUDA context.  The
// pool differs from the device's default pool in two settings:
//   - its release threshold is unbounded: memory freed by a call stays
//     mapped for the next one.  The default pool returns freed memory to the
//     system at every synchronisation, and the next call pays the mapping of
//     its workspace again (about 1 ms per GB: a third of a 30 ms solve whose
//     workspace is 6 GB);
//   - reuse across streams through dependencies the driver inserts itself is
//     off: a block freed on one stream and still pending there is not handed
//     to another stream (the pool grows instead), so that concurrent solves
//     on separate streams are never ordered behind one another by their
//     scratch.  A block whose free has completed is reused on any stream.
// trsm_workspace_trim hands the idle memory back; an allocation that fails
// trims the pools and retries once.
// Small plans' L~ comes from a second pool, so that a plan's block does not
// sit in the middle of the workspaces' memory.  Destroyed plans leave at most
// kKeepPlans of it mapped: a program that held thousands of plans gets the
// rest back at its next synchronisation.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_runtime.h>

#include <mutex>

#include "internal.h"
#include "trsm_gb300.h"

namespace trsm {

unsigned long long current_context_id() {
  static PFN_cuCtxGetCurrent_v4000 get_current = nullptr;
  static PFN_cuCtxGetId_v12000 get_id = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &p, 4000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      get_current = reinterpret_cast<PFN_cuCtxGetCurrent_v4000>(p);
    if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      get_id = reinterpret_cast<PFN_cuCtxGetId_v12000>(p);
  });
  if (!get_current || !get_id) return 0;
  CUcontext ctx = nullptr;
  unsigned long long id = 0;
  if (get_current(&ctx) != CUDA_SUCCESS || ctx == nullptr) return 0;
  if (get_id(ctx, &id) != CUDA_SUCCESS) return 0;
  return id;
}

namespace {

constexpr int kMaxDevices = 64;
constexpr unsigned long long kKeepPlans = 256ull << 20;

struct DevicePool {
  unsigned long long ctx_id = 0;  // context the pool was made in (0: none yet)
  cudaMemPool_t pool = nullptr;
  cudaMemPool_t plans = nullptr;
  bool anchored = false;  // keep_small_block has run in this context
};

std::mutex g_pool_mutex;
DevicePool g_pools[kMaxDevices];

cudaError_t make_pool(int dev, unsigned long long keep, cudaMemPool_t* out) {
  cudaMemPoolProps props = {};
  props.allocType = cudaMemAllocationTypePinned;
  props.handleTypes = cudaMemHandleTypeNone;
  props.location.type = cudaMemLocationTypeDevice;
  props.location.id = dev;
  cudaMemPool_t p = nullptr;
  cudaError_t e = cudaMemPoolCreate(&p, &props);
  if (e != cudaSuccess) return e;
  int no = 0;
  e = cudaMemPoolSetAttribute(p, cudaMemPoolAttrReleaseThreshold, &keep);
  if (e == cudaSuccess) e = cudaMemPoolSetAttribute(p, cudaMemPoolReuseAllowInternalDependencies, &no);
  if (e != cudaSuccess) {
    cudaMemPoolDestroy(p);
    return e;
  }
  *out = p;
  return cudaSuccess;
}

// The pools of the current device, made at their first use in the current
// context.  Those of an earlier context (before a cudaDeviceReset) went away
// with that context and are not destroyed again.
cudaError_t current_pools(DevicePool* out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  unsigned long long id = current_context_id();
  if (id == 0) {
    e = cudaFree(nullptr);  // makes the device's primary context current
    if (e != cudaSuccess) return e;
    id = current_context_id();
  }
  std::lock_guard<std::mutex> lock(g_pool_mutex);
  DevicePool& d = g_pools[dev];
  if (d.pool == nullptr || id == 0 || id != d.ctx_id) {
    DevicePool fresh;
    fresh.ctx_id = id;
    e = make_pool(dev, ~0ull, &fresh.pool);
    if (e != cudaSuccess) return e;
    e = make_pool(dev, kKeepPlans, &fresh.plans);
    if (e != cudaSuccess) {
      cudaMemPoolDestroy(fresh.pool);
      return e;
    }
    d = fresh;
  }
  *out = d;
  return cudaSuccess;
}

cudaError_t alloc_from(cudaMemPool_t DevicePool::*which, void** p, size_t bytes, cudaStream_t s) {
  *p = nullptr;
  DevicePool d;
  cudaError_t e = current_pools(&d);
  if (e != cudaSuccess) return e;
  e = cudaMallocFromPoolAsync(p, bytes, d.*which, s);
  if (e == cudaErrorMemoryAllocation) {
    cudaGetLastError();
    cudaMemPoolTrimTo(d.pool, 0);
    cudaMemPoolTrimTo(d.plans, 0);
    e = cudaMallocFromPoolAsync(p, bytes, d.*which, s);
  }
  return e;
}

}  // namespace

cudaError_t ws_alloc(void** p, size_t bytes, cudaStream_t s) { return alloc_from(&DevicePool::pool, p, bytes, s); }

cudaError_t plan_alloc(void** p, size_t bytes, cudaStream_t s) { return alloc_from(&DevicePool::plans, p, bytes, s); }

// cudaMalloc cuts small allocations from blocks of a few MB, which cudaFree
// unmaps when the last one in them goes.  A plan's status word would
// otherwise map and unmap such a block each time: a 64 x 64 plan took 187 us
// to make and 62 us to destroy, 88 and 4 us with the block kept.  One word
// per device and context is never freed.
void keep_small_block() {
  DevicePool now;
  if (current_pools(&now) != cudaSuccess || now.anchored) return;
  int dev = 0;
  cudaGetDevice(&dev);
  std::lock_guard<std::mutex> lock(g_pool_mutex);
  DevicePool& d = g_pools[dev];
  if (d.anchored || d.pool != now.pool) return;
  void* word = nullptr;
  if (cudaMalloc(&word, sizeof(int)) != cudaSuccess) {
    cudaGetLastError();
    return;
  }
  d.anchored = true;
}

cudaError_t ws_free(void* p, cudaStream_t s) { return p ? cudaFreeAsync(p, s) : cudaSuccess; }

}  // namespace trsm

extern "C" int trsm_workspace_trim(size_t keep_bytes) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= trsm::kMaxDevices) {
    cudaGetLastError();
    return TRSM_ECUDA;
  }
  trsm::DevicePool now;
  {
    std::lock_guard<std::mutex> lock(trsm::g_pool_mutex);
    const trsm::DevicePool& d = trsm::g_pools[dev];
    if (d.pool == nullptr || d.ctx_id != trsm::current_context_id()) return TRSM_SUCCESS;  // nothing held
    now = d;
  }
  // keep_bytes in all: the workspaces' pool first, the plans' what is left
  unsigned long long held = 0;
  cudaError_t e = cudaMemPoolTrimTo(now.pool, keep_bytes);
  if (e == cudaSuccess) e = cudaMemPoolGetAttribute(now.pool, cudaMemPoolAttrReservedMemCurrent, &held);
  if (e == cudaSuccess) e = cudaMemPoolTrimTo(now.plans, held < keep_bytes ? keep_bytes - held : 0);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return TRSM_ECUDA;
  }
  return TRSM_SUCCESS;
}

extern "C" size_t trsm_workspace_reserved_bytes(void) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= trsm::kMaxDevices) {
    cudaGetLastError();
    return 0;
  }
  std::lock_guard<std::mutex> lock(trsm::g_pool_mutex);
  const trsm::DevicePool& d = trsm::g_pools[dev];
  if (d.pool == nullptr || d.ctx_id != trsm::current_context_id()) return 0;
  unsigned long long v = 0, w = 0;
  if (cudaMemPoolGetAttribute(d.pool, cudaMemPoolAttrReservedMemCurrent, &v) != cudaSuccess ||
      cudaMemPoolGetAttribute(d.plans, cudaMemPoolAttrReservedMemCurrent, &w) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return static_cast<size_t>(v + w);
}
