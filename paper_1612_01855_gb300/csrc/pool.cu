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
// trims the pool and retries once.
// Small plans' L~ comes from blocks that destroyed plans leave to the next
// ones, kKeepPlans of them at most.  The blocks are cudaMalloc's, not a
// memory pool's: a caller may share trsm_plan_lt's pointer by CUDA IPC or with
// a peer device.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_runtime.h>

#include <mutex>
#include <utility>
#include <vector>

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
  std::vector<std::pair<void*, size_t>> idle;  // blocks of destroyed plans, the oldest first
  size_t idle_bytes = 0, live_bytes = 0;       // of those, and of the blocks that plans hold
  bool anchored = false;  // keep_small_block has run in this context
};

std::mutex g_pool_mutex;
DevicePool g_pools[kMaxDevices];

cudaError_t make_pool(int dev, cudaMemPool_t* out) {
  cudaMemPoolProps props = {};
  props.allocType = cudaMemAllocationTypePinned;
  props.handleTypes = cudaMemHandleTypeNone;
  props.location.type = cudaMemLocationTypeDevice;
  props.location.id = dev;
  cudaMemPool_t p = nullptr;
  cudaError_t e = cudaMemPoolCreate(&p, &props);
  if (e != cudaSuccess) return e;
  unsigned long long keep = ~0ull;
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

// The pool of the current device, made at its first use in the current
// context; g_pools[*device] is of that context then.  Those of an earlier
// context (before a cudaDeviceReset) went away with that context, the plans'
// blocks too, and are not destroyed again.
cudaError_t current_pool(cudaMemPool_t* out, int* device = nullptr) {
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
    e = make_pool(dev, &fresh.pool);
    if (e != cudaSuccess) return e;
    d = std::move(fresh);
  }
  *out = d.pool;
  if (device) *device = dev;
  return cudaSuccess;
}

// cudaFrees the oldest idle blocks of a device until at most `keep` bytes of
// them are left.  Not under the lock: cudaFree may wait for the device.
void free_idle_blocks(int dev, size_t keep) {
  for (;;) {
    void* p = nullptr;
    {
      std::lock_guard<std::mutex> lock(g_pool_mutex);
      DevicePool& d = g_pools[dev];
      if (d.idle.empty() || d.idle_bytes <= keep) return;
      p = d.idle.front().first;
      d.idle_bytes -= d.idle.front().second;
      d.idle.erase(d.idle.begin());
    }
    cudaFree(p);
  }
}

// Returns what the library holds idle on a device, so that an allocation that
// failed may be tried again.
void release_idle(cudaMemPool_t pool, int dev) {
  cudaGetLastError();
  cudaMemPoolTrimTo(pool, 0);
  free_idle_blocks(dev, 0);
}

// Size of a plan's block: the granularity in which cudaMalloc maps memory,
// less for those it cuts from one mapping.
size_t block_bytes(size_t bytes) {
  const size_t g = bytes <= (size_t)1 << 20 ? (size_t)64 << 10 : (size_t)2 << 20;
  return (bytes + g - 1) / g * g;
}

}  // namespace

cudaError_t ws_alloc(void** p, size_t bytes, cudaStream_t s) {
  *p = nullptr;
  cudaMemPool_t pool = nullptr;
  int dev = 0;
  cudaError_t e = current_pool(&pool, &dev);
  if (e != cudaSuccess) return e;
  e = cudaMallocFromPoolAsync(p, bytes, pool, s);
  if (e == cudaErrorMemoryAllocation) {
    // cudaFree is not for a capturing thread: the idle blocks stay then
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusActive;
    if (cudaStreamIsCapturing(s, &cap) == cudaSuccess && cap == cudaStreamCaptureStatusNone) {
      release_idle(pool, dev);
    } else {
      cudaGetLastError();
      cudaMemPoolTrimTo(pool, 0);
    }
    e = cudaMallocFromPoolAsync(p, bytes, pool, s);
  }
  return e;
}

cudaError_t plan_alloc(void** p, size_t bytes, PlanBlock* block) {
  *p = nullptr;
  cudaMemPool_t pool = nullptr;
  int dev = 0;
  cudaError_t e = current_pool(&pool, &dev);
  if (e != cudaSuccess) return e;
  const size_t need = block_bytes(bytes);
  {
    std::lock_guard<std::mutex> lock(g_pool_mutex);
    DevicePool& d = g_pools[dev];
    block->bytes = need;
    block->ctx_id = d.ctx_id;
    for (size_t i = d.idle.size(); i-- > 0;) {  // the latest first
      if (d.idle[i].second != need) continue;
      *p = d.idle[i].first;
      d.idle.erase(d.idle.begin() + i);
      d.idle_bytes -= need;
      d.live_bytes += need;
      return cudaSuccess;
    }
  }
  e = cudaMalloc(p, need);
  if (e == cudaErrorMemoryAllocation) {
    release_idle(pool, dev);
    e = cudaMalloc(p, need);
  }
  if (e != cudaSuccess) return e;
  std::lock_guard<std::mutex> lock(g_pool_mutex);
  if (g_pools[dev].ctx_id == block->ctx_id) g_pools[dev].live_bytes += need;
  return cudaSuccess;
}

void plan_free(void* p, const PlanBlock& block, bool unused) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) dev = 0;
  const unsigned long long id = current_context_id();
  if (id != block.ctx_id) return;  // it went away with its context
  bool kept = false;
  {
    std::lock_guard<std::mutex> lock(g_pool_mutex);
    DevicePool& d = g_pools[dev];
    if (id != 0 && id == d.ctx_id) {  // without an id nothing is kept
      d.live_bytes -= block.bytes;
      if (unused) try {
          d.idle.emplace_back(p, block.bytes);
          d.idle_bytes += block.bytes;
          kept = true;
        } catch (...) {  // no host memory for the entry
        }
    }
  }
  if (!kept) cudaFree(p);
  else free_idle_blocks(dev, kKeepPlans);
}

// cudaMalloc cuts small allocations from blocks of a few MB, which cudaFree
// unmaps when the last one in them goes.  A plan's status word would
// otherwise map and unmap such a block each time: a 64 x 64 plan took 187 us
// to make and 62 us to destroy, 88 and 4 us with the block kept.  One word
// per device and context is never freed.
void keep_small_block() {
  cudaMemPool_t pool = nullptr;
  int dev = 0;
  if (current_pool(&pool, &dev) != cudaSuccess) return;
  std::lock_guard<std::mutex> lock(g_pool_mutex);
  DevicePool& d = g_pools[dev];
  if (d.anchored || d.pool != pool) return;
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
  cudaMemPool_t pool = nullptr;
  {
    std::lock_guard<std::mutex> lock(trsm::g_pool_mutex);
    const trsm::DevicePool& d = trsm::g_pools[dev];
    if (d.pool == nullptr || d.ctx_id != trsm::current_context_id()) return TRSM_SUCCESS;  // nothing held
    pool = d.pool;
  }
  // keep_bytes in all: the workspaces' pool first, the idle blocks what is left
  unsigned long long held = 0;
  cudaError_t e = cudaMemPoolTrimTo(pool, keep_bytes);
  if (e == cudaSuccess) e = cudaMemPoolGetAttribute(pool, cudaMemPoolAttrReservedMemCurrent, &held);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return TRSM_ECUDA;
  }
  size_t live = 0;
  {
    std::lock_guard<std::mutex> lock(trsm::g_pool_mutex);
    live = trsm::g_pools[dev].live_bytes;
  }
  trsm::free_idle_blocks(dev, keep_bytes > held + live ? keep_bytes - held - live : 0);
  cudaGetLastError();
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
  unsigned long long v = 0;
  if (cudaMemPoolGetAttribute(d.pool, cudaMemPoolAttrReservedMemCurrent, &v) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return static_cast<size_t>(v) + d.idle_bytes + d.live_bytes;
}
