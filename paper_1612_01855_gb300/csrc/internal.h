// Internal declarations shared by the library's translation units.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <vector>

#include "trsm_gb300.h"

namespace trsm {
struct MixedPlan;
struct SlicedPlan;
// A block of device memory that passes from plan to plan (pool.cu); 0 bytes: none.
struct PlanBlock {
  size_t bytes = 0;
  unsigned long long ctx_id = 0;  // context it was made in
};
}

// The plan behind trsm_handle_t.
struct trsm_plan_s {
  int64_t n = 0, n0 = 0, N = 0, ldt = 0;
  double* Lt = nullptr;   // L~: n x n, leading dimension ldt
  int* status = nullptr;  // sticky device status of solves
  int device = 0;
  trsm::PlanBlock lt_block;  // where Lt is a block of plan_alloc
  trsm::MixedPlan* mixed = nullptr;    // low-precision data (trsm_plan_mixed), or null
  trsm::SlicedPlan* sliced = nullptr;  // residues of the sliced schedule (trsm_plan_sliced), or null
};

namespace trsm {

// Frees the mixed-precision part of a plan (no-op when absent).
// Device bytes of the plan's mixed-precision data (0 without it).
size_t mixed_bytes(const trsm_plan_s* h);
void mixed_release(trsm_plan_s* h);
// The same for the residues of the sliced schedule.
size_t sliced_bytes(const trsm_plan_s* h);
void sliced_release(trsm_plan_s* h);
// X = L^-1 B by the sliced schedule (sched_sliced.cu).  X may alias B (same
// leading dimension): the first step reads every row of B and keeps the later
// rows' updates in the workspace before any other row of X is written.
int solve_sliced(trsm_plan_s* h, const double* B, int64_t k, int64_t ldb, double* X, int64_t ldx,
                 cudaStream_t s);

// A diagonal block to invert in place: top-left element at A + off, order m;
// row0 is its first row in the caller's numbering (for singular reports).
struct DiagBlock {
  int64_t off;
  int64_t m;
  int64_t row0;
};

// Inverts every listed diagonal block of A (leading dimension ld) in place
// by recursive triangular inversion; the strict upper triangle of each block
// must hold zeros on entry.  The smallest row index with a zero or non-finite
// pivot is folded (atomic min) into *sing_dev.  Asynchronous on `s`;
// allocates its scratch stream-ordered.  `host` takes the descriptors that a
// copy on `s` reads: the caller keeps it until `s` has been waited for.
// Returns a cudaError_t.
cudaError_t invert_diag_blocks(double* A, int64_t ld, const std::vector<DiagBlock>& blocks,
                               unsigned long long* sing_dev, std::vector<unsigned char>& host, cudaStream_t s);

// Lt(i, j) = (i >= j) ? L(i, j) : 0 for an n x n matrix.
cudaError_t copy_lower(const double* L, int64_t ldl, double* Lt, int64_t ldt, int64_t n,
                       cudaStream_t s);

// Packs the diagonal blocks of L into P (N blocks of n0 x n0, ld n0),
// lower triangle only, zero elsewhere.
cudaError_t pack_diag_blocks(const double* L, int64_t ldl, double* P, int64_t n, int64_t n0,
                             cudaStream_t s);

// W (n x k, ldw) = B (n x k, ldb).
// Zeroes the strictly upper part of the n0 x n0 diagonal blocks of Lt.
cudaError_t zero_upper_blocks(double* Lt, int64_t ldt, int64_t n, int64_t n0, cudaStream_t s);

cudaError_t copy_panel(const double* B, int64_t ldb, double* W, int64_t ldw, int64_t n,
                       int64_t k, cudaStream_t s);

// Solve with a planned L~: see solve.cu.
size_t solve_workspace_bytes(int64_t n, int64_t n0, int64_t k);
cudaError_t solve_enqueue(const double* Lt, int64_t ldt, int64_t n, int64_t n0, const double* B,
                          int64_t k, int64_t ldb, double* X, int64_t ldx, void* ws,
                          int* status_dev, cudaStream_t s);

// The solve by columns (solve_cols.cu): CW columns per group, S CTAs per
// group; use: whether it is expected to be faster than the tile tasks.
struct ColPlan {
  bool use = false;
  int S = 0, CW = 0, stages = 0;
  size_t smem = 0;
};
ColPlan col_plan(int64_t n, int64_t n0, int64_t k);
// The plan with a given S and CW; S is 0 where that cannot run.
ColPlan col_plan_as(int64_t n, int64_t n0, int64_t k, int S, int CW);
cudaError_t col_solve(const ColPlan& p, const double* Lt, int64_t ldt, int64_t n, int64_t n0, const double* B, int64_t k,
                      int64_t ldb, double* X, int64_t ldx, int* status_dev, cudaStream_t s);

// The solve by whichever of the two is expected to be faster (cols is col_plan
// of n, n0 and k); ws may be null when that is the one by columns.
cudaError_t solve_any(const ColPlan& cols, const double* Lt, int64_t ldt, int64_t n, int64_t n0, const double* B,
                      int64_t k, int64_t ldb, double* X, int64_t ldx, void* ws, int* status_dev, cudaStream_t s);

// Device status word and device ordinal of a plan (for entry points that
// live outside api.cu).
int* plan_status_word(trsm_handle_t h);
int plan_device(trsm_handle_t h);

// Stream-ordered device allocations of the library's workspaces.  They come
// from a library-owned memory pool of the current device that keeps freed
// memory for reuse: the device's default pool returns freed memory to the
// system at every synchronisation, and a large workspace then pays its
// mapping again at each call (about 1 ms per GB).  trsm_workspace_trim
// returns the pool's idle memory (pool.cu).
cudaError_t ws_alloc(void** p, size_t bytes, cudaStream_t s);
// Memory of a plan, cudaMalloc's, from the blocks that destroyed plans left
// where one fits.  plan_free gives it back; unused: the device has finished all
// work that may use it, so that the next plan may have it.  keep_small_block
// makes cudaMalloc and cudaFree of single words cheap.
cudaError_t plan_alloc(void** p, size_t bytes, PlanBlock* block);
void plan_free(void* p, const PlanBlock& block, bool unused);
void keep_small_block();
cudaError_t ws_free(void* p, cudaStream_t s);
template <class T>
cudaError_t ws_alloc(T** p, size_t bytes, cudaStream_t s) {
  return ws_alloc(reinterpret_cast<void**>(p), bytes, s);
}

// A kernel launched with programmatic dependence on the one before it in the
// stream: it may be set up while that one still runs, and must call
// grid_dependency_wait before it touches global memory (in every CTA, before
// any return, so that its end implies the end of its predecessors).  The
// kernel before it lets it start early by calling grid_launch_dependents: the
// short element-wise kernels of a chain do, so that the tensor-core kernel
// after them finds its barriers and tensor memory set up.  The tensor-core
// kernels do not: CTAs that wait beside them slow them down (n = 16384, k =
// 256, sliced, us: 1298 without any of this, 1327 with both kinds letting go
// early, 1218 with the element-wise ones alone; refined n = 3000, k = 128:
// 1295, 965, 925), and a CTA that waits must not hold tensor memory that one
// of them still has to get.
// Such a kernel runs beside the ones before it, so nothing they write is
// read-only for its lifetime: it reads by plain loads, after its wait. No
// __ldg and no const __restrict__ pointer (either allows the read-only path,
// which need not see those writes, and a load that moves above the wait).
// cluster: CTAs per cluster (1: none).
template <class... KArgs, class... Args>
cudaError_t launch_dependent(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                             unsigned cluster, Args&&... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[2]{};
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = cluster;
  at[1].val.clusterDim.y = at[1].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = cluster > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, kern, static_cast<KArgs>(args)...);
}

#ifdef __CUDACC__
__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
#endif

// Unique id of the calling thread's current CUDA context (0 if none is
// current or the driver entry points are unavailable): caches of device
// addresses and pools are keyed by it, so that they are remade after a
// cudaDeviceReset.
unsigned long long current_context_id();

// Launch accounting (every kernel launch of the library goes through here).
void count_launch(int64_t n = 1);

// Number of SMs and CTAs per SM of the persistent solve kernel on the
// current device (cached per device).
int device_sm_count();

}  // namespace trsm
