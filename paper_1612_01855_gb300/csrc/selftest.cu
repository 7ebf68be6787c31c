// Self-tests of the bounded waits: each kernel waits on something that
// nothing will ever signal, with a short limit, and must give up, record the
// error and return (freeing the tensor memory it holds, with no copy under
// way) instead of hanging.
// They exercise the same wait routines as the solve kernels.
#include <cuda_runtime.h>

#include "internal.h"
#include "tc_engine.cuh"
#include "trsm_gb300.h"
#include "trsm_gb300_engine.h"
#include "wait.cuh"

namespace trsm {
namespace {

// A dependency-counter wait (as in the blocked and batched solves) on a
// counter that stays 0.
__global__ void counter_wait_selftest_kernel(const int* counter, int* err, long long limit_ns) {
  if (threadIdx.x == 0) wait_geq_bounded(counter, 1, err, 1, limit_ns, 1LL << 40, 2048);
}

// An mbarrier wait (as in the tcgen05 kernels) on a barrier that never
// receives its arrival, by a CTA that holds tensor memory.
__global__ void mbarrier_wait_selftest_kernel(int* err, long long limit_ns) {
  __shared__ uint64_t bar;
  __shared__ uint32_t tbase;
  __shared__ int abort_sh;
  const int warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) {
    tc::mbar_init(&bar, 1);
    abort_sh = 0;
    tc::fence_mbar_init();
  }
  if (warp == 0) {
    tc::tmem_alloc(&tbase, 32);
    tc::tmem_relinquish();
  }
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  if (threadIdx.x == 0) tc::mbar_wait_limit(&bar, 0, &abort_sh, limit_ns);
  __syncthreads();
  if (warp == 0) {
    tc::tc_fence_after();
    tc::tmem_dealloc(tbase, 32);
  }
  if (threadIdx.x == 0 && abort_sh) atomicExch(err, 1);
}

// A ring of bulk copies (as in the solve by columns) whose consumer never
// gives a stage back: the loader gives up and drains the copies it has issued.
// *err: 1 when they were all there by then, else 2.
__global__ void ring_selftest_kernel(const unsigned char* src, int* err, long long limit_ns) {
  constexpr int kStages = 3, kBytes = 8192;
  __shared__ __align__(128) unsigned char buf[kStages * kBytes];
  __shared__ uint64_t full_bar[kStages], empty_bar;
  __shared__ int abort_sh, same_sh;
  if (threadIdx.x == 0) {
    for (int q = 0; q < kStages; ++q) tc::mbar_init(&full_bar[q], 1);
    tc::mbar_init(&empty_bar, 1);
    abort_sh = 0;
    same_sh = 1;
    tc::fence_mbar_init();
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int q = 0; q < kStages; ++q) {
      tc::mbar_arrive_expect_tx(&full_bar[q], kBytes);
      tc::bulk_load(buf + q * kBytes, src + q * kBytes, kBytes, &full_bar[q]);
    }
    if (!tc::mbar_wait_limit(&empty_bar, 0, &abort_sh, limit_ns)) tc::drain_ring(full_bar, kStages, kStages);
    for (int q = 0; q < kStages; ++q)
      if (!tc::mbar_try_wait(&full_bar[q], 0)) same_sh = 0;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < kStages * kBytes; i += blockDim.x)
    if (buf[i] != src[i]) same_sh = 0;
  __syncthreads();
  if (threadIdx.x == 0 && abort_sh) atomicExch(err, same_sh ? 1 : 2);
}

// A wait for another CTA of the cluster (as in the solve by columns) that
// sends nothing; both leave the cluster together.
__global__ void __cluster_dims__(2, 1, 1) cluster_wait_selftest_kernel(int* err, long long limit_ns) {
  __shared__ uint64_t bar;
  __shared__ int abort_sh;
  if (threadIdx.x == 0) {
    tc::mbar_init(&bar, 1);
    abort_sh = 0;
    tc::fence_mbar_init();
  }
  __syncthreads();
  tc::cluster_sync();
  if (threadIdx.x == 0 && tc::cluster_rank() == 0) tc::mbar_wait_cluster(&bar, 0, &abort_sh, limit_ns);
  __syncthreads();
  tc::cluster_sync();
  if (threadIdx.x == 0 && abort_sh) atomicExch(err, 1);
}

constexpr size_t kRingBytes = 3 * 8192;

}  // namespace
}  // namespace trsm

extern "C" int trsm_wait_selftest(int kind, int64_t limit_us, void* stream) {
  if ((kind != 0 && kind != 1 && kind != 3 && kind != 4) || limit_us < 1 || limit_us > 2000000) return TRSM_EINVAL;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  int* buf = nullptr;  // [0]: the counter nobody raises, [1]: the error word; from 256 bytes on: the ring's source
  cudaError_t e = trsm::ws_alloc(reinterpret_cast<void**>(&buf), 256 + trsm::kRingBytes, s);
  if (e != cudaSuccess) return TRSM_ENOMEM;
  e = cudaMemsetAsync(buf, 0, 2 * sizeof(int), s);
  unsigned char* src = reinterpret_cast<unsigned char*>(buf) + 256;
  if (e == cudaSuccess) e = cudaMemsetAsync(src, 0x5A, trsm::kRingBytes, s);
  const long long limit_ns = static_cast<long long>(limit_us) * 1000;
  if (e == cudaSuccess) {
    if (kind == 0)
      trsm::counter_wait_selftest_kernel<<<1, 32, 0, s>>>(buf, buf + 1, limit_ns);
    else if (kind == 1)
      trsm::mbarrier_wait_selftest_kernel<<<1, 64, 0, s>>>(buf + 1, limit_ns);
    else if (kind == 3)
      trsm::ring_selftest_kernel<<<1, 256, 0, s>>>(src, buf + 1, limit_ns);
    else
      trsm::cluster_wait_selftest_kernel<<<2, 32, 0, s>>>(buf + 1, limit_ns);
    trsm::count_launch();
    e = cudaGetLastError();
  }
  int h_err = 0;
  if (e == cudaSuccess) e = cudaMemcpyAsync(&h_err, buf + 1, sizeof(int), cudaMemcpyDeviceToHost, s);
  trsm::ws_free(buf, s);
  cudaError_t e2 = cudaStreamSynchronize(s);
  if (e == cudaSuccess) e = e2;
  if (e != cudaSuccess) {
    cudaGetLastError();
    return TRSM_ECUDA;
  }
  if (h_err > 1) return TRSM_ECUDA;  // copies were still under way after the drain
  return h_err ? TRSM_ETIMEOUT : TRSM_SUCCESS;
}
