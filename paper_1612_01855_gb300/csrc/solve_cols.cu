// Blocked solve by columns: Algorithm It-Inv-TRSM (Section 6.2) with every
// few columns of the right-hand side solved by one CTA, or by a cluster of
// CTAs, on their own.
//
// The columns of X are independent (Section 2.3.4), and GB300's FP64 pipe is
// so narrow (2 multiply-adds per SM and clock) that a CTA can stream all of
// L~ from L2 for one or a few columns without the loads mattering: 8 / CW
// bytes per multiply-add, at most 16 bytes per SM and clock.  So where the
// tile tasks of solve.cu are bound by their dependency chain (a 32 x 32
// tile's chunk of 32 takes 8 us on an SM, and a block row takes two tasks of
// n0 / 32 chunks one after the other, plus their waits), the columns are
// dealt to the SMs instead, with no dependency between groups of CTAs.
//
// Right-looking: once X_b = L~_bb W_b is known, W_l -= L_lb X_b for every
// l > b.  With fewer columns than SMs the S CTAs of a cluster share a column
// group: CTA r owns the block rows l = r (mod S), keeps their W_l in its
// shared memory and gets every X_b from its owner (distributed shared
// memory).  The owner of block row b + 1 updates it first and sends X_{b+1}
// before it goes on with its other rows, so that the chain of block rows is
// two products of order n0 and a signal long.
//
// Every sum is the one of the tile tasks and of the batched launch (a fused
// multiply-add chain over a block column in increasing index from zero, the
// blocks subtracted in increasing order): the results are the same bits.
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cmath>

#include "internal.h"
#include "tc_engine.cuh"

namespace trsm {

namespace {

constexpr int kWarps = 8;                      // consumers; one more warp loads
constexpr int kThreads = 32 * (kWarps + 1);
constexpr int kMaxRows = 32 * kWarps;          // longest block: a row group per warp
constexpr int kStageDoubles = 4096;            // 32 KB of L~ per stage
constexpr int kMaxStages = 6;
constexpr int kMaxCluster = 8;                 // the portable cluster size
constexpr int kMaxCols = 8;                    // columns of a group
constexpr size_t kMaxShared = 226 * 1024;

struct ColArgs {
  const double* Lt;
  int64_t ldt;
  const double* B;
  int64_t ldb;
  double* X;
  int64_t ldx;
  int64_t n, k;
  int n0, N;
  int S;         // CTAs per column group
  int RG;        // 32-row groups of a block
  int NB;        // block rows of a stage of the plain updates: as many as the warps cover
  int KC1, KCn;  // columns of a stage of one block row, and of NB
  int pitch;     // doubles per column of a block row in a stage
  int stages;
  int* status;
};

// Barrier among the consumers.
__device__ __forceinline__ void sync_consumers() {
  asm volatile("bar.sync 1, %0;" ::"n"(32 * kWarps) : "memory");
}

__device__ __forceinline__ void st_cluster(uint32_t addr, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(addr), "d"(v) : "memory");
}

// acc[i] += sum over c in [0, len) of st[c pitch] v[c CW + i G], i < M, in
// increasing c.  M is a constant: a multiply-add that a predicate switches
// off takes its turn in the narrow FP64 pipe all the same.
template <int CW, int M>
__device__ __forceinline__ void dot_columns(const double* st, int pitch, const double* v, int G, int len,
                                            double (&acc)[CW]) {
#pragma unroll 8
  for (int c = 0; c < len; ++c) {
    const double x = st[c * pitch];
#pragma unroll
    for (int i = 0; i < M; ++i) acc[i] = fma(x, v[c * CW + i * G], acc[i]);
  }
}

// Shared memory: the stages of L~, then W [own block rows][n0][CW] and xs
// [S + 1][n0][CW], the X_b that have arrived: an owner's next X_b waits for
// all its updates, so no CTA is ever more than S of them behind.
//
// The loading warp streams every piece of L~ the CTA needs, in the order it
// is needed, through a ring of 32 KB stages, a bulk copy per column and block
// row: it runs ahead of the dependency chain, so that a block row finds its
// operands in shared memory.  (Plain loads by the threads that use them,
// eight in flight each, moved 1 TB/s in all.)
template <int CW>
__global__ void __launch_bounds__(kThreads, 1) col_solve_kernel(const ColArgs a) {
  extern __shared__ __align__(16) double sm[];
  __shared__ uint64_t full_bar[kMaxStages], empty_bar[kMaxStages], x_bar[kMaxCluster + 1];
  __shared__ int abort_sh;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int S = a.S;
  const int rank = S > 1 ? static_cast<int>(tc::cluster_rank()) : 0;
  const int64_t j0 = static_cast<int64_t>(blockIdx.x / S) * CW;
  const int nc = static_cast<int>(min(static_cast<int64_t>(CW), a.k - j0));
  const int own = (a.N - rank + S - 1) / S;  // block rows rank, rank + S, ...
  const size_t block_doubles = static_cast<size_t>(a.n0) * CW;
  double* W = sm + static_cast<size_t>(a.stages) * kStageDoubles;
  double* xs = W + static_cast<size_t>((a.N + S - 1) / S) * block_doubles;  // the same place in every CTA
  volatile int* abort_flag = &abort_sh;
  auto rows_of = [&](int l) { return static_cast<int>(min(static_cast<int64_t>(a.n0), a.n - static_cast<int64_t>(l) * a.n0)); };
  // own block rows that X_b updates, the one of the chain aside: from this index on
  auto first_rest = [&](int b) {
    const int l = (b + 1) % S == rank ? b + 2 : b + 1;
    return l <= rank ? 0 : (l - rank + S - 1) / S;
  };
  if (tid == 0) {
    abort_sh = 0;
    for (int q = 0; q < a.stages; ++q) {
      tc::mbar_init(&full_bar[q], 1);
      tc::mbar_init(&empty_bar[q], kWarps);
    }
    for (int q = 0; q <= S; ++q) tc::mbar_init(&x_bar[q], 1);
    tc::fence_mbar_init();
  }
  __syncthreads();
  if (S > 1) tc::cluster_sync();

  if (warp == kWarps) {
    int it = 0;
    bool ok = true;
    // columns [c0, c0 + cols) of L~ in the own block rows of index [t0, t1)
    // (the first of which goes to place t0 - base of the stage)
    auto stage = [&](int64_t c0, int cols, int t0, int t1, int base, int kc) {
      const int q = it % a.stages;
      ok = it < a.stages || tc::mbar_wait(&empty_bar[q], ((it / a.stages) - 1) & 1, abort_flag);
      if (!ok) return;
      uint32_t bytes = 0;  // whole pairs of rows, up to the even leading dimension
      for (int t = t0; t < t1; ++t) bytes += static_cast<uint32_t>((rows_of(rank + S * t) + 1) / 2 * 16 * cols);
      if (lane == 0) tc::mbar_arrive_expect_tx(&full_bar[q], bytes);
      __syncwarp();
      for (int t = t0; t < t1; ++t) {
        const int l = rank + S * t;
        const uint32_t b = static_cast<uint32_t>((rows_of(l) + 1) / 2 * 16);
        double* dst = sm + static_cast<size_t>(q) * kStageDoubles + static_cast<size_t>((t - base) * kc) * a.pitch;
        for (int c = lane; c < cols; c += 32)
          tc::bulk_load(dst + static_cast<size_t>(c) * a.pitch, a.Lt + (c0 + c) * a.ldt + static_cast<int64_t>(l) * a.n0, b,
                        &full_bar[q]);
      }
      ++it;
    };
    auto one = [&](int l, int b) {  // L_lb for an own l, up to the diagonal
      const int cols = rows_of(b), t = l / S;
      for (int q = 0; q < cols && ok; q += a.KC1)
        stage(static_cast<int64_t>(b) * a.n0 + q, min(a.KC1, cols - q), t, t + 1, t, a.KC1);
    };
    if (rank == 0) one(0, 0);
    for (int b = 0; b + 1 < a.N && ok; ++b) {
      if ((b + 1) % S == rank) {
        one(b + 1, b);
        one(b + 1, b + 1);
      }
      const int t0 = first_rest(b);
      for (int g = t0 / a.NB; t0 < own && g * a.NB < own && ok; ++g)
        for (int q = 0; q < a.n0 && ok; q += a.KCn)
          stage(static_cast<int64_t>(b) * a.n0 + q, min(a.KCn, a.n0 - q), max(t0, g * a.NB), min(own, (g + 1) * a.NB),
                g * a.NB, a.KCn);
    }
    if (!ok && lane == 0) tc::drain_ring(full_bar, a.stages, it);
  } else {
    int it = 0;
    bool ok = true;
    // Two divisions of the work.  The plain updates: a warp takes 32 rows of
    // one of NB block rows, every column.  The chain's products: 32 rows of
    // the block row, every G-th column.
    const int blk = warp / a.RG, rg = warp % a.RG, G = kWarps / a.RG;
    const bool rows_on = blk < a.NB, cols_on = blk < G;
    const int mine = cols_on && blk < CW ? (CW - blk + G - 1) / G : 0;  // columns of the chain's products
    const int row = rg * 32 + lane;
    for (int t = 0; t < own; ++t) {
      const int l = rank + S * t, ml = rows_of(l);
      for (int e = tid; e < ml * CW; e += 32 * kWarps) {
        const int r = e % ml, c = e / ml;
        W[static_cast<size_t>(t) * block_doubles + r * CW + c] =
            c < nc ? a.B[(j0 + c) * a.ldb + static_cast<int64_t>(l) * a.n0 + r] : 0.0;
      }
    }
    sync_consumers();
    double acc[CW];
    // acc[i] = sum over the columns of block (l, b) of L~(row, q) v[q][blk + i G]
    auto chain_product = [&](int l, int cols, int kend, const double* v) {
      const int rr = min(row, rows_of(l) - 1);
#pragma unroll
      for (int i = 0; i < CW; ++i) acc[i] = 0.0;
      for (int q = 0; q < cols && ok; q += a.KC1) {
        const int s = it % a.stages;
        ok = tc::mbar_wait(&full_bar[s], (it / a.stages) & 1, abort_flag);
        if (!ok) break;
        const double* st = sm + static_cast<size_t>(s) * kStageDoubles + rr;
        const int end = min(min(a.KC1, cols - q), kend - q);
        // one to four columns a warp, or all of them (G = 1)
        const double* vq = v + static_cast<size_t>(q) * CW + blk;
        if (mine == CW) dot_columns<CW, CW>(st, a.pitch, vq, G, end, acc);
        else if (mine == 1) dot_columns<CW, 1>(st, a.pitch, vq, G, end, acc);
        else if (mine == 2) dot_columns<CW, (CW < 2 ? CW : 2)>(st, a.pitch, vq, G, end, acc);
        else if (mine == 3) dot_columns<CW, (CW < 3 ? CW : 3)>(st, a.pitch, vq, G, end, acc);
        else if (mine == 4) dot_columns<CW, (CW < 4 ? CW : 4)>(st, a.pitch, vq, G, end, acc);
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(&empty_bar[s]);
        ++it;
      }
    };
    // X_l = L~_ll W_l, to global memory and to every CTA of the cluster
    auto solve_block = [&](int l) {
      const int ml = rows_of(l), slot = l % (S + 1);
      chain_product(l, ml, min(rg * 32 + 32, ml), W + static_cast<size_t>(l / S) * block_doubles);
      double* x = xs + static_cast<size_t>(slot) * block_doubles;
      if (cols_on && row < ml) {
#pragma unroll
        for (int i = 0; i < CW; ++i) {
          if (i >= mine) break;
          const int c = blk + i * G;
          if (S > 1)
            for (int r = 0; r < S; ++r) st_cluster(tc::cluster_addr(x + row * CW + c, r), acc[i]);
          else
            x[row * CW + c] = acc[i];
          if (c < nc) a.X[(j0 + c) * a.ldx + static_cast<int64_t>(l) * a.n0 + row] = acc[i];
        }
      }
      sync_consumers();
      if (S > 1) {
        if (tid < S) tc::mbar_arrive_cluster(tc::cluster_addr(&x_bar[slot], tid));
      } else if (tid == 0) {
        tc::mbar_arrive(&x_bar[slot]);
      }
    };
    if (rank == 0) solve_block(0);
    for (int b = 0; b + 1 < a.N; ++b) {
      const int slot = b % (S + 1);
      const double* x = xs + static_cast<size_t>(slot) * block_doubles;
      tc::mbar_wait_cluster(&x_bar[slot], (b / (S + 1)) & 1, abort_flag, tc::kMbarWaitNs);
      if ((b + 1) % S == rank) {
        const int l = b + 1, ml = rows_of(l);
        double* w = W + static_cast<size_t>(l / S) * block_doubles;
        chain_product(l, a.n0, a.n0, x);
        sync_consumers();  // the other division's updates of these rows are done
        if (cols_on && row < ml) {
#pragma unroll
          for (int i = 0; i < CW; ++i)
            if (i < mine) w[row * CW + blk + i * G] -= acc[i];
        }
        sync_consumers();
        solve_block(l);
      }
      const int t0 = first_rest(b);
      for (int g = t0 / a.NB; t0 < own && g * a.NB < own; ++g) {
        const int t = g * a.NB + blk, l = rank + S * t;
        const bool on = rows_on && t >= t0 && t < own;
        const int ml = on ? rows_of(l) : 1;
        const int rr = min(row, ml - 1);
#pragma unroll
        for (int c = 0; c < CW; ++c) acc[c] = 0.0;
        for (int q = 0; q < a.n0 && ok; q += a.KCn) {
          const int s = it % a.stages;
          ok = tc::mbar_wait(&full_bar[s], (it / a.stages) & 1, abort_flag);
          if (!ok) break;
          if (on)
            dot_columns<CW, CW>(sm + static_cast<size_t>(s) * kStageDoubles + static_cast<size_t>(blk * a.KCn) * a.pitch + rr,
                                a.pitch, x + static_cast<size_t>(q) * CW, 1, min(a.KCn, a.n0 - q), acc);
          __syncwarp();
          if (lane == 0) tc::mbar_arrive(&empty_bar[s]);
          ++it;
        }
        if (on && row < ml) {
          double* w = W + static_cast<size_t>(t) * block_doubles + static_cast<size_t>(row) * CW;
#pragma unroll
          for (int c = 0; c < CW; ++c) w[c] -= acc[c];
        }
      }
      // every wait ends at once after an abort: the loop runs out quickly
    }
  }
  __syncthreads();
  if (tid == 0 && abort_sh) atomicOr(a.status, 1);
  if (S > 1) tc::cluster_sync();  // no CTA ends while another may still write to it
}

size_t fixed_bytes(int64_t n0, int64_t N, int S, int CW) {
  return sizeof(double) * static_cast<size_t>(CW) * static_cast<size_t>(((N + S - 1) / S + S + 1) * n0);
}

template <int CW>
cudaError_t launch(const ColArgs& a, unsigned grid, size_t smem, cudaStream_t s) {
  auto kern = col_solve_kernel<CW>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxShared);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = static_cast<unsigned>(a.S);
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = a.S > 1 ? 1 : 0;
  e = cudaLaunchKernelEx(&cfg, kern, a);
  count_launch();
  return e != cudaSuccess ? e : cudaGetLastError();
}

// Clusters of S CTAs that are resident at once, one CTA per SM: less than the
// SMs over S, since a cluster lies within a GPC (GB300: 152, 76, 46, 36, 28,
// 23, 15, 15 for S = 1 .. 8).
int resident_clusters(int S) {
  static std::atomic<int> cache[128][kMaxCluster + 1];
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 128) dev = 0;
  int n = cache[dev][S].load(std::memory_order_relaxed);
  if (n > 0) return n;
  auto kern = col_solve_kernel<1>;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(static_cast<unsigned>(S));
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = kMaxShared;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = static_cast<unsigned>(S);
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxShared) != cudaSuccess ||
      cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess || n < 1) {
    cudaGetLastError();
    n = std::max(1, device_sm_count() / S);
  }
  cache[dev][S].store(n, std::memory_order_relaxed);
  return n;
}

}  // namespace

namespace {

// The block orders that run by columns: a row group per warp, whole 16-byte
// pairs of rows in every column.
bool cols_ok(int64_t n0, int64_t N) { return n0 <= kMaxRows && (N == 1 || n0 % 2 == 0) && N <= 1 << 20; }

// One way to run: S CTAs on CW columns.  S is 0 where their rows do not fit.
struct ColShape {
  ColPlan plan;
  double share = 0;       // column groups an SM (of S, a cluster) takes
  bool together = false;  // CTAs of more than one on an SM at a time
};
ColShape col_shape(int64_t n0, int64_t N, int64_t k, int S, int CW) {
  ColShape c;
  const size_t fixed = fixed_bytes(n0, N, S, CW);
  constexpr size_t kStage = kStageDoubles * sizeof(double);
  if (fixed + 2 * kStage > kMaxShared) return c;
  c.share = std::ceil(static_cast<double>((k + CW - 1) / CW) / resident_clusters(S));
  const size_t room = c.share > 1 ? kMaxShared / 2 : kMaxShared;  // two CTAs on an SM where there are more
  // (their registers too: 102 a thread for 18 warps)
  c.together = fixed + 2 * kStage <= room && (c.share <= 1 || CW <= 6);
  c.plan.S = S;
  c.plan.CW = CW;
  c.plan.stages = static_cast<int>(std::min<size_t>(((c.together ? room : kMaxShared) - fixed) / kStage, kMaxStages));
  c.plan.smem = fixed + c.plan.stages * kStage;
  return c;
}

}  // namespace

ColPlan col_plan_as(int64_t n, int64_t n0, int64_t k, int S, int CW) {
  const int64_t N = (n + n0 - 1) / n0;
  if (!cols_ok(n0, N) || S < 1 || S > kMaxCluster || S > N || CW < 1 || CW > kMaxCols) return ColPlan();
  return col_shape(n0, N, k, S, CW).plan;
}

ColPlan col_plan(int64_t n, int64_t n0, int64_t k) {
  ColPlan best;
  const int64_t N = (n + n0 - 1) / n0;
  if (!cols_ok(n0, N)) return best;
  const int RG = static_cast<int>((n0 + 31) / 32);
  double t_best = 1e300;
  for (int S = 1; S <= kMaxCluster && S <= N; ++S) {
    for (int CW = 1; CW <= kMaxCols && CW <= k; ++CW) {
      const ColShape shape = col_shape(n0, N, k, S, CW);
      if (shape.plan.S == 0) continue;
      const double share = shape.share;
      const bool together = shape.together;
      // Clocks.  Throughput: the multiply-adds at 2 per clock (1.12 times
      // that for one or two columns: the loads of L~) and the reductions of
      // the own block rows.  upd: a block of an update; diag: a diagonal
      // product, whose row groups stop at their own last column.  The chain of
      // block rows: the two one after the other (the first row has its
      // diagonal product alone), one dependent multiply-add every 125 clocks or
      // their throughput, and a signal.  What a CTA alone on its SM waits for
      // its own part of the chain is lost, beyond the throughput that is
      // counted already, and its start too; of the shorter of work and chain a
      // quarter shows.
      const double b = 32.0 * RG, own = static_cast<double>(N) / S;
      const double upd = 0.5 * b * b * CW, diag = 0.25 * b * (b + 32) * CW;
      const double busy = (CW <= 2 ? 1.12 : 1.0) * (0.5 * N * (N - 1) * upd + N * diag) / S + own * 3000.0;
      const double first = std::max(125.0 * b, diag), step = std::max(250.0 * b, upd + diag);
      const double lost = share > 1 && together
                              ? 0.0
                              : ((N - 1) * (step - upd - diag) + first - diag) / S + (share > 1 ? 2000.0 : 0.0);
      const double chain = S > 1 ? (N - 1) * (step + 3000.0) + first + 3000.0 : 0.0;
      const double rounds = together ? std::ceil(share / 2) : share;
      const double work = share * (busy + (S > 1 ? 0.0 : lost));
      const double t = std::max(work, rounds * chain) + 0.25 * std::min(work, rounds * chain);
      if (t < t_best) {
        t_best = t;
        best = shape.plan;
      }
    }
  }
  if (best.S == 0) return best;
  // The tile tasks of solve.cu: the multiply-adds of 32-wide column tiles on
  // all SMs, and the chain of the S and near-U tasks of n0 / 32 chunks each,
  // which overlap the more the longer the former is.  Fitted to (us, tile
  // tasks / columns): n0 = 64, n = 300 k = 2000 414 / 329, 900 x 1500 1487 /
  // 1258, 512 x 512 538 / 206, 1000 x 200 1026 / 294, 1000 x 37 1001 / 159;
  // n0 = 256, 2048 x 500 2914 / 2280, 4096 x 150 4849 / 2540, 4096 x 400 7284 /
  // 6655, 4096 x 800 11890 / 13220, 8192 x 64 9071 / 5262, 8192 x 152 12570 /
  // 9896, 8192 x 300 19400 / 17420, 3017 x 507 5163 / 4709, 1454 x 1147 2720 /
  // 2509, 1112 x 988 1741 / 1530.  Below n = 300 the division matters more than
  // the form (us by columns a group, one CTA each): 64 x 1 8.4 / 8.4 / 8.4 / - /
  // 12.4 for 1, 2, 3, 5 of them, 64 x 4 the same, 64 x 8 the same, 128 x 1 at
  // n0 = 128 11.2 for 1, 17.4 for 3, 7 x 1 4.5 for 1, 5.1 for 8.
  const double tiles =
      0.25 * static_cast<double>(n) * n * static_cast<double>((k + 31) / 32 * 32) / device_sm_count();
  const double tile_chain = N * (2.0 * RG * 16400 + 30000);
  const double exposed = std::min(1.0, std::max(0.1, 1.4 - 0.36 * tiles / tile_chain));
  best.use = 1.03 * t_best < tiles + exposed * tile_chain;
  return best;
}

cudaError_t col_solve(const ColPlan& p, const double* Lt, int64_t ldt, int64_t n, int64_t n0, const double* B, int64_t k,
                      int64_t ldb, double* X, int64_t ldx, int* status_dev, cudaStream_t s) {
  ColArgs a;
  a.Lt = Lt;
  a.ldt = ldt;
  a.B = B;
  a.ldb = ldb;
  a.X = X;
  a.ldx = ldx;
  a.n = n;
  a.k = k;
  a.n0 = static_cast<int>(n0);
  a.N = static_cast<int>((n + n0 - 1) / n0);
  a.S = p.S;
  a.RG = static_cast<int>((n0 + 31) / 32);
  a.NB = kWarps / a.RG;
  a.pitch = (a.n0 + 1) / 2 * 2;
  a.KC1 = std::min(a.n0, kStageDoubles / a.pitch);
  a.KCn = std::min(a.n0, kStageDoubles / (a.pitch * a.NB));
  a.stages = p.stages;
  a.status = status_dev;
  const unsigned grid = static_cast<unsigned>((k + p.CW - 1) / p.CW * p.S);
  switch (p.CW) {
    case 1: return launch<1>(a, grid, p.smem, s);
    case 2: return launch<2>(a, grid, p.smem, s);
    case 3: return launch<3>(a, grid, p.smem, s);
    case 4: return launch<4>(a, grid, p.smem, s);
    case 5: return launch<5>(a, grid, p.smem, s);
    case 6: return launch<6>(a, grid, p.smem, s);
    case 7: return launch<7>(a, grid, p.smem, s);
    default: return launch<8>(a, grid, p.smem, s);
  }
}

cudaError_t solve_any(const ColPlan& cols, const double* Lt, int64_t ldt, int64_t n, int64_t n0, const double* B,
                      int64_t k, int64_t ldb, double* X, int64_t ldx, void* ws, int* status_dev, cudaStream_t s) {
  if (cols.use) return col_solve(cols, Lt, ldt, n, n0, B, k, ldb, X, ldx, status_dev, s);
  return solve_enqueue(Lt, ldt, n, n0, B, k, ldb, X, ldx, ws, status_dev, s);
}

}  // namespace trsm
