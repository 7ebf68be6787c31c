// Batched recursive triangular inversion of diagonal blocks
// (Algorithm RecTriInv, Section 5.1, applied to every diagonal block as in
// Algorithm Diagonal-Inverter, Section 6.1).
//
// The recursion L^-1 = [L11^-1 0; -(L22^-1 L21) L11^-1  L22^-1] is run
// bottom-up over all blocks at once: the two half inversions of a node are
// independent (the paper runs them on disjoint processor sub-grids), so on
// one GPU every node of the same height across every diagonal block is
// processed by one launch.  Leaves (order <= 32) are inverted by one CTA
// each; each internal node costs two batched tile-GEMM launches per height:
//   T      = -(L22^-1 * L21)   (the first multiply of RecTriInv)
//   L21^-1 =  T * L11^-1       (the second multiply)
// exploiting the triangular factor to skip K ranges that multiply zeros.
//
// Bound by the FP64 pipe (2 multiply-adds per SM and clock), so what counts
// is that every SM has work to the end.  The tiles of a launch differ in
// their K range (32 to h), and are launched longest first, at most four CTAs
// to an SM (enough to keep its pipe full, as in the blocked solve): the SMs
// that finish early find short tiles left.  With every tile resident from
// the start, in row order, the pipe was busy half of the time: n = 8192, n0 =
// 512, us: the last height's products 458 + 328, all of them 1155, the leaves
// (a warp each, 850 dependent FP64 instructions of 64 clocks) 55.
#include <algorithm>
#include <cstdio>
#include <vector>

#include "fp64_leaf.cuh"
#include "fp64_tile.cuh"
#include "internal.h"

namespace trsm {

namespace {

constexpr int LEAF = 32;  // leaf order; also the tile size of the combines

struct LeafDesc {
  int64_t off;   // element offset of the leaf's top-left corner
  int64_t row0;  // first row in the caller's numbering
  int32_t m;     // order (<= LEAF)
  int32_t pad;
};

struct NodeDesc {
  int64_t off;    // element offset of the node's top-left corner
  int64_t toff;   // element offset of this node's T (r x h, ld r) in scratch
  int32_t h;      // order of L11 (a multiple of LEAF)
  int32_t r;      // order of L22
  int32_t tr;     // ceil(r / TILE)
  int32_t tc;     // h / TILE
};

struct FirstSingular {
  unsigned long long* sing;
  __device__ void operator()(int64_t row) const { atomicMin(sing, static_cast<unsigned long long>(row)); }
};

// One CTA per leaf, in place.
__global__ void __launch_bounds__(NTHREADS) leaf_inverse_kernel(double* __restrict__ A, int64_t ld,
                                                                const LeafDesc* __restrict__ leaves,
                                                                unsigned long long* __restrict__ sing) {
  __shared__ double ls[LEAF][LEAF + 1], tb[16][17];
  const LeafDesc d = leaves[blockIdx.x];
  leaf_invert_block<double>(A + d.off, ld, d.m, A + d.off, ld, ls, tb, FirstSingular{sing}, d.row0);
}

// acc = A(rows [0, m), K [kbeg, kend)) B(K [kbeg, kend), 32 columns), as
// tile_mma of fp64_tile.cuh with the next chunk's loads issued before the
// current chunk's multiply-adds (two shared-memory buffers, one barrier per
// chunk).  kTri: A's last chunk is its diagonal one, A(r, kend - m + ...) = 0
// to the right of row r: warp w, which holds rows 8 w to 8 w + 7, stops it
// after 8 (w + 1) steps.
struct PipeSmem {
  TileSmem buf[2];
};
template <bool kTri>
__device__ __forceinline__ void tile_product(const double* __restrict__ A, int64_t lda, const double* __restrict__ B,
                                             int64_t ldb, int m, int64_t kbeg, int64_t kend, PipeSmem& sm,
                                             double (&acc)[TM][TN]) {
  constexpr int kPer = KCH * TILE / NTHREADS;  // elements of either operand per thread and chunk
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int ty = tid >> 4, tx = tid & 15;
  double ra[kPer], rb[kPer];
  auto load = [&](int64_t k0) {
#pragma unroll
    for (int it = 0; it < kPer; ++it) {
      const int64_t ta = k0 + w + 4 * it, tb = k0 + lane;
      ra[it] = (lane < m && ta < kend) ? A[ta * lda + lane] : 0.0;
      rb[it] = tb < kend ? B[static_cast<int64_t>(w + 4 * it) * ldb + tb] : 0.0;
    }
  };
  auto store = [&](TileSmem& b) {
#pragma unroll
    for (int it = 0; it < kPer; ++it) {
      b.a[w + 4 * it][lane] = ra[it];
      b.b[lane][w + 4 * it] = rb[it];
    }
  };
  zero_acc(acc);
  load(kbeg);
  store(sm.buf[0]);
  __syncthreads();
  int cur = 0;
  for (int64_t k0 = kbeg; k0 < kend; k0 += KCH) {
    const bool more = k0 + KCH < kend;
    if (more) load(k0 + KCH);
    const TileSmem& b = sm.buf[cur];
    const int steps = static_cast<int>(imin64(KCH, kend - k0));
    const int end = kTri && !more ? min(steps, 8 * w + 8) : steps;
#pragma unroll 8
    for (int kk = 0; kk < end; ++kk) {
      double av[TM], bv[TN];
#pragma unroll
      for (int i = 0; i < TM; ++i) av[i] = b.a[kk][ty * TM + i];
#pragma unroll
      for (int j = 0; j < TN; ++j) bv[j] = b.b[kk][tx * TN + j];
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j] = fma(av[i], bv[j], acc[i][j]);
    }
    if (more) store(sm.buf[cur ^ 1]);  // last read before the previous barrier
    __syncthreads();
    cur ^= 1;
  }
}

// T = -(L22^-1 * L21): one TILE x TILE tile of T per CTA.  Row tile a of the
// lower triangular L22^-1 only meets K < (a + 1) TILE: blockIdx.y counts the
// row tiles from the last.  blockIdx.x: node and column tile, `cols` of them
// per node.
__global__ void __launch_bounds__(NTHREADS) combine_first_kernel(const double* __restrict__ A, int64_t ld,
                                                                 const NodeDesc* __restrict__ nodes, int cols,
                                                                 double* __restrict__ T) {
  __shared__ PipeSmem sm;
  const NodeDesc nd = nodes[blockIdx.x / cols];
  const int a = nd.tr - 1 - static_cast<int>(blockIdx.y), b = blockIdx.x % cols;
  if (a < 0 || b >= nd.tc) return;
  const double* L22inv = A + nd.off + (int64_t)nd.h * ld + nd.h;
  const double* L21 = A + nd.off + nd.h;
  double acc[TM][TN];
  tile_product<true>(L22inv + a * TILE, ld, L21 + (int64_t)b * TILE * ld, ld, min(TILE, nd.r - a * TILE), 0,
                     min((a + 1) * TILE, nd.r), sm, acc);
  const int ty = threadIdx.x >> 4, tx = threadIdx.x & 15;
  double* To = T + nd.toff;
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    const int row = a * TILE + ty * TM + i;
    if (row >= nd.r) continue;
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      const int col = b * TILE + tx * TN + j;
      To[(int64_t)col * nd.r + row] = -acc[i][j];
    }
  }
}

// L21^-1 = T * L11^-1, written over L21.  Column tile b of the lower
// triangular L11^-1 only meets K >= b TILE: blockIdx.y is the column tile.
// blockIdx.x: node and row tile, `rows` of them per node.
__global__ void __launch_bounds__(NTHREADS) combine_second_kernel(double* __restrict__ A, int64_t ld,
                                                                  const NodeDesc* __restrict__ nodes, int rows,
                                                                  const double* __restrict__ T) {
  __shared__ PipeSmem sm;
  const NodeDesc nd = nodes[blockIdx.x / rows];
  const int a = blockIdx.x % rows, b = blockIdx.y;
  if (a >= nd.tr || b >= nd.tc) return;
  double acc[TM][TN];
  tile_product<false>(T + nd.toff + a * TILE, nd.r, A + nd.off + (int64_t)b * TILE * ld, ld,
                      min(TILE, nd.r - a * TILE), (int64_t)b * TILE, nd.h, sm, acc);
  const int ty = threadIdx.x >> 4, tx = threadIdx.x & 15;
  double* Out = A + nd.off + nd.h;
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    const int row = a * TILE + ty * TM + i;
    if (row >= nd.r) continue;
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      const int col = b * TILE + tx * TN + j;
      Out[(int64_t)col * ld + row] = acc[i][j];
    }
  }
}

// Lt = the lower triangle of L.  VEC: both matrices' columns start on 16-byte
// boundaries (aligned bases, even leading dimensions), and each thread moves
// a pair of rows with one 16-byte load and store; the pair that straddles
// the diagonal loads its lower element alone, and pairs above the diagonal
// are written as zeros without reading L.
template <bool VEC>
__global__ void copy_lower_kernel(const double* __restrict__ L, int64_t ldl, double* __restrict__ Lt,
                                  int64_t ldt, int64_t n) {
  for (int64_t j = blockIdx.y; j < n; j += gridDim.y) {
    const double* src = L + j * ldl;
    double* dst = Lt + j * ldt;
    if constexpr (VEC) {
      for (int64_t i = 2 * (blockIdx.x * (int64_t)blockDim.x + threadIdx.x); i < n;
           i += 2 * (int64_t)gridDim.x * blockDim.x) {
        if (i + 1 < n) {
          double2 v = make_double2(0.0, 0.0);
          if (i >= j) v = *reinterpret_cast<const double2*>(src + i);
          else if (i + 1 == j) v.y = src[i + 1];
          *reinterpret_cast<double2*>(dst + i) = v;
        } else {
          dst[i] = (i >= j) ? src[i] : 0.0;
        }
      }
    } else {
      for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
           i += (int64_t)gridDim.x * blockDim.x)
        dst[i] = (i >= j) ? src[i] : 0.0;
    }
  }
}

__global__ void pack_blocks_kernel(const double* __restrict__ L, int64_t ldl, double* __restrict__ P,
                                   int64_t n, int64_t n0, int64_t nblocks) {
  // blockIdx.y enumerates (block, column) pairs; threads run over rows.
  for (int64_t bc = blockIdx.y; bc < nblocks * n0; bc += gridDim.y) {
    const int64_t b = bc / n0, c = bc % n0;
    const int64_t s0 = b * n0;
    const int64_t m = min(n0, n - s0);
    for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < n0;
         r += (int64_t)gridDim.x * blockDim.x) {
      double v = 0.0;
      if (r < m && c < m && r >= c) v = L[(s0 + c) * ldl + s0 + r];
      P[b * n0 * n0 + c * n0 + r] = v;
    }
  }
}

// W = B (n x k).  VEC: 16-byte loads and stores of row pairs, as above.
template <bool VEC>
__global__ void copy_panel_kernel(const double* __restrict__ B, int64_t ldb, double* __restrict__ W,
                                  int64_t ldw, int64_t n, int64_t k) {
  for (int64_t j = blockIdx.y; j < k; j += gridDim.y) {
    const double* src = B + j * ldb;
    double* dst = W + j * ldw;
    if constexpr (VEC) {
      for (int64_t i = 2 * (blockIdx.x * (int64_t)blockDim.x + threadIdx.x); i < n;
           i += 2 * (int64_t)gridDim.x * blockDim.x) {
        if (i + 1 < n) *reinterpret_cast<double2*>(dst + i) = *reinterpret_cast<const double2*>(src + i);
        else dst[i] = src[i];
      }
    } else {
      for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
           i += (int64_t)gridDim.x * blockDim.x)
        dst[i] = src[i];
    }
  }
}

// Columns of both matrices start on 16-byte boundaries.
inline bool pairs_aligned(const void* a, int64_t lda, const void* b, int64_t ldb) {
  return ((reinterpret_cast<uintptr_t>(a) | reinterpret_cast<uintptr_t>(b)) & 15) == 0 && (lda % 2) == 0 &&
         (ldb % 2) == 0;
}

// Host-side recursion tree.  A node of order m > LEAF splits at
// h = LEAF * ceil(m / (2*LEAF)) so that h is a multiple of the tile size.
struct TreeBuilder {
  int64_t ld;
  std::vector<LeafDesc> leaves;
  std::vector<std::vector<NodeDesc>> by_height;  // index = height - 1

  int build(int64_t off, int64_t m, int64_t row0) {
    if (m <= LEAF) {
      leaves.push_back(LeafDesc{off, row0, (int32_t)m, 0});
      return 0;
    }
    const int64_t h = LEAF * ((m + 2 * LEAF - 1) / (2 * LEAF));
    const int64_t r = m - h;
    const int h1 = build(off, h, row0);
    const int h2 = build(off + h * ld + h, r, row0 + h);
    const int ht = 1 + std::max(h1, h2);
    if ((int)by_height.size() < ht) by_height.resize(ht);
    NodeDesc nd{};
    nd.off = off;
    nd.h = (int32_t)h;
    nd.r = (int32_t)r;
    nd.tr = (int32_t)((r + TILE - 1) / TILE);
    nd.tc = (int32_t)(h / TILE);
    by_height[ht - 1].push_back(nd);
    return ht;
  }
};

}  // namespace

cudaError_t invert_diag_blocks(double* A, int64_t ld, const std::vector<DiagBlock>& blocks,
                               unsigned long long* sing_dev, std::vector<unsigned char>& host, cudaStream_t s) {
  TreeBuilder tb;
  tb.ld = ld;
  for (const DiagBlock& b : blocks)
    if (b.m > 0) tb.build(b.off, b.m, b.row0);
  if (tb.leaves.empty()) return cudaSuccess;

  // T scratch offsets (scratch reused across heights: heights run one after
  // another on the stream).
  int64_t scratch_elems = 0;
  size_t node_total = 0;
  for (auto& lvl : tb.by_height) {
    int64_t toff = 0;
    for (NodeDesc& nd : lvl) {
      nd.toff = toff;
      toff += (int64_t)nd.r * nd.h;
    }
    scratch_elems = std::max(scratch_elems, toff);
    node_total += lvl.size();
  }
  const size_t leaf_bytes = tb.leaves.size() * sizeof(LeafDesc);
  const size_t node_bytes = node_total * sizeof(NodeDesc);
  host.resize(leaf_bytes + node_bytes);
  memcpy(host.data(), tb.leaves.data(), leaf_bytes);
  size_t pos = leaf_bytes;
  for (auto& lvl : tb.by_height) {
    memcpy(host.data() + pos, lvl.data(), lvl.size() * sizeof(NodeDesc));
    pos += lvl.size() * sizeof(NodeDesc);
  }
  void* desc = nullptr;
  double* T = nullptr;
  cudaError_t e = trsm::ws_alloc(&desc, host.size(), s);
  if (e != cudaSuccess) return e;
  if (scratch_elems > 0) {
    e = trsm::ws_alloc((void**)&T, sizeof(double) * (size_t)scratch_elems, s);
    if (e != cudaSuccess) {
      trsm::ws_free(desc, s);
      return e;
    }
  }
  e = cudaMemcpyAsync(desc, host.data(), host.size(), cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) {
    const LeafDesc* d_leaves = (const LeafDesc*)desc;
    leaf_inverse_kernel<<<(unsigned)tb.leaves.size(), NTHREADS, 0, s>>>(A, ld, d_leaves, sing_dev);
    count_launch();
    e = cudaGetLastError();
    const NodeDesc* d_nodes = (const NodeDesc*)((unsigned char*)desc + leaf_bytes);
    // shared memory that four CTAs of the products take up
    constexpr int kPad = 56 * 1024 - (int)sizeof(PipeSmem);
    if (e == cudaSuccess && node_total > 0) {
      e = cudaFuncSetAttribute(combine_first_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kPad);
      if (e == cudaSuccess)
        e = cudaFuncSetAttribute(combine_second_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kPad);
    }
    for (auto& lvl : tb.by_height) {
      if (e != cudaSuccess) break;
      const unsigned nn = (unsigned)lvl.size();
      int tr = 1, tc = 1;
      for (const NodeDesc& nd : lvl) {
        tr = std::max(tr, nd.tr);
        tc = std::max(tc, nd.tc);
      }
      combine_first_kernel<<<dim3(nn * tc, tr), NTHREADS, kPad, s>>>(A, ld, d_nodes, tc, T);
      combine_second_kernel<<<dim3(nn * tr, tc), NTHREADS, kPad, s>>>(A, ld, d_nodes, tr, T);
      count_launch(2);
      e = cudaGetLastError();
      d_nodes += nn;
    }
  }
  if (T) trsm::ws_free(T, s);
  trsm::ws_free(desc, s);
  return e;
}

static dim3 grid2d(int64_t rows, int64_t cols) {
  const int64_t gx = std::min<int64_t>((rows + 255) / 256, 64);
  const int64_t gy = std::min<int64_t>(cols, 65535);
  return dim3((unsigned)std::max<int64_t>(gx, 1), (unsigned)std::max<int64_t>(gy, 1));
}

cudaError_t copy_lower(const double* L, int64_t ldl, double* Lt, int64_t ldt, int64_t n,
                       cudaStream_t s) {
  if (pairs_aligned(L, ldl, Lt, ldt))
    copy_lower_kernel<true><<<grid2d((n + 1) / 2, n), 256, 0, s>>>(L, ldl, Lt, ldt, n);
  else
    copy_lower_kernel<false><<<grid2d(n, n), 256, 0, s>>>(L, ldl, Lt, ldt, n);
  count_launch();
  return cudaGetLastError();
}

cudaError_t pack_diag_blocks(const double* L, int64_t ldl, double* P, int64_t n, int64_t n0,
                             cudaStream_t s) {
  const int64_t nb = (n + n0 - 1) / n0;
  pack_blocks_kernel<<<grid2d(n0, nb * n0), 256, 0, s>>>(L, ldl, P, n, n0, nb);
  count_launch();
  return cudaGetLastError();
}

// Zeroes the strictly upper part of every n0 x n0 diagonal block of Lt
// (what a copy of the lower trapezoid of each block column brings along).
__global__ void zero_upper_blocks_kernel(double* __restrict__ Lt, int64_t ldt, int64_t n, int64_t n0) {
  const int64_t nb = (n + n0 - 1) / n0;
  for (int64_t bc = blockIdx.y; bc < nb * n0; bc += gridDim.y) {
    const int64_t b = bc / n0, c = bc % n0, s0 = b * n0;
    if (s0 + c >= n) continue;
    for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < c; r += (int64_t)gridDim.x * blockDim.x)
      Lt[(s0 + c) * ldt + s0 + r] = 0.0;
  }
}

cudaError_t zero_upper_blocks(double* Lt, int64_t ldt, int64_t n, int64_t n0, cudaStream_t s) {
  const int64_t nb = (n + n0 - 1) / n0;
  zero_upper_blocks_kernel<<<grid2d(n0, nb * n0), 256, 0, s>>>(Lt, ldt, n, n0);
  count_launch();
  return cudaGetLastError();
}

cudaError_t copy_panel(const double* B, int64_t ldb, double* W, int64_t ldw, int64_t n, int64_t k,
                       cudaStream_t s) {
  if (pairs_aligned(B, ldb, W, ldw))
    copy_panel_kernel<true><<<grid2d((n + 1) / 2, k), 256, 0, s>>>(B, ldb, W, ldw, n, k);
  else
    copy_panel_kernel<false><<<grid2d(n, k), 256, 0, s>>>(B, ldb, W, ldw, n, k);
  count_launch();
  return cudaGetLastError();
}

}  // namespace trsm
