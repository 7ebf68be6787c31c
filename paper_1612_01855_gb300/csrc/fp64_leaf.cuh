// Inversion of a triangular block of order up to 32 by one CTA, shared by
// the plan's inversion and the batched launch.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "fp64_tile.cuh"

namespace trsm {

// Inverse of the leading m x m (m <= 32) lower triangle of A (leading
// dimension lda) into out (leading dimension ldo, the m x m part only), by
// RecTriInv with the whole CTA: the block, padded with an identity to 32
// rows, is cut into four 8 x 8 leaves inverted by column substitution (one
// thread per leaf column), then combined at h = 8 (two nodes) and h = 16,
// T = -(L22^-1 L21) first and T L11^-1 second.  ls (32 x 33) holds the
// block, tb (16 x 17) the T factor; out may be A.  An entry that is not
// finite reaches no row above its own: the first product leaves out what meets
// the zeros above L22^-1's diagonal (by a select: a loop that ends at the
// diagonal costs 7 of 326 us of a plan and solve at n = 512).  A zero or
// non-finite pivot is reported as bad(row), rows counted from row0.  Every
// thread of the CTA (NTHREADS) must call it (it synchronises).  Out of line: it
// runs only in the inversion phase of the batched launch.
template <class T, class Bad>
__device__ __noinline__ void leaf_invert_block(const T* A, int64_t lda, int m, T* out, int64_t ldo, T (*ls)[33],
                                               T (*tb)[17], Bad bad, int64_t row0) {
  const int tid = threadIdx.x;
  // the lower triangle, the identity past m, zeros elsewhere; every load in
  // flight before the first store
  {
    T v[8];
#pragma unroll
    for (int it = 0; it < 8; ++it) {
      const int e = tid + NTHREADS * it, c = e >> 5, r = e & 31;
      v[it] = (r < m && c < m && r >= c) ? A[static_cast<int64_t>(c) * lda + r] : (r == c && r >= m ? T(1) : T(0));
    }
#pragma unroll
    for (int it = 0; it < 8; ++it) {
      const int e = tid + NTHREADS * it;
      ls[e >> 5][e & 31] = v[it];  // ls[col][row]
    }
  }
  __syncthreads();
  // leaves: thread (b, c) of the first warp forms column c of leaf b's inverse
  T y[8];
  const int lb = tid >> 3, lc = tid & 7, o = 8 * lb;
  if (tid < 32) {
    const T piv = ls[o + lc][o + lc];
    if (o + lc < m && (piv == T(0) || !isfinite(static_cast<double>(piv))))
      bad(row0 + o + lc);
#pragma unroll
    for (int r = 0; r < 8; ++r) y[r] = (r == lc) ? T(1) : T(0);
#pragma unroll
    for (int l = 0; l < 8; ++l) {
      y[l] = y[l] / ls[o + l][o + l];
#pragma unroll
      for (int r = l + 1; r < 8; ++r) y[r] = fma(-ls[o + l][o + r], y[l], y[r]);
    }
  }
  __syncthreads();
  if (tid < 32) {
#pragma unroll
    for (int r = 0; r < 8; ++r) ls[o + lc][o + r] = y[r];
  }
  __syncthreads();
  // combine level h: nodes of order 2h at base b = 2 h q; lanes over rows
#pragma unroll
  for (int h = 8; h <= 16; h *= 2) {
    const int nodes = 32 / (2 * h), rows = nodes * h, outs = rows * h;
    for (int e = tid; e < outs; e += NTHREADS) {
      const int rr = e % rows, c = e / rows, q = rr / h, r = rr % h, b = 2 * h * q;
      T acc = T(0);
      for (int p = 0; p < h; ++p) acc = fma(ls[b + h + p][b + h + r], p <= r ? ls[b + c][b + h + p] : T(0), acc);
      tb[q * h + c][r] = -acc;
    }
    __syncthreads();
    for (int e = tid; e < outs; e += NTHREADS) {
      const int rr = e % rows, c = e / rows, q = rr / h, r = rr % h, b = 2 * h * q;
      T acc = T(0);
      for (int p = c; p < h; ++p) acc = fma(tb[q * h + p][r], ls[b + c][b + p], acc);
      ls[b + c][b + h + r] = acc;
    }
    __syncthreads();
  }
  for (int e = tid; e < m * m; e += NTHREADS) {
    const int c = e / m, r = e % m;
    out[static_cast<int64_t>(c) * ldo + r] = ls[c][r];
  }
  __syncthreads();  // ls may be refilled right after
}

}  // namespace trsm
