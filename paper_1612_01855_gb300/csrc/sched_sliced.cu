// The sliced schedule of the blocked solve: Algorithm It-Inv-TRSM (Section
// 6.2) in its right-looking order, with both of its matrix multiplies on
// the BF16 tensor cores in a residue number system (rns.h; every factor to 48
// bits of its row's, or column's, maximum, exact products):
//
//   for i = 0 .. N-1:
//     X(S_i)      = L~_ii W(S_i)                 product, FP64 result
//     W(T_{i+1}) -= L(T_{i+1}, S_i) X(S_i)       product, FP64 update
//
// with W = B to begin with (the first step reads B and writes W).  FP64
// arithmetic remains for the last step of every product: one conversion and
// one or two multiply-adds per output.  GB300 runs FP64 only on its DFMA
// units (about 1.25 TFLOP/s), while the 15 bf16 products of an FP64-class
// product run at the tensor rate: n^2 k of FP64 work takes 15 n^2 k BF16
// operations (splitting into eight 6-bit digits, the form before, took 36).
//
// Everything runs on the caller's stream.  (A look-ahead, the rows of the
// next block on one stream and the rest of the update on another, is slower
// than one product over all rows: the two share the SMs, and the far update
// of one step delays the next one's.  n = 16384, k = 256, n0 = 2048: 1.71
// against 1.57 ms.)
//
// The plan keeps two residue operands (trsm_plan_sliced):
//   off: L off its diagonal blocks, one exponent per row and block column
//        (chunks of n0 along K), read by the trailing updates;
//   inv: the rows of the inverted diagonal blocks below their diagonal, read
//        by the diagonal multiplies, whose diagonal term is applied in FP64.
// The diagonal blocks are left out of `off`, and the diagonal out of `inv`:
// a row's exponent would otherwise follow its diagonal entry, and its other
// entries would keep fewer significant bits.
#include <cuda_runtime.h>

#include <algorithm>

#include "internal.h"
#include "rns.h"
#include "trsm_gb300.h"

namespace trsm {

struct SlicedPlan {
  void* buf = nullptr;  // off, then inv, then diag
  RnsOperand off, inv;
  double* diag = nullptr;  // diagonal of L~ (of the inverted blocks), applied in FP64
  int64_t nb = 0;      // block order: min(n0, n)
  size_t bytes = 0;
};

size_t sliced_bytes(const trsm_plan_s* h) { return (h && h->sliced) ? h->sliced->bytes : 0; }

void sliced_release(trsm_plan_s* h) {
  if (!h || !h->sliced) return;
  if (h->sliced->buf) cudaFree(h->sliced->buf);
  delete h->sliced;
  h->sliced = nullptr;
}

namespace {
inline size_t al256(size_t x) { return (x + 255) / 256 * 256; }

// A wait that ran out in one of the solve's tensor-core kernels (*err set)
// becomes the plan's sticky timeout status, read by trsm_sync_status.
__global__ void fold_error_kernel(const int* err, int* status) {
  if (*err) atomicOr(status, 1);
}

// The block orders the sliced products accept: a single block of at most
// kChunk rows (the diagonal multiply alone), or blocks of a multiple of 64
// rows up to kChunk (a K step of 64 never straddles two block columns, and
// a block's sums stay exact).
bool sliced_shape_ok(int64_t n, int64_t n0, int64_t N) {
  if (N == 1) return n <= kChunk;
  return n0 % 64 == 0 && n0 <= kChunk;
}
}  // namespace

namespace {

// The columns [0, k) of one panel.
struct Panel {
  const double* B;
  int64_t ldb;
  double* X;
  int64_t ldx, k;
};

cudaError_t solve_panel(const trsm_plan_s* h, const Panel& pn, double* W, int64_t ld, const RnsOperand& P,
                        const RnsScratch& sc, int* err, cudaStream_t s) {
  const SlicedPlan* sp = h->sliced;
  const int64_t n = h->n, N = h->N, nb = sp->nb;
  const RnsClass full = rns_class(8);
  cudaError_t e = cudaSuccess;
  for (int64_t i = 0; i < N && e == cudaSuccess; ++i) {
    const int64_t s0 = i * nb, m = std::min(nb, n - s0);
    // the first block row reads B itself, and its update starts W from it
    const double* src = i == 0 ? pn.B : W;
    const int64_t lds = i == 0 ? pn.ldb : ld;
    // X(S_i) = L~_ii W(S_i): the columns of W(S_i) are the B operand's rows
    e = rns_rows(src + s0, lds, m, P, full, s);
    RnsProduct p;
    p.A = sp->inv;
    p.a_row0 = s0;
    p.B = P;
    p.M = p.K = m;
    p.N = pn.k;
    p.lower = true;
    p.mode = kRnsDiag;
    p.Y = pn.X + s0;
    p.ldy = pn.ldx;
    p.S = src + s0;
    p.lds = lds;
    p.dg = sp->diag + s0;
    if (e == cudaSuccess) e = rns_product(p, sc, err, s);
    if (e != cudaSuccess || i == N - 1) break;
    // W(T_{i+1}) -= L(T_{i+1}, S_i) X(S_i)
    e = rns_rows(pn.X + s0, pn.ldx, m, P, full, s);
    const int64_t s1 = s0 + nb;
    RnsProduct u;
    u.A = rns_chunk(sp->off, i);  // rows from s0 on
    u.a_row0 = nb;
    u.B = P;
    u.M = n - s1;
    u.N = pn.k;
    u.K = m;
    u.Y = W + s1;
    u.ldy = ld;
    u.S = src + s1;
    u.lds = lds;
    if (e == cudaSuccess) e = rns_product(u, sc, err, s);
  }
  return e;
}

// Columns of X are independent: wide right-hand sides go in panels of at
// most this many bytes of residues (of a block row of W or X).
constexpr size_t kPanelBytes = 1ull << 30;

}  // namespace

int solve_sliced(trsm_plan_s* h, const double* B, int64_t k, int64_t ldb, double* X, int64_t ldx,
                 cudaStream_t s) {
  SlicedPlan* sp = h->sliced;
  const int64_t n = h->n, N = h->N, nb = sp->nb;
  const int64_t ld = (n + 3) / 4 * 4;
  const int64_t kmax = std::max<int64_t>(256, static_cast<int64_t>(kPanelBytes / (2 * kModuli * nb)) / 256 * 256);
  const int64_t npan = (k + kmax - 1) / kmax;
  const int64_t kp = npan == 1 ? k : ((k + npan - 1) / npan + 255) / 256 * 256;
  const size_t wbytes = N > 1 ? al256(sizeof(double) * static_cast<size_t>(ld) * static_cast<size_t>(kp)) : 0;
  const size_t pbytes = rns_operand_bytes(kp, nb, nb);
  // the last, narrower panel may take narrower tiles than the others
  const int64_t klast = k - (npan - 1) * kp;
  const size_t sbytes = al256(std::max(rns_scratch_bytes(n, kp), rns_scratch_bytes(n, klast)));
  unsigned char* ws = nullptr;
  cudaError_t e = trsm::ws_alloc(reinterpret_cast<void**>(&ws), wbytes + pbytes + sbytes + 256, s);
  if (e != cudaSuccess) return e == cudaErrorMemoryAllocation ? TRSM_ENOMEM : TRSM_ECUDA;
  double* W = reinterpret_cast<double*>(ws);
  unsigned char* scratch = ws + wbytes + pbytes;
  int* err = reinterpret_cast<int*>(scratch + sbytes);
  e = cudaMemsetAsync(err, 0, sizeof(int), s);
  for (int64_t j0 = 0; j0 < k && e == cudaSuccess; j0 += kp) {
    const Panel pn{B + j0 * ldb, ldb, X + j0 * ldx, ldx, std::min(kp, k - j0)};
    // the residues of W(S_i) are dead once X(S_i) is there: one buffer
    RnsOperand P = rns_operand_view(ws + wbytes, pn.k, nb, nb);
    const RnsScratch sc = rns_scratch_view(scratch, n, pn.k);
    P.zmax = sc.zmax;
    e = rns_scratch_clear(sc, s);
    if (e == cudaSuccess) e = solve_panel(h, pn, W, ld, P, sc, err, s);
  }
  if (e == cudaSuccess) {
    fold_error_kernel<<<1, 1, 0, s>>>(err, plan_status_word(h));
    count_launch();
    e = cudaGetLastError();
  }
  trsm::ws_free(ws, s);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return e == cudaErrorMemoryAllocation ? TRSM_ENOMEM : TRSM_ECUDA;
  }
  return TRSM_SUCCESS;
}

}  // namespace trsm

extern "C" int trsm_plan_sliced(trsm_handle_t h, void* stream) {
  if (!h) return TRSM_EINVAL;
  const int64_t n = h->n, N = h->N, nb = std::min(h->n0, h->n);
  if (!trsm::sliced_shape_ok(n, nb, N)) return TRSM_EINVAL;
  if (h->sliced) return TRSM_SUCCESS;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  auto* sp = new (std::nothrow) trsm::SlicedPlan;
  if (!sp) return TRSM_ENOMEM;
  sp->nb = nb;
  const size_t ob = N > 1 ? trsm::rns_operand_bytes(n, n, nb, true) : 0;
  const size_t ib = trsm::rns_operand_bytes(n, nb, nb);
  const size_t db = sizeof(double) * static_cast<size_t>(n);
  cudaError_t e = cudaMalloc(&sp->buf, ob + ib + db);
  double* tmp = nullptr;
  if (e == cudaSuccess) e = trsm::ws_alloc(reinterpret_cast<void**>(&tmp), sizeof(double) * n * std::max(n, nb), s);
  if (e == cudaSuccess && N > 1) {
    sp->off = trsm::rns_operand_view(sp->buf, n, n, nb, true);
    e = trsm::rns_offdiag_block_rows(h->Lt, h->ldt, n, nb, sp->off, tmp, s);
  }
  if (e == cudaSuccess) {
    sp->inv = trsm::rns_operand_view(static_cast<unsigned char*>(sp->buf) + ob, n, nb, nb);
    sp->diag = reinterpret_cast<double*>(static_cast<unsigned char*>(sp->buf) + ob + ib);
    e = trsm::rns_inverse_block_rows(h->Lt, h->ldt, n, nb, sp->inv, sp->diag, tmp, s);
  }
  if (tmp) trsm::ws_free(tmp, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) {
    cudaGetLastError();
    if (sp->buf) cudaFree(sp->buf);
    delete sp;
    return e == cudaErrorMemoryAllocation ? TRSM_ENOMEM : TRSM_ECUDA;
  }
  sp->bytes = ob + ib + db;
  h->sliced = sp;
  return TRSM_SUCCESS;
}
