// Residue-number-system products on the BF16 tensor cores (tcgen05): see
// rns.h for the method.  Two parts: the residues of an operand
// (residue_rows_kernel), and the product kernel (rns_product_kernel), whose
// epilogue reduces each modulus' FP32 sums to bytes and which puts an output
// tile's integer products together (Chinese remainder theorem) and applies
// them when its last modulus is there.
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <type_traits>

#include "internal.h"
#include "rns.h"
#include "tc_engine.cuh"
#include "tc_host.h"
#include "trsm_gb300_engine.h"

namespace trsm {
namespace rns {

// The pairwise coprime moduli <= 179 of the largest product, in descending
// order, so that a prefix of them serves the narrower classes: M = 2^109.6,
// 2^102.6 and 2^95.5 for 15, 14 and 13.  179 is the largest modulus whose
// residues, rounding slack included, stay within 90.
constexpr int kP[kModuli] = {179, 178, 177, 173, 169, 167, 163, 161, 157, 155, 151, 149, 139, 137, 131};
constexpr int kMaxResidue = 90;
static_assert(kChunk * kMaxResidue * kMaxResidue < (1 << 24), "a chunk's sums must be exact in FP32");

constexpr int kNonFinite = INT16_MAX;  // exponent of a (row, chunk) that holds an infinity or a NaN
// 6-bit digits of zeros that end the integers of two factors, together, from
// which their product is put together exactly: nine digits are left of 48 and
// 48 bits.
constexpr int kExactDigits = 7;
constexpr float kRound = 12582912.f;   // 1.5 * 2^23: x + kRound - kRound rounds |x| < 2^22 to an integer
constexpr int kStepK = 64;             // one 128-byte swizzled row of bf16

// ------------------------------------------------------------- residues
struct ResidueConsts {
  float p[kModuli], inv[kModuli];  // modulus and its reciprocal
  float c16[kModuli], c32[kModuli];  // 2^16 and 2^32 modulo p, symmetric
};

// round(a 2^(bits - e)) as three signed 16-bit limbs (the top one up to
// 2^16), from the bit fields of `a` with integer operations only (GB300's
// FP64 pipe is narrow): a = +-m 2^(E - 1075) with m the 53-bit significand,
// so the rounded value is m shifted right by (1075 - E) - (bits - e) >= 5
// bits, rounded to nearest.  The limbs become floats by the add of a
// constant that holds them in its low mantissa bits.
__device__ __forceinline__ void limbs_of(double a, int bits, int e, float& v0, float& v1, float& v2) {
  const unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(a));
  const int E = static_cast<int>((b >> 52) & 0x7FF);
  unsigned long long m = b & ((1ull << 52) - 1);
  if (E != 0) m |= 1ull << 52;
  const int rsh = (1075 - (E != 0 ? E : 1)) - (bits - e);
  long long v = 0;
  if (rsh < 64) v = static_cast<long long>((m + (1ull << (rsh - 1))) >> rsh);
  if (b >> 63) v = -v;
  const int l0 = static_cast<int16_t>(v);
  v = (v - l0) >> 16;
  const int l1 = static_cast<int16_t>(v);
  v = (v - l1) >> 16;
  v0 = __int_as_float(0x4B400000 + l0) - kRound;
  v1 = __int_as_float(0x4B400000 + l1) - kRound;
  v2 = __int_as_float(0x4B400000 + static_cast<int>(v)) - kRound;
}

// Residue of v2 2^32 + v1 2^16 + v0: the limbs times the residues of 2^16
// and 2^32 sum to at most 2^16 * 89 + 2^15 * 90 < 2^23.2, exact in FP32; the
// quotient's rounding error (below 0.01) leaves |r| <= p / 2 + 0.01 p, at
// most 90.
__device__ __forceinline__ float residue_of(float v0, float v1, float v2, float p, float inv, float c16, float c32) {
  const float s = fmaf(v2, c32, fmaf(v1, c16, v0));
  const float q = fmaf(s, inv, kRound) - kRound;
  return fmaf(-p, q, s);
}

// Two small integers as a pair of bf16: the upper halves of the floats
// (exact: at most eight significant bits).
__device__ __forceinline__ uint32_t bf16_pair(float lo, float hi) {
  return __byte_perm(__float_as_uint(lo), __float_as_uint(hi), 0x7632);
}

// kWarps warps per (row, chunk), 8 / kWarps of them per CTA; each lane
// converts four consecutive values at a time and stores four residues (8
// bytes) per modulus.  The chunk's values stay in registers between the
// maximum and the conversion (at most 2048 / (32 kWarps) = 8 a lane), so
// they are read once.  Bound by HBM: 8 bytes read and 2 bytes per modulus
// written per value.  zeros[r ex_stride + c]: the 6-bit digits (0 to 7) that
// end every integer of the (row, chunk) in zeros; their maximum is folded into
// *zmax.  A value with one of its lowest 11 bits set leaves none, which settles
// nearly every warp with one vote.
template <int kWarps>
__global__ void __launch_bounds__(256) residue_rows_kernel(const double* src, int64_t ld, int64_t rows,
                                                           int64_t K, int64_t nch, int64_t kc, int64_t ex_stride,
                                                           __nv_bfloat16* __restrict__ dst, int64_t kb,
                                                           int16_t* __restrict__ ex, int8_t* __restrict__ zeros,
                                                           int* zmax, int moduli, int bits, int tri, int vec,
                                                           const __grid_constant__ ResidueConsts rc) {
  constexpr int kUnits = 8 / kWarps;             // (row, chunk) pairs per CTA
  constexpr int kGroups = kWarps == 8 ? 2 : 1;   // groups of four values per lane
  __shared__ unsigned long long smax[8];
  __shared__ int slow[8];
  grid_launch_dependents();
  grid_dependency_wait();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int unit = warp / kWarps, wu = warp % kWarps;
  const int64_t u = blockIdx.x * static_cast<int64_t>(kUnits) + unit;
  const bool on = u < rows * nch;
  const int64_t r = on ? u / nch : 0, c = on ? u % nch : 0;
  const int64_t k0 = c * kc, k1 = min(K, k0 + kc);
  const bool live = on && !(tri && r < k0);
  const double* p = src + r * ld;
  double v[kGroups][4];
  unsigned long long mb = 0;
  uint32_t tail = 0;
#pragma unroll
  for (int g = 0; g < kGroups; ++g) {
    const int64_t k = k0 + 4 * (g * 32 * kWarps + wu * 32 + lane);
#pragma unroll
    for (int q = 0; q < 4; ++q) v[g][q] = 0.0;
    if (live && vec && k + 3 < k1) {
      const double2 a = *reinterpret_cast<const double2*>(p + k), b = *reinterpret_cast<const double2*>(p + k + 2);
      v[g][0] = a.x, v[g][1] = a.y, v[g][2] = b.x, v[g][3] = b.y;
    } else if (live) {
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (k + q < k1) v[g][q] = p[k + q];
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(v[g][q])) & ~(1ull << 63);
      mb = b > mb ? b : mb;
      tail |= static_cast<uint32_t>(b);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long b = __shfl_xor_sync(0xffffffffu, mb, o);
    mb = b > mb ? b : mb;
  }
  // the lowest bit that is set in any value of the warp: 2^(low - 1075)
  int low = INT_MIN;
  if (!__any_sync(0xffffffffu, (tail & 0x7FF) != 0)) {
    low = INT_MAX;
#pragma unroll
    for (int i = 0; i < 4 * kGroups; ++i) {
      const unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(v[i / 4][i % 4])) & ~(1ull << 63);
      const int E = static_cast<int>(b >> 52), z = __ffsll(static_cast<long long>(b & ((1ull << 52) - 1)));
      if (b != 0) low = min(low, max(E, 1) + (z != 0 ? z - 1 : 52));
    }
    low = __reduce_min_sync(0xffffffffu, low);
  }
  if constexpr (kWarps > 1) {
    if (lane == 0) smax[warp] = mb, slow[warp] = low;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
      const unsigned long long b = smax[unit * kWarps + w];
      mb = b > mb ? b : mb;
    }
  }
  if (!live) return;
  // e with max|a| < 2^e: a normal max = 1.f 2^(E - 1023) < 2^(E - 1022)
  int e = 0;
  bool finite = true;
  if (mb != 0) {
    const int E = static_cast<int>(mb >> 52);
    finite = E != 0x7FF;
    e = E != 0 ? E - 1022 : -1022;
  }
  if (wu == 0 && lane == 0) {
    ex[r * ex_stride + c] = static_cast<int16_t>(finite ? e : kNonFinite);
    if constexpr (kWarps > 1)
      for (int w = 1; w < kWarps; ++w) low = min(low, slow[warp + w]);
    int z = 0;
    if (finite && mb != 0 && low != INT_MIN) z = min(max(low - 1075 + bits - e, 0) / 6, 7);
    zeros[r * ex_stride + c] = static_cast<int8_t>(z);
    if (z != 0) atomicMax(zmax, z);
  }
  // the last chunk's last block is filled up with zeros
  const int64_t kw1 = (c == nch - 1) ? kb * kStepK : k1;
  // base of the chunk (of the whole operand unless it is triangular), its
  // blocks, and the row's place in it
  int64_t blocks = kb, place = r, kbase = 0, nrows = rows;
  if (tri) {
    dst += kModuli * kc * (c * rows - kc * (c * (c - 1) / 2));
    blocks = (kw1 - k0) / kStepK;
    kbase = k0;
    place = r - k0;
    nrows = rows - k0;
  }
  const int64_t plane = blocks * nrows * kStepK;
#pragma unroll
  for (int g = 0; g < kGroups; ++g) {
    const int64_t k = k0 + 4 * (g * 32 * kWarps + wu * 32 + lane);
    if (k >= kw1) continue;
    float l0[4], l1[4], l2[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) limbs_of(finite ? v[g][q] : 0.0, bits, e, l0[q], l1[q], l2[q]);
    __nv_bfloat16* d = dst + ((k - kbase) / kStepK * nrows + place) * kStepK + k % kStepK;
#pragma unroll
    for (int m = 0; m < kModuli; ++m) {
      if (m >= moduli) break;
      float t[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) t[q] = residue_of(l0[q], l1[q], l2[q], rc.p[m], rc.inv[m], rc.c16[m], rc.c32[m]);
      uint2 pk;
      pk.x = bf16_pair(t[0], t[1]);
      pk.y = bf16_pair(t[2], t[3]);
      *reinterpret_cast<uint2*>(d + m * plane) = pk;  // 8-byte aligned: k is a multiple of 4
    }
  }
}

// Row-major copy of the strictly lower triangle of a column-major n x n
// matrix (zeros on and above the diagonal).  The diagonal is kept out of the
// residues: it usually dominates its row, and integers relative to the row
// maximum would cost the off-diagonal entries their low bits; the product's
// last step applies it in FP64 instead.  With n0 > 0 the n0 x n0 diagonal
// blocks are zeroed as well (the trailing updates of the sliced schedule
// read only the entries outside them, and leaving the diagonal blocks out
// keeps their large entries from setting the row exponents).  Only chunks of
// kc columns that the row's residues keep are written.
__global__ void transpose_lower_kernel(const double* __restrict__ L, int64_t ldl, double* __restrict__ T, int64_t n,
                                       int64_t n0, int64_t kc) {
  __shared__ double tile[32][33];
  const int64_t bi = blockIdx.y * 32, bj = blockIdx.x * 32;  // source rows bi.., cols bj..
  if (bj >= ((bi + 31) / kc + 1) * kc) return;
  const int tx = threadIdx.x, ty = threadIdx.y;  // 32 x 8
  for (int yy = ty; yy < 32; yy += 8) {
    const int64_t i = bi + tx, j = bj + yy;
    double v = 0.0;
    if (i < n && j < n && i > j && (n0 == 0 || i / n0 != j / n0)) v = L[j * ldl + i];
    tile[yy][tx] = v;  // tile[col][row]
  }
  __syncthreads();
  for (int yy = ty; yy < 32; yy += 8) {
    const int64_t i = bi + yy, j = bj + tx;  // write row i, column j of T (row-major)
    if (i < n && j < n) T[i * n + j] = tile[tx][yy];
  }
}

// Row-major n x n0 copy of the rows of L~'s diagonal blocks below their
// diagonal: T(r, c) = L~(r, b n0 + c) for c < r - b n0 (b = r / n0), zero
// elsewhere; diag[r] = L~(r, r).  The diagonal stays out of the residues
// (applied in FP64 by the diagonal multiply): it dominates the rows of the
// inverse, and integers relative to it would leave the other entries few
// significant bits.
__global__ void transpose_diag_blocks_kernel(const double* __restrict__ L, int64_t ldl, double* __restrict__ T,
                                             double* __restrict__ diag, int64_t n, int64_t n0) {
  __shared__ double tile[32][33];
  const int64_t bi = blockIdx.y * 32, bj = blockIdx.x * 32;  // rows r, block columns c
  const int tx = threadIdx.x, ty = threadIdx.y;
  for (int yy = ty; yy < 32; yy += 8) {
    const int64_t r = bi + tx, c = bj + yy;
    double v = 0.0;
    if (r < n && c < n0) {
      const int64_t b0 = r / n0 * n0;
      if (b0 + c < r) v = L[(b0 + c) * ldl + r];
      if (b0 + c == r) diag[r] = L[r * ldl + r];
    }
    tile[yy][tx] = v;
  }
  __syncthreads();
  for (int yy = ty; yy < 32; yy += 8) {
    const int64_t r = bi + yy, c = bj + tx;
    if (r < n && c < n0) T[r * n0 + c] = tile[tx][yy];
  }
}

// -------------------------------------------------------------- product
// Chinese remainder constants of the first `n` moduli: with y_m the inverse
// of M / p_m modulo p_m, the integer x with residues r_m is sum_m r_m w_m, w_m =
// y_m M / p_m, less a multiple of M, and x / M the fraction of sum_m r_m y_m / p_m.
//
// By the fraction: limb[m] holds y_m / p_m to 72 binary places: the first 32
// (their products wrap modulo 1, as the fraction does), then two limbs of 20,
// of which 15 products with a byte sum to less than 2^31.  Rounded at 2^-72 and
// then at 2^-64 it leaves x off by at most 3.2 M 2^-64 (2^47.3 for 15 moduli),
// to either side alike, against roundings of 48-bit factors that add up to 2^51
// over a full chunk.
//
// Exactly: short factors are not rounded, and the fraction alone would lose
// exact results that eight 6-bit digits had (1 * 1 and 3 * 5 came out as
// 0.9999999999999988 and 14.999999999999995).  Pairs of at most nine digits
// (kExactDigits) are put together in integers of 128 bits (combine_checked):
// the fraction to 31 places (frac) gives the multiple of M and the bits of x
// from 2^96 on, the sums modulo 2^96 the others.  Not every pair takes this
// form because it costs 5 to 10 % where none is short (us: n = 3000, k = 200,
// n0 = 256 514 by the fraction, 569 exactly; n = 16384, k = 256, n0 = 2048
// 1215 and 1313; n = k = 8192 6280 and 6865).  An L of entries +-2^-14, all
// pairs short: 690, 1596 and 7009 us.
struct CrtConsts {
  int n;
  float p[kModuli], inv[kModuli];
  int limb[kModuli][3];
  double msc;  // M 2^-64
};

// Those of the exact form, which few products take: in constant memory, not
// among the arguments of every launch.
struct ExactConsts {
  int frac[kModuli];        // y_m / p_m times 2^31
  uint32_t w[kModuli][3];   // the words of w_m modulo 2^96, the lower two signed
  uint32_t m[3];            // those of M
  int top;                  // M 2^-79
};

constexpr int inverse_mod(int a, int p) {
  int y = 1;
  while (a * y % p != 1) ++y;  // a and p are coprime
  return y;
}

// v modulo 2^96 = w[0] + w[1] 2^32 + w[2] 2^64 with the lower two read as
// signed words.
constexpr void low_words(unsigned __int128 v, uint32_t (&w)[3]) {
  for (int i = 0; i < 3; ++i) {
    w[i] = static_cast<uint32_t>(v);
    v = (v >> 32) + (w[i] >> 31);  // a negative word takes one more of the next
  }
}

constexpr unsigned __int128 modulus_product(int n) {
  unsigned __int128 M = 1;
  for (int m = 0; m < n; ++m) M *= static_cast<unsigned>(kP[m]);
  return M;
}

constexpr ExactConsts make_exact_consts(int n) {
  ExactConsts c{};
  const unsigned __int128 M = modulus_product(n);
  for (int m = 0; m < n; ++m) {
    const unsigned p = static_cast<unsigned>(kP[m]);
    const unsigned y = static_cast<unsigned>(inverse_mod(static_cast<int>((M / p) % p), kP[m]));
    c.frac[m] = static_cast<int>(((static_cast<uint64_t>(y) << 32) / p + 1) >> 1);
    low_words(M / p * y, c.w[m]);
  }
  low_words(M, c.m);
  c.top = static_cast<int>(static_cast<int64_t>(M >> 79));
  return c;
}

__constant__ ExactConsts kExact[3] = {make_exact_consts(13), make_exact_consts(14), make_exact_consts(15)};


struct ProductArgs {
  int M, N, K, R, C;        // sizes, row tiles (of 128 or, for CTA pairs, 256 rows) and column tiles
  int a_row0, a_k0, b_row0, b_k0;  // first rows, and first blocks of 64 along K
  int a_kb, b_kb;           // blocks of 64 per modulus
  int GR, GC;               // tile group: GR x GC tiles, every modulus of one before the next
  int wave;                 // units (CTAs or pairs)
  int lower, mode;
  int bits;                 // bits of A plus bits of B
  uint2* resid;             // [128-row tile][modulus][8-column group][128 rows] bytes of 8 columns
  int item_cols;            // columns of an output tile that one CTA combines at a time: 16 or 32
  int depth;                // items a CTA holds: 1, or 2 to take one while another is combined
  int* ctrl;                // control words
  int* count;               // [128-row tile] reducing warps that have finished a modulus of it
  int* ready;               // finished 128-row tiles in the order they came, plus one (0: not written yet)
  int* taken;               // items taken of the tile at a list position (may run past the number there is)
  const int16_t* eA;        // A's exponents: eA[r a_ex] (already at the first row and the chunk)
  int64_t a_ex;
  const int16_t* eB;
  int64_t b_ex;
  const int8_t *zA, *zB;    // zero digits of their factors, beside the exponents
  const int *zmaxA, *zmaxB; // the most that a row of either operand has
  double* Y;
  int64_t ldy;
  const double* S;
  int64_t lds;
  const double* dg;
  const double* X;
  int64_t ldx;
  CrtConsts k;
};

// Control words: the list position below which every item has been taken,
// the output tiles finished (read together, 8 bytes), the CTAs that have
// ended; kZeros: a zmax for B, which stays.
constexpr long long kLingerNs = 20000;
constexpr int kHead = 0, kReady = 1, kExited = 2, kZeros = 4, kCtrlWords = 64;

constexpr int kMaxRegs = 96;  // 19 warps: five on one scheduler, whose file holds 512 registers a lane

template <int BN, bool kPair>
struct Shape {
  static constexpr uint32_t A_SL = 128u * 128u;
  static constexpr uint32_t B_SL = static_cast<uint32_t>(kPair ? BN / 2 : BN) * 128u;
  static constexpr uint32_t STAGE = A_SL + B_SL;  // per CTA
  static constexpr int STAGES = static_cast<int>(196608u / STAGE) < 8 ? static_cast<int>(196608u / STAGE) : 8;
  static constexpr size_t SMEM_BYTES = static_cast<size_t>(STAGES) * STAGE + 1024;
  static constexpr uint32_t TMEM_COLS = 2u * BN;  // two accumulator buffers: 128, 256 or 512
  static constexpr int kEpiWarps = 8;  // two per TMEM lane quadrant, half of the columns each
  static constexpr int kCombWarps = 8;  // 32 rows and half of an item's columns each
  static constexpr int kThreads = 64 + 32 * (kEpiWarps + kCombWarps) + 32;
  static constexpr int kSlabs = BN / 16;
  static constexpr int kTileRows = kPair ? 256 : 128;
  static_assert(BN == 64 || BN == 128 || BN == 256, "tile width");
};

// Tile number -> (modulus, row tile, column tile).  Groups of GR x GC output
// tiles, one after the other; within a group modulus by modulus, so that the
// CTAs in flight share one modulus' operand planes in L2 and a group's
// residues (GR GC BN 128 bytes per modulus) are still there when its last
// modulus puts them together.  With a triangular A the last row tiles carry
// the longest K ranges and run first.
__device__ __forceinline__ void tile_of(const ProductArgs& a, int lin, int& m, int& tm, int& tn) {
  const int nm = a.k.n;
  const int gr = lin / (a.GR * a.C * nm);
  const int g0 = gr * a.GR, gsz = min(a.GR, a.R - g0);
  int rem = lin - g0 * a.C * nm;
  const int gc = rem / (gsz * a.GC * nm);
  const int c0 = gc * a.GC, csz = min(a.GC, a.C - c0);
  rem -= gsz * c0 * nm;
  m = rem / (gsz * csz);
  rem -= m * gsz * csz;
  tn = c0 + rem / gsz;
  const int r = g0 + rem % gsz;
  tm = a.lower ? a.R - 1 - r : r;
}

template <int kRows>
__device__ __forceinline__ int k_steps(const ProductArgs& a, int tm) {
  const int kend = a.lower ? min(a.K, (tm + 1) * kRows) : a.K;
  return (kend + kStepK - 1) / kStepK;
}

// The t-th tile of unit u (a CTA or a pair), or -1.  The tiles are dealt in a
// snake (odd rounds in reverse), which evens out the K lengths of a
// triangular A: with straight rounds a unit met the same row of every tile
// group, and the units of the long rows took 2.7 times the average.
__device__ __forceinline__ int nth_tile(const ProductArgs& a, int u, int t, int total) {
  const int base = t * a.wave, w = min(a.wave, total - base);
  if (u >= w) return -1;
  return base + ((t & 1) ? w - 1 - u : u);
}

// FP32 integer sums of one modulus -> their residues as bytes (four per
// word): |v| < 2^24, the quotient's error stays below 0.02, |r| <= 92.
__device__ __forceinline__ uint32_t residue_byte(uint32_t v, float p, float inv) {
  const float f = __uint_as_float(v);
  const float q = fmaf(f, inv, kRound) - kRound;
  return __float_as_uint(fmaf(-p, q, f) + kRound);  // low byte: the residue in two's complement
}
__device__ __forceinline__ uint32_t pack4(uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  return __byte_perm(__byte_perm(a, b, 0x0040), __byte_perm(c, d, 0x0040), 0x5410);
}

// Byte j of w, sign-extended, in one instruction (a selector nibble with its
// top bit set gives copies of the byte's sign).
__device__ __forceinline__ int signed_byte(uint32_t w, int j) {
  int r;
  asm("prmt.b32 %0, %1, 0, %2;" : "=r"(r) : "r"(w), "r"(0x8880 + 0x1111 * j));
  return r;
}

// x 2^n where the result may leave the normal range.
__device__ __noinline__ double scaled_slow(double x, double msc, int n) { return ldexp(x * msc, n); }

// x 2^sc, rounded to the nearest double, from the sums over an output's
// residues (S: with frac, A0 .. A2: with the words of w).  frac's roundings
// leave x / M off by at most 2^-21.5, and |x| < 0.36 M: the nearest integer to
// S is the multiple of M, and the error of x's bits from 2^64 on is below 2^25.
__device__ __forceinline__ double exact_value(const ExactConsts& k, long long S, long long A0, long long A1, uint32_t A2,
                                              int sc) {
  const int q = static_cast<int>((S + (1ll << 30)) >> 31);
  const long long frac = S - (static_cast<long long>(q) << 31);
  A0 -= static_cast<long long>(q) * static_cast<int>(k.m[0]);
  A1 -= static_cast<long long>(q) * static_cast<int>(k.m[1]);
  A2 -= static_cast<uint32_t>(q) * k.m[2];
  A1 += A0 >> 32;
  A2 += static_cast<uint32_t>(A1 >> 32);
  // x = hi 2^64 + lo, the bits of hi from 32 on from the fraction
  const long long h = (frac * k.top) >> 16;
  long long hi = h + static_cast<int>(A2 - static_cast<uint32_t>(h));
  unsigned long long lo = (static_cast<unsigned long long>(A1) << 32) | static_cast<uint32_t>(A0);
  const bool neg = hi < 0;
  if (neg) {
    lo = 0 - lo;
    hi = ~hi + (lo == 0);
  }
  if (hi == 0 && lo == 0) return 0.0;
  // the 64 bits from the leading one on; hi is below 2^44
  const int lz = hi != 0 ? __clzll(hi) : __clzll(static_cast<long long>(lo));
  const unsigned long long t = hi != 0 ? (static_cast<unsigned long long>(hi) << lz) | (lo >> (64 - lz)) : lo << lz;
  const bool rest = (t & 0x3FF) != 0 || (hi != 0 && (lo << lz) != 0);
  const long long m = static_cast<long long>((t >> 11) + ((t >> 10) & 1 & (rest ? 1 : t >> 11)));
  const int e = (hi != 0 ? 127 : 63) - lz;  // x = 1.f 2^e
  const int E = e + sc >= -1022 && e + sc <= 1022 ? e + sc : e;
  const double v = __longlong_as_double(m + (static_cast<long long>(E + 1022) << 52));
  return E == e + sc ? (neg ? -v : v) : scaled_slow(neg ? -v : v, 1.0, sc);
}

// The sums of an output's residues with the limbs.
struct Fraction {
  uint32_t s0 = 0;
  int s1 = 0, s2 = 0;
  __device__ __forceinline__ void add(const CrtConsts& k, int m, int r) {
    s0 += static_cast<uint32_t>(r) * static_cast<uint32_t>(k.limb[m][0]);
    s1 += r * k.limb[m][1];
    s2 += r * k.limb[m][2];
  }
  // the fraction to 64 binary places, as a signed number in [-1/2, 1/2)
  __device__ __forceinline__ double value() const {
    return static_cast<double>(static_cast<long long>(
        (static_cast<unsigned long long>(s0) << 32) + (static_cast<unsigned long long>(static_cast<long long>(s1)) << 12) +
        static_cast<unsigned long long>(static_cast<long long>((s2 + 128) >> 8))));
  }
};

// One output from its base (S, or S - dg X) and its product's fraction f; ea
// and eb are the exponents of its factors.
__device__ __forceinline__ double apply_fraction(const ProductArgs& a, double f, int ea, int eb, double dg, double base) {
  const long long sign = a.mode == kRnsDiag ? 0 : static_cast<long long>(1ull << 63);
  const int sc = ea + eb - a.bits;
  if (sc >= -1050 && sc <= 970) {
    // msc = 1.x 2^31 to 1.x 2^45: the scale is normal in this range
    const double scale = __longlong_as_double((__double_as_longlong(a.k.msc) + (static_cast<long long>(sc) << 52)) ^ sign);
    // the diagonal term, usually the larger, is not rounded on its own
    return a.mode == kRnsDiag ? fma(dg, base, f * scale) : fma(f, scale, base);
  }
  if (ea == kNonFinite || eb == kNonFinite) return __longlong_as_double(0x7FF8000000000000ll);
  const double v = scaled_slow(f, a.k.msc, sc);
  return a.mode == kRnsDiag ? fma(dg, base, v) : base - v;
}

// combine_tile where the operands' zero digits allow exact pairs: a pair's
// product exactly if its factors are short, the others' by the fraction, so
// that an output depends on its own row and column alone.  A role of its own:
// a call from combine_tile's loop, never taken, made the kernel spill and cost
// 2 % at n = 3000, k = 200.
template <int BN>
__device__ __forceinline__ void combine_checked(const ProductArgs& a, int tile, int tm, int tn, int row, int cg0, int cg1) {
  const int grow = tm * 128 + row;
  if (grow >= a.M) return;
  const ExactConsts& k = kExact[a.k.n - 13];
  const int ea = a.eA[static_cast<int64_t>(grow) * a.a_ex], za = a.zA[static_cast<int64_t>(grow) * a.a_ex];
  const double dg = a.mode != kRnsUpdate ? a.dg[grow] : 0.0;
#pragma unroll 1
  for (int cg = cg0; cg < cg1; ++cg) {
    const int col0 = tn * BN + cg * 8;
    const uint2* rp = a.resid + (static_cast<int64_t>(tile) * a.k.n * (BN / 8) + cg) * 128 + row;
    uint2 rv[kModuli];
#pragma unroll
    for (int m = 0; m < kModuli; ++m)
      rv[m] = m < a.k.n ? __ldcg(rp + static_cast<int64_t>(m) * (BN / 8) * 128) : make_uint2(0, 0);
#pragma unroll 1
    for (int j = 0; j < 8; ++j) {
      const int64_t col = col0 + j;
      if (col >= a.N) break;
      const int eb = a.eB[col * a.b_ex];
      double base = a.S[col * a.lds + grow];
      if (a.mode == kRnsResidual) base = fma(-dg, a.X[col * a.ldx + grow], base);
      double y;
      if (za + a.zB[col * a.b_ex] >= kExactDigits) {  // both finite
        long long S = 0, A0 = 0, A1 = 0;
        uint32_t A2 = 0;
#pragma unroll
        for (int m = 0; m < kModuli; ++m) {
          const int r = signed_byte(j < 4 ? rv[m].x : rv[m].y, j & 3);
          S += static_cast<long long>(r) * k.frac[m];
          A0 += static_cast<long long>(r) * static_cast<int>(k.w[m][0]);
          A1 += static_cast<long long>(r) * static_cast<int>(k.w[m][1]);
          A2 += static_cast<uint32_t>(r) * k.w[m][2];
        }
        const double v = exact_value(k, S, A0, A1, A2, ea + eb - a.bits);
        y = a.mode == kRnsDiag ? fma(dg, base, v) : base - v;
      } else {
        Fraction f;
#pragma unroll
        for (int m = 0; m < kModuli; ++m) f.add(a.k, m, signed_byte(j < 4 ? rv[m].x : rv[m].y, j & 3));
        y = apply_fraction(a, f.value(), ea, eb, dg, base);
      }
      a.Y[col * a.ldy + grow] = y;
    }
  }
}

// Puts the integer products of the 8-column groups [cg0, cg1) of an output
// tile together from their residues and applies them, a row per lane.  Per
// output: 15 byte extractions and 45 multiply-adds, then a conversion and one
// or two FP64 operations.
template <int BN>
__device__ __forceinline__ void combine_tile(const ProductArgs& a, int tile, int tm, int tn, int row, int cg0, int cg1) {
  const int grow = tm * 128 + row;
  if (grow >= a.M) return;
  const int ea = a.eA[static_cast<int64_t>(grow) * a.a_ex];
  const double dg = a.mode != kRnsUpdate ? a.dg[grow] : 0.0;
  const int nm = a.k.n;
#pragma unroll 1
  for (int cg = cg0; cg < cg1; ++cg) {
    const int col0 = tn * BN + cg * 8;
    const int ncol = min(8, a.N - col0);
    if (ncol <= 0) break;
    // every load of the group in flight before the first use
    const uint2* rp = a.resid + (static_cast<int64_t>(tile) * nm * (BN / 8) + cg) * 128 + row;
    uint2 rv[kModuli];
#pragma unroll
    for (int m = 0; m < kModuli; ++m)
      rv[m] = m < nm ? __ldcg(rp + static_cast<int64_t>(m) * (BN / 8) * 128) : make_uint2(0, 0);
    const int16_t* eBp = a.eB + static_cast<int64_t>(col0) * a.b_ex;
    int eb8[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) eb8[j] = j < ncol ? eBp[static_cast<int64_t>(j) * a.b_ex] : 0;
    const double* Sp = a.S + static_cast<int64_t>(col0) * a.lds + grow;
    double base[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) base[j] = j < ncol ? Sp[static_cast<int64_t>(j) * a.lds] : 0.0;
    if (a.mode == kRnsResidual) {
      const double* Xp = a.X + static_cast<int64_t>(col0) * a.ldx + grow;
#pragma unroll
      for (int j = 0; j < 8; ++j)
        if (j < ncol) base[j] = fma(-dg, Xp[static_cast<int64_t>(j) * a.ldx], base[j]);
    }
    double* Yp = a.Y + static_cast<int64_t>(col0) * a.ldy + grow;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      Fraction f;
#pragma unroll
      for (int m = 0; m < kModuli; ++m) f.add(a.k, m, signed_byte(j < 4 ? rv[m].x : rv[m].y, j & 3));
      if (j >= ncol) continue;
      Yp[static_cast<int64_t>(j) * a.ldy] = apply_fraction(a, f.value(), ea, eb8[j], dg, base[j]);
    }
  }
}

// One CTA per SM; a tile is 128 x BN sums of one modulus.  Warp 0 loads
// (TMA, a ring of 48 KB stages at BN = 256), warp 1 owns TMEM and issues the
// MMAs into two accumulator buffers in turn, warps 2-9 reduce a finished
// buffer to bytes in global memory while the next tile's MMAs run.  The CTA
// that finishes the last modulus of an output tile (a counter per tile)
// appends the tile to a list; warp 18 of every CTA takes items of 128 x 32
// outputs from the list for its warps 10-17, which combine them beside the
// MMAs.  A CTA ends when its own tiles are finished and the list is empty:
// none waits for another for longer than kLingerNs, so they need not be
// co-resident, and the last to end leaves the control words zero.
//
// Bound by the tensor pipe where K and the columns are long (the residual at
// n = 16384, k = 4096, 14 moduli: 9.8 ms, 1570 TFLOP/s of bf16 where the
// box's sustained cuBLAS rate is 1728; 20.2 ms before, with 28 digit-pair
// products), by reading A's residues from HBM where N is one tile
// (n = 16384, k = 256), by the last steps' latency where there are few tiles
// (256 x 200 at K = 256: 16 us).  What the division of the work is for
// (measured on that residual): 40 ms with the reducing warps of the finishing
// CTA combining, which made it late, hence the last at its next tiles too;
// 18-22 ms with other warps of the finishing CTA combining whole tiles (SMs
// idle 40 % of the time behind the last ones); 21 ms with one
// compare-and-swap counter for all items (one success per round trip to L2).
//
// kPair: two CTAs of a cluster work on 256 x BN tiles (cta_group::2): each
// loads its 128 rows of A and half of B's rows, 32 KB per step of K at BN =
// 256 against 48 KB for a CTA alone, since operand delivery from L2, not the
// tensor pipe, limits the 128 x 256 tiles.
template <int BN, bool kPair>
__global__ void __maxnreg__(kMaxRegs)
    rns_product_kernel(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB,
                       const __grid_constant__ ProductArgs a, int* err) {
  using S = Shape<BN, kPair>;
  constexpr int STAGES = S::STAGES;
  constexpr uint32_t IDESC = kPair ? tc::idesc_m256_bf16(BN) : tc::idesc_m128(BN, false);
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  __shared__ uint64_t full_bar[STAGES], empty_bar[STAGES], tfull_bar[2], tempty_bar[2];
  __shared__ uint64_t qfull_bar[2], qempty_bar[2];
  __shared__ int queue[2];  // items to combine (tile * items + part), -1: no more
  __shared__ uint32_t tmem_base_sh;
  __shared__ int abort_sh, done_sh;  // done_sh: reducing warps that have ended
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = kPair ? static_cast<int>(tc::cluster_rank()) : 0;
  const int unit = kPair ? static_cast<int>(blockIdx.x >> 1) : static_cast<int>(blockIdx.x);
  const int total = a.R * a.C * a.k.n;
  const int out_tiles = (a.M + 127) / 128 * a.C;
  const int items = BN / a.item_cols;  // per output tile
  if (threadIdx.x == 0) {
    tc::prefetch_map(&mapA);
    tc::prefetch_map(&mapB);
    for (int q = 0; q < STAGES; ++q) {
      tc::mbar_init(&full_bar[q], 1);
      tc::mbar_init(&empty_bar[q], 1);
    }
    for (int b = 0; b < 2; ++b) {
      tc::mbar_init(&tfull_bar[b], 1);
      tc::mbar_init(&tempty_bar[b], (kPair ? 2 : 1) * S::kEpiWarps);
    }
    for (int q = 0; q < 2; ++q) {
      tc::mbar_init(&qfull_bar[q], 1);
      tc::mbar_init(&qempty_bar[q], S::kCombWarps);
    }
    abort_sh = 0;
    done_sh = 0;
    tc::fence_mbar_init();
  }
  if (warp == 1) {
    if constexpr (kPair) {
      tc::tmem_alloc_pair(&tmem_base_sh, S::TMEM_COLS);
    } else {
      tc::tmem_alloc(&tmem_base_sh, S::TMEM_COLS);
      tc::tmem_relinquish();
    }
  }
  tc::tc_fence_before();
  __syncwarp();
  if constexpr (kPair) tc::cluster_sync();
  else __syncthreads();
  tc::tc_fence_after();
  const uint32_t tbase = tmem_base_sh;
  volatile int* abort_flag = &abort_sh;
  grid_dependency_wait();

  if (warp == 0) {
    if (lane == 0) {
      int it = 0, lin;
      bool ok = true;
      for (int t = 0; ok && (lin = nth_tile(a, unit, t, total)) >= 0; ++t) {
        int m, tm, tn;
        tile_of(a, lin, m, tm, tn);
        const int nkb = k_steps<S::kTileRows>(a, tm);
        for (int i = 0; i < nkb; ++i, ++it) {
          const int q = it % STAGES;
          if (it >= STAGES && !tc::mbar_wait(&empty_bar[q], ((it / STAGES) - 1) & 1, abort_flag)) {
            ok = false;
            break;
          }
          uint8_t* sa = smem + static_cast<size_t>(q) * S::STAGE;
          const int az = m * a.a_kb + a.a_k0 + i, ay = a.a_row0 + tm * S::kTileRows + rank * 128;
          const int bz = m * a.b_kb + a.b_k0 + i, by = a.b_row0 + tn * BN + rank * (BN / 2);
          if constexpr (kPair) {
            // both CTAs' loads complete on the leader's barrier
            if (rank == 0) tc::mbar_arrive_expect_tx(&full_bar[q], 2 * S::STAGE);
            const uint32_t bar = tc::cluster_addr(&full_bar[q], 0);
            tc::tma_load_3d_pair(sa, &mapA, bar, 0, ay, az);
            tc::tma_load_3d_pair(sa + S::A_SL, &mapB, bar, 0, by, bz);
          } else {
            tc::mbar_arrive_expect_tx(&full_bar[q], S::STAGE);
            tc::tma_load_3d(sa, &mapA, &full_bar[q], 0, ay, az);
            tc::tma_load_3d(sa + S::A_SL, &mapB, &full_bar[q], 0, by, bz);
          }
        }
      }
      // A pair's copies complete on the leader's barriers alone, so the leader
      // waits for both CTAs'; the other one's are no later than its wait that
      // gave up, hundreds of polls.
      if (!ok && rank == 0) tc::drain_ring(full_bar, STAGES, it);
      // the leader's last commits have landed here before this CTA may end
      if constexpr (kPair)
        for (int i = max(0, it - STAGES); ok && i < it; ++i)
          ok = tc::mbar_wait(&empty_bar[i % STAGES], (i / STAGES) & 1, abort_flag);
    }
  } else if (warp == 1) {
    if (lane == 0 && rank == 0) {
      int it = 0, lin;
      bool ok = true;
      for (int t = 0; ok && (lin = nth_tile(a, unit, t, total)) >= 0; ++t) {
        int m, tm, tn;
        tile_of(a, lin, m, tm, tn);
        const int nkb = k_steps<S::kTileRows>(a, tm);
        const int b = t & 1, use = t >> 1;
        if (use > 0 && !tc::mbar_wait(&tempty_bar[b], (use - 1) & 1, abort_flag)) break;
        tc::tc_fence_after();
        const uint32_t acc = tbase + static_cast<uint32_t>(b * BN);
        for (int i = 0; i < nkb; ++i, ++it) {
          const int q = it % STAGES;
          if (!tc::mbar_wait(&full_bar[q], (it / STAGES) & 1, abort_flag)) {
            ok = false;
            break;
          }
          tc::tc_fence_after();
          const uint32_t sa = tc::smem_u32(smem + static_cast<size_t>(q) * S::STAGE);
          const uint64_t ad = tc::desc_kmajor<128>(sa), bd = tc::desc_kmajor<128>(sa + S::A_SL);
#pragma unroll
          for (int kk = 0; kk < 4; ++kk) {  // +32 bytes along K per MMA: start address field += 2
            const uint32_t accumulate = (i > 0 || kk > 0) ? 1u : 0u;
            if constexpr (kPair) tc::mma_pair(acc, ad + 2u * kk, bd + 2u * kk, IDESC, accumulate);
            else tc::mma<false>(acc, ad + 2u * kk, bd + 2u * kk, IDESC, accumulate);
          }
          if constexpr (kPair) tc::mma_commit_pair(&empty_bar[q]);
          else tc::mma_commit(&empty_bar[q]);
        }
        if (!ok) break;
        if constexpr (kPair) tc::mma_commit_pair(&tfull_bar[b]);
        else tc::mma_commit(&tfull_bar[b]);
      }
    }
  } else if (warp < 2 + S::kEpiWarps) {
    const int quad = warp & 3;  // the TMEM lane quadrant this warp may read
    const int half = (warp - 2) >> 2;
    const int row = quad * 32 + lane;
    // Publishes this warp's bytes of a tile's modulus and counts it; the last
    // warp of the last modulus makes the tile ready.  Called after the next
    // tile's first reads, when the stores have long drained: the fence and
    // the atomic would otherwise add about 2 us to every tile.
    int pending = -1;
    auto publish = [&]() {
      __syncwarp();
      if (lane == 0 && pending >= 0) {
        __threadfence();
        if (atomicAdd(a.count + pending, 1) == a.k.n * S::kEpiWarps - 1) {
          __threadfence();
          atomicExch(a.ready + atomicAdd(a.ctrl + kReady, 1), pending + 1);
        }
      }
      pending = -1;
    };
    int lin;
    for (int t = 0; (lin = nth_tile(a, unit, t, total)) >= 0; ++t) {
      int m, tm, tn;
      tile_of(a, lin, m, tm, tn);
      const int b = t & 1, use = t >> 1;
      if (!tc::mbar_wait(&tfull_bar[b], use & 1, abort_flag)) break;
      tc::tc_fence_after();
      const float p = a.k.p[m], inv = a.k.inv[m];
      const int row_tile = kPair ? 2 * tm + rank : tm;
      const int tile = row_tile * a.C + tn;
      const bool live = row_tile * 128 < a.M;  // a pair's second half may lie past the last row
      uint2* out = a.resid + (static_cast<int64_t>(tile) * a.k.n + m) * (BN / 8) * 128 + row;
      const uint32_t acc = tbase + (static_cast<uint32_t>(quad * 32) << 16) + static_cast<uint32_t>(b * BN);
      if (live) {
#pragma unroll 1
        for (int sl = half * (S::kSlabs / 2); sl < (half + 1) * (S::kSlabs / 2); sl += 2) {
          uint32_t v0[16], v1[16];
          tc::tmem_ld16(acc + static_cast<uint32_t>(sl * 16), v0);
          tc::tmem_ld16(acc + static_cast<uint32_t>(sl * 16 + 16), v1);
          tc::tmem_wait_ld();
          uint32_t w0[4], w1[4];
#pragma unroll
          for (int g = 0; g < 4; ++g) {
            w0[g] = pack4(residue_byte(v0[4 * g], p, inv), residue_byte(v0[4 * g + 1], p, inv),
                          residue_byte(v0[4 * g + 2], p, inv), residue_byte(v0[4 * g + 3], p, inv));
            w1[g] = pack4(residue_byte(v1[4 * g], p, inv), residue_byte(v1[4 * g + 1], p, inv),
                          residue_byte(v1[4 * g + 2], p, inv), residue_byte(v1[4 * g + 3], p, inv));
          }
          if (pending >= 0) publish();
          __stcg(out + 2 * sl * 128, make_uint2(w0[0], w0[1]));
          __stcg(out + (2 * sl + 1) * 128, make_uint2(w0[2], w0[3]));
          __stcg(out + (2 * sl + 2) * 128, make_uint2(w1[0], w1[1]));
          __stcg(out + (2 * sl + 3) * 128, make_uint2(w1[2], w1[3]));
        }
      }
      tc::tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        if (kPair && rank != 0) tc::mbar_arrive_cluster(tc::cluster_addr(&tempty_bar[b], 0));
        else tc::mbar_arrive(&tempty_bar[b]);
      }
      if (live) pending = tile;
    }
    publish();
    if (lane == 0) {
      __threadfence();  // this warp's list entries before its end
      atomicAdd(&done_sh, 1);
    }
  } else if (warp < 2 + S::kEpiWarps + S::kCombWarps) {
    const int w = warp - 2 - S::kEpiWarps;
    const int groups = a.item_cols / 16;  // 8-column groups per warp
    // zero digits are rare: the operands' most settle which form runs
    auto combine_items = [&](auto checked) {
      for (int i = 0;; ++i) {
        const int q = i & 1;
        if (!tc::mbar_wait(&qfull_bar[q], (i >> 1) & 1, abort_flag)) break;
        const int item = queue[q];
        if (item < 0) break;
        const int tile = item / items;
        const int cg0 = item % items * (2 * groups) + (w >> 2) * groups;
        if constexpr (decltype(checked)::value)
          combine_checked<BN>(a, tile, tile / a.C, tile % a.C, (w & 3) * 32 + lane, cg0, cg0 + groups);
        else
          combine_tile<BN>(a, tile, tile / a.C, tile % a.C, (w & 3) * 32 + lane, cg0, cg0 + groups);
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(&qempty_bar[q]);
      }
    };
    if (*a.zmaxA + *a.zmaxB >= kExactDigits) combine_items(std::true_type());
    else combine_items(std::false_type());
  } else {
    int pushed = 0;
    // true once the item `back` before the next one has been combined
    auto combined = [&](int back) {
      const int i = pushed - back;
      return i < 0 || tc::mbar_wait(&qempty_bar[i & 1], (i >> 1) & 1, abort_flag);
    };
    auto push = [&](int entry) {
      if (lane == 0) {
        queue[pushed & 1] = entry;
        tc::mbar_arrive(&qfull_bar[pushed & 1]);
      }
      ++pushed;
    };
    bool ok = true;
    long long t_done = 0;
    while (ok && __all_sync(0xffffffffu, combined(a.depth))) {
      // the end is read before the list: what this CTA appended is seen
      const bool done = *const_cast<volatile int*>(&done_sh) == S::kEpiWarps;
      if (done) __threadfence();
      const unsigned long long both = *reinterpret_cast<volatile unsigned long long*>(a.ctrl);
      const int head = static_cast<int>(both & 0xffffffffu), left = static_cast<int>(both >> 32) - head;
      // a lane per list position from the head on
      const bool listed = lane < left;
      const bool spent = listed && *const_cast<volatile int*>(a.taken + head + lane) >= items;
      const unsigned open = __ballot_sync(0xffffffffu, listed && !spent);
      const unsigned gone = __ballot_sync(0xffffffffu, spent);
      if (lane == 0 && (gone & 1u)) atomicMax(a.ctrl + kHead, head + (gone == ~0u ? 32 : __ffs(~gone) - 1));
      if (open) {
        // CTAs that look at the same time spread over the open positions
        const int pick = __fns(open, 0, 1 + static_cast<int>(blockIdx.x) % __popc(open));
        int item = -1;
        if (lane == pick) {
          const int part = atomicAdd(a.taken + head + lane, 1);
          if (part < items) {
            // the entry follows its count at once
            const volatile int* entry = a.ready + head + lane;
            const long long t0 = tc::globaltimer_ns();
            int tile;
            while ((tile = *entry) == 0)
              if (tc::globaltimer_ns() - t0 > tc::kMbarWaitNs) break;
            __threadfence();
            item = tile > 0 ? (tile - 1) * items + part : -2;
          }
        }
        item = __shfl_sync(0xffffffffu, item, pick);
        if (item >= 0) push(item);
        if (item == -2) {
          *abort_flag = 1;
          ok = false;
        }
      } else if (left <= 32) {
        // With its own tiles finished a CTA stays a little for the others'
        // last ones (a bounded time: they may not even have started).
        if (done && t_done == 0) t_done = tc::globaltimer_ns();
        const bool leave = done && (head + left >= out_tiles || tc::globaltimer_ns() - t_done > kLingerNs);
        if (__any_sync(0xffffffffu, leave || *abort_flag)) break;
        __nanosleep(100);
      }
    }
    if (__all_sync(0xffffffffu, combined(2))) push(-1);
  }
  // a pair's CTAs stay until no signal to the other is under way
  if constexpr (kPair) {
    __syncwarp();
    tc::cluster_sync();
  } else {
    __syncthreads();
  }
  if (warp == 1) {
    tc::tc_fence_after();
    if constexpr (kPair) tc::tmem_dealloc_pair(tbase, S::TMEM_COLS);
    else tc::tmem_dealloc(tbase, S::TMEM_COLS);
  }
  if (threadIdx.x == 0 && abort_sh) atomicExch(err, 1);
  // the last CTA to end clears the control words for the next product
  if (warp == 2) {
    int last = 0;
    if (lane == 0) {
      __threadfence();
      last = atomicAdd(a.ctrl + kExited, 1) == static_cast<int>(gridDim.x) - 1;
    }
    if (__shfl_sync(0xffffffffu, last, 0)) {
      for (int i = lane; i < out_tiles; i += 32) a.count[i] = a.ready[i] = a.taken[i] = 0;
      if (lane < 3) a.ctrl[lane] = 0;
    }
  }
}

}  // namespace rns

// ---------------------------------------------------------------- host
namespace {

using rns::kP;

rns::ResidueConsts make_residue_consts() {
  rns::ResidueConsts c{};
  for (int m = 0; m < kModuli; ++m) {
    const int p = kP[m];
    auto sym = [p](int64_t v) {
      const int64_t r = v % p;
      return static_cast<float>(2 * r > p ? r - p : r);
    };
    c.p[m] = static_cast<float>(p);
    c.inv[m] = 1.f / static_cast<float>(p);
    c.c16[m] = sym(int64_t(1) << 16);
    c.c32[m] = sym(int64_t(1) << 32);
  }
  return c;
}

rns::CrtConsts make_crt_consts(int n) {
  rns::CrtConsts c{};
  c.n = n;
  const unsigned __int128 M = rns::modulus_product(n);
  for (int m = 0; m < n; ++m) {
    const int p = kP[m];
    c.p[m] = static_cast<float>(p);
    c.inv[m] = 1.f / static_cast<float>(p);
    uint64_t rem = static_cast<uint64_t>(
        rns::inverse_mod(static_cast<int>((M / static_cast<unsigned>(p)) % static_cast<unsigned>(p)), p));
    for (int q = 0; q < 3; ++q) {
      rem <<= q == 0 ? 32 : 20;
      c.limb[m][q] = static_cast<int>(static_cast<uint32_t>(rem / static_cast<unsigned>(p)));
      rem %= static_cast<unsigned>(p);
    }
    c.limb[m][2] += 2 * rem >= static_cast<unsigned>(p);  // to nearest
  }
  c.msc = static_cast<double>(M) * 0x1p-64;
  return c;
}

const rns::CrtConsts& crt_consts(int n) {
  static const rns::CrtConsts k13 = make_crt_consts(13), k14 = make_crt_consts(14), k15 = make_crt_consts(15);
  return n == 13 ? k13 : n == 14 ? k14 : k15;
}

inline size_t al256(size_t x) { return (x + 255) / 256 * 256; }

// Column tile: 256 wide (the rate of 128 x 256 MMAs and the fewest operand
// bytes per product), narrower where that leaves less padding.
inline int tile_cols(int64_t N) { return N <= 64 ? 64 : N <= 128 ? 128 : 256; }

// Residue bytes of one launch: more column tiles than fit go in several
// launches one after the other.  At 15 moduli the bytes of about 1000 output
// tiles, 100 waves of tiles on 152 SMs.
constexpr int64_t kResidueBytes = 512ll << 20;

struct TilePlan {
  int bn;
  int64_t R, C;  // row and column tiles
  int64_t cap;   // output tiles whose residues the scratch holds: at least a column of tiles
};
TilePlan tile_plan(int64_t M, int64_t N) {
  TilePlan t;
  t.bn = tile_cols(N);
  t.R = (M + 127) / 128;
  t.C = (N + t.bn - 1) / t.bn;
  t.cap = std::min(t.R * t.C, std::max<int64_t>(t.R, kResidueBytes / (128ll * t.bn * kModuli)));
  return t;
}

template <int BN, bool kPair>
cudaError_t launch_product(const CUtensorMap& ma, const CUtensorMap& mb, const rns::ProductArgs& a, unsigned units,
                           int* err, cudaStream_t s) {
  using S = rns::Shape<BN, kPair>;
  auto kern = rns::rns_product_kernel<BN, kPair>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(S::SMEM_BYTES));
  if (e != cudaSuccess) return e;
  e = launch_dependent(kern, dim3(kPair ? 2 * units : units), dim3(S::kThreads), S::SMEM_BYTES, s, kPair ? 2 : 1, ma, mb, a,
                       err);
  count_launch();
  return e != cudaSuccess ? e : cudaGetLastError();
}

template <int kWarps>
cudaError_t launch_residues(const double* src, int64_t ld, int64_t K, const RnsOperand& o, RnsClass c, bool vec,
                            const rns::ResidueConsts& rc, cudaStream_t s) {
  const int64_t units = o.rows * o.nch, per = 8 / kWarps;
  return launch_dependent(rns::residue_rows_kernel<kWarps>, dim3(static_cast<unsigned>((units + per - 1) / per)), dim3(256),
                          0, s, 1, src, ld, o.rows, K, o.nch, o.kc, o.ex_ld, o.res, o.kb, o.ex, o.zeros, o.zmax, c.moduli, c.bits,
                          o.tri ? 1 : 0, vec ? 1 : 0, rc);
}

}  // namespace

// Residues of a rows x K operand: every chunk's moduli x blocks x rows x 64.
static size_t residue_bytes(int64_t rows, int64_t K, int64_t kc, bool tri) {
  constexpr int64_t kS = rns::kStepK;
  size_t values = 0;
  if (!tri) {
    values = static_cast<size_t>((K + kS - 1) / kS) * kS * rows;
  } else {
    for (int64_t k0 = 0; k0 < K; k0 += kc)
      values += static_cast<size_t>((std::min(kc, K - k0) + kS - 1) / kS) * kS * (rows - k0);
  }
  return al256(sizeof(__nv_bfloat16) * kModuli * values);
}

size_t rns_operand_bytes(int64_t rows, int64_t K, int64_t kc, bool tri) {
  // residues, a word for zmax, exponents, zero digits
  const size_t pairs = static_cast<size_t>(rows) * ((K + kc - 1) / kc);
  return residue_bytes(rows, K, kc, tri) + 256 + al256(sizeof(int16_t) * pairs) + al256(pairs);
}

RnsOperand rns_operand_view(void* base, int64_t rows, int64_t K, int64_t kc, bool tri) {
  RnsOperand o;
  o.rows = rows;
  o.K = K;
  o.kb = (K + rns::kStepK - 1) / rns::kStepK;
  o.kc = kc;
  o.nch = o.ex_ld = (K + kc - 1) / kc;
  o.tri = tri;
  o.res = static_cast<__nv_bfloat16*>(base);
  unsigned char* p = static_cast<unsigned char*>(base) + residue_bytes(rows, K, kc, tri);
  o.zmax = reinterpret_cast<int*>(p);
  o.ex = reinterpret_cast<int16_t*>(p + 256);
  o.zeros = reinterpret_cast<int8_t*>(p + 256 + al256(sizeof(int16_t) * static_cast<size_t>(rows) * o.nch));
  return o;
}

RnsOperand rns_chunk(const RnsOperand& o, int64_t c) {
  RnsOperand v = o;
  const int64_t k0 = c * o.kc;
  v.tri = false;
  v.rows = o.rows - k0;
  v.K = std::min(o.kc, o.K - k0);
  v.kb = (v.K + rns::kStepK - 1) / rns::kStepK;
  v.nch = 1;
  v.res += kModuli * o.kc * (c * o.rows - o.kc * (c * (c - 1) / 2));
  v.ex += k0 * o.ex_ld + c;
  v.zeros += k0 * o.ex_ld + c;
  return v;
}

cudaError_t rns_rows(const double* src, int64_t ld, int64_t K, const RnsOperand& o, RnsClass c, cudaStream_t s) {
  if (K < 1 || K > o.K || (K < o.K && o.nch != 1) || o.kc > kChunk || c.moduli < 1 || c.moduli > kModuli ||
      c.bits < 1 || c.bits > kBitsFull)
    return cudaErrorInvalidValue;
  if (o.rows == 0) return cudaSuccess;
  static const rns::ResidueConsts rc = make_residue_consts();
  // pairs of values in 16-byte loads where every row starts on one
  const bool vec = (reinterpret_cast<uintptr_t>(src) & 15) == 0 && ld % 2 == 0;
  // as many warps per (row, chunk) as it has groups of 128 values (the
  // padded row of a single chunk included)
  const int64_t w = std::min<int64_t>(o.kc, o.kb * rns::kStepK);
  const cudaError_t e = w <= 128   ? launch_residues<1>(src, ld, K, o, c, vec, rc, s)
                        : w <= 256 ? launch_residues<2>(src, ld, K, o, c, vec, rc, s)
                        : w <= 512 ? launch_residues<4>(src, ld, K, o, c, vec, rc, s)
                                   : launch_residues<8>(src, ld, K, o, c, vec, rc, s);
  count_launch();
  return e != cudaSuccess ? e : cudaGetLastError();
}

static cudaError_t transpose_and_reduce(const double* L, int64_t ldl, int64_t n, int64_t n0, const RnsOperand& o,
                                        double* tmp, cudaStream_t s) {
  if (!o.tri || o.rows != n) return cudaErrorInvalidValue;
  dim3 grid(static_cast<unsigned>((n + 31) / 32), static_cast<unsigned>((n + 31) / 32));
  rns::transpose_lower_kernel<<<grid, dim3(32, 8), 0, s>>>(L, ldl, tmp, n, n0, o.kc);
  count_launch();
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaMemsetAsync(o.zmax, 0, sizeof(int), s);
  if (e != cudaSuccess) return e;
  return rns_rows(tmp, n, n, o, RnsClass{kModuli, kBitsFull}, s);
}

cudaError_t rns_lower_rows(const double* L, int64_t ldl, int64_t n, const RnsOperand& o, double* tmp, cudaStream_t s) {
  return transpose_and_reduce(L, ldl, n, 0, o, tmp, s);
}

cudaError_t rns_offdiag_block_rows(const double* Lt, int64_t ldt, int64_t n, int64_t n0, const RnsOperand& off,
                                   double* tmp, cudaStream_t s) {
  if (off.rows != n || off.K != n || off.kc != n0) return cudaErrorInvalidValue;
  return transpose_and_reduce(Lt, ldt, n, n0, off, tmp, s);
}

cudaError_t rns_inverse_block_rows(const double* Lt, int64_t ldt, int64_t n, int64_t n0, const RnsOperand& inv,
                                   double* diag, double* tmp, cudaStream_t s) {
  if (inv.rows != n || inv.K != n0 || inv.nch != 1) return cudaErrorInvalidValue;
  dim3 grid(static_cast<unsigned>((n0 + 31) / 32), static_cast<unsigned>((n + 31) / 32));
  rns::transpose_diag_blocks_kernel<<<grid, dim3(32, 8), 0, s>>>(Lt, ldt, tmp, diag, n, n0);
  count_launch();
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaMemsetAsync(inv.zmax, 0, sizeof(int), s);
  if (e != cudaSuccess) return e;
  return rns_rows(tmp, n0, n0, inv, RnsClass{kModuli, kBitsFull}, s);
}

// The control words, and three words per output tile.
static size_t control_bytes(int64_t tiles) {
  return al256(sizeof(int) * (rns::kCtrlWords + 3 * static_cast<size_t>(tiles)));
}

size_t rns_scratch_bytes(int64_t M, int64_t N) {
  const TilePlan t = tile_plan(M, N);
  return control_bytes(t.cap) + static_cast<size_t>(t.cap) * 128 * t.bn * kModuli;
}

RnsScratch rns_scratch_view(void* base, int64_t M, int64_t N) {
  RnsScratch sc;
  sc.tiles = tile_plan(M, N).cap;
  sc.ctrl = static_cast<int*>(base);
  sc.zmax = sc.ctrl + rns::kZeros;
  sc.resid = static_cast<unsigned char*>(base) + control_bytes(sc.tiles);
  return sc;
}

cudaError_t rns_scratch_clear(const RnsScratch& sc, cudaStream_t s) {
  return cudaMemsetAsync(sc.ctrl, 0, control_bytes(sc.tiles), s);
}

cudaError_t rns_product(const RnsProduct& p, const RnsScratch& sc, int* err, cudaStream_t s) {
  if (p.M <= 0 || p.N <= 0) return cudaSuccess;
  // [k0, k0 + K) within one chunk of either factor, from a whole block on
  if (p.A.tri || p.B.tri || p.K < 1 || p.a_k0 / p.A.kc != (p.a_k0 + p.K - 1) / p.A.kc || p.b_k0 / p.B.kc != (p.b_k0 + p.K - 1) / p.B.kc ||
      p.a_k0 + p.K > p.A.K || p.b_k0 + p.K > p.B.K || p.a_row0 < 0 || p.a_row0 + p.M > p.A.rows || p.b_row0 < 0 ||
      p.b_row0 + p.N > p.B.rows || p.a_k0 % rns::kStepK != 0 || p.b_k0 % rns::kStepK != 0 || p.K > kChunk || !p.S || !p.Y ||
      (p.mode != kRnsUpdate && !p.dg) || (p.mode == kRnsResidual && !p.X))
    return cudaErrorInvalidValue;
  const TilePlan t = tile_plan(p.M, p.N);
  const int64_t Cp = std::min(t.C, sc.tiles / t.R);  // column tiles per launch
  if (Cp < 1 || t.R * Cp * kModuli > INT_MAX / 2 || p.A.rows > INT_MAX / 2 || p.B.rows > INT_MAX / 2 ||
      std::max(p.A.kb, p.B.kb) * kModuli > INT_MAX / 2)
    return cudaErrorInvalidValue;
  CUtensorMap ma, mb;
  // pairs unless the second CTA's rows would all lie past the last one
  const bool pair = p.M > 128;
  constexpr int kS = rns::kStepK;
  if (!tc::make_kmajor_map(&ma, p.A.res, false, kS, p.A.rows, kS, kModuli * p.A.kb, p.A.rows * kS, 128, 1, 128) ||
      !tc::make_kmajor_map(&mb, p.B.res, false, kS, p.B.rows, kS, kModuli * p.B.kb, p.B.rows * kS,
                           pair ? t.bn / 2 : t.bn, 1, 128))
    return cudaErrorInvalidValue;
  rns::ProductArgs a;
  a.M = static_cast<int>(p.M);
  a.K = static_cast<int>(p.K);
  a.R = static_cast<int>(pair ? (t.R + 1) / 2 : t.R);
  a.a_row0 = static_cast<int>(p.a_row0);
  a.a_k0 = static_cast<int>(p.a_k0 / rns::kStepK);
  a.b_k0 = static_cast<int>(p.b_k0 / rns::kStepK);
  a.a_kb = static_cast<int>(p.A.kb);
  a.b_kb = static_cast<int>(p.B.kb);
  a.lower = p.lower ? 1 : 0;
  a.mode = p.mode;
  a.bits = kBitsFull + p.cls.bits;
  a.ctrl = sc.ctrl;
  a.count = sc.ctrl + rns::kCtrlWords;
  a.ready = a.count + sc.tiles;
  a.taken = a.ready + sc.tiles;
  a.resid = static_cast<uint2*>(sc.resid);
  a.eA = p.A.ex + p.a_row0 * p.A.ex_ld + p.a_k0 / p.A.kc;
  a.a_ex = p.A.ex_ld;
  a.b_ex = p.B.ex_ld;
  a.zA = p.A.zeros + p.a_row0 * p.A.ex_ld + p.a_k0 / p.A.kc;
  a.zmaxA = p.A.zmax;
  a.zmaxB = p.B.zmax;
  a.ldy = p.ldy;
  a.lds = p.lds;
  a.dg = p.dg;
  a.ldx = p.ldx;
  a.k = crt_consts(p.cls.moduli);
  const int64_t sms = device_sm_count();
  for (int64_t c0 = 0; c0 < t.C; c0 += Cp) {
    const int64_t col0 = c0 * t.bn, ncol = std::min(p.N - col0, Cp * t.bn);
    a.N = static_cast<int>(ncol);
    a.C = static_cast<int>((ncol + t.bn - 1) / t.bn);
    a.GC = std::min(a.C, 8);
    a.GR = std::max(1, (pair ? 32 : 64) / a.GC);
    a.b_row0 = static_cast<int>(p.b_row0 + col0);
    const int64_t b_at = (p.b_row0 + col0) * p.B.ex_ld + p.b_k0 / p.B.kc;
    a.eB = p.B.ex + b_at;
    a.zB = p.B.zeros + b_at;
    a.Y = p.Y + col0 * p.ldy;
    a.S = p.S + col0 * p.lds;
    a.X = p.X ? p.X + col0 * p.ldx : nullptr;
    const int64_t total = static_cast<int64_t>(a.R) * a.C * a.k.n;
    a.wave = static_cast<int>(std::min(pair ? std::max<int64_t>(1, sms / 2) : sms, total));
    // small products: narrow items, one at a time, so that every CTA gets some
    const int64_t ctas = pair ? 2 * a.wave : a.wave;
    const bool small = (p.M + 127) / 128 * a.C * (t.bn / 32) < 2 * ctas;
    a.item_cols = small ? 16 : 32;
    a.depth = small ? 1 : 2;
    const unsigned u = static_cast<unsigned>(a.wave);
    const cudaError_t e = t.bn == 256   ? (pair ? launch_product<256, true>(ma, mb, a, u, err, s)
                                                : launch_product<256, false>(ma, mb, a, u, err, s))
                          : t.bn == 128 ? (pair ? launch_product<128, true>(ma, mb, a, u, err, s)
                                                : launch_product<128, false>(ma, mb, a, u, err, s))
                                        : (pair ? launch_product<64, true>(ma, mb, a, u, err, s)
                                                : launch_product<64, false>(ma, mb, a, u, err, s));
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t rns_residual(const RnsOperand& Ls, const double* diag, const RnsOperand& Xs, const double* X, int64_t ldx,
                         const double* B, int64_t ldb, double* R, int64_t ldr, int planes, const RnsScratch& sc,
                         int* err, cudaStream_t s) {
  if (planes < 5 || planes > 8 || Ls.kc != Xs.kc || Ls.K != Xs.K || Ls.rows != Ls.K || !Ls.tri)
    return cudaErrorInvalidValue;
  const int64_t n = Ls.rows, k = Xs.rows;
  cudaError_t e = cudaSuccess;
  // chunk by chunk of K: the rows from the chunk's first on (the first chunk
  // starts R from B and the diagonal term)
  for (int64_t k0 = 0; k0 < n && e == cudaSuccess; k0 += Ls.kc) {
    RnsProduct p;
    p.A = rns_chunk(Ls, k0 / Ls.kc);
    p.B = Xs;
    p.b_k0 = k0;
    p.M = n - k0;
    p.N = k;
    p.K = std::min<int64_t>(Ls.kc, n - k0);
    p.cls = rns_class(planes);
    p.lower = true;
    p.mode = k0 == 0 ? kRnsResidual : kRnsUpdate;
    p.Y = R + k0;
    p.ldy = ldr;
    p.S = k0 == 0 ? B : R + k0;
    p.lds = k0 == 0 ? ldb : ldr;
    p.dg = diag;
    p.X = X;
    p.ldx = ldx;
    e = rns_product(p, sc, err, s);
  }
  return e;
}

}  // namespace trsm

namespace {
__global__ void copy_diag_kernel(const double* __restrict__ L, int64_t ldl, int64_t n, double* __restrict__ d) {
  const int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  if (i < n) d[i] = L[i * ldl + i];
}
}  // namespace

extern "C" int trsm_residual_sliced(const double* L_dev, int64_t n, int64_t ldl, const double* X_dev, int64_t k,
                                    int64_t ldx, const double* B_dev, int64_t ldb, double* R_dev, int64_t ldr,
                                    int planes, int* err_dev, void* stream) {
  if (!L_dev || !X_dev || !B_dev || !R_dev || !err_dev || n < 1 || k < 1 || ldl < n || ldx < n || ldb < n || ldr < n ||
      planes < 5 || planes > 8)
    return -1;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const size_t lb = trsm::rns_operand_bytes(n, n, trsm::kChunk, true);
  const size_t xb = trsm::rns_operand_bytes(k, n);
  const size_t tb = (sizeof(double) * static_cast<size_t>(n) * n + 255) / 256 * 256;
  const size_t db = (sizeof(double) * static_cast<size_t>(n) + 255) / 256 * 256;
  const size_t sb = trsm::rns_scratch_bytes(n, k);
  unsigned char* buf = nullptr;
  cudaError_t e = trsm::ws_alloc(reinterpret_cast<void**>(&buf), lb + xb + tb + db + sb, s);
  if (e != cudaSuccess) return -3;
  const trsm::RnsOperand Ls = trsm::rns_operand_view(buf, n, n, trsm::kChunk, true);
  trsm::RnsOperand Xs = trsm::rns_operand_view(buf + lb, k, n);
  double* diag = reinterpret_cast<double*>(buf + lb + xb + tb);
  const trsm::RnsScratch sc = trsm::rns_scratch_view(buf + lb + xb + tb + db, n, k);
  Xs.zmax = sc.zmax;
  e = trsm::rns_scratch_clear(sc, s);
  if (e == cudaSuccess) e = trsm::rns_lower_rows(L_dev, ldl, n, Ls, reinterpret_cast<double*>(buf + lb + xb), s);
  if (e == cudaSuccess) {
    copy_diag_kernel<<<static_cast<unsigned>((n + 255) / 256), 256, 0, s>>>(L_dev, ldl, n, diag);
    trsm::count_launch();
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = trsm::rns_rows(X_dev, ldx, n, Xs, trsm::rns_class(planes), s);
  if (e == cudaSuccess)
    e = trsm::rns_residual(Ls, diag, Xs, X_dev, ldx, B_dev, ldb, R_dev, ldr, planes, sc, err_dev, s);
  trsm::ws_free(buf, s);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return -4;
  }
  return 0;
}
