// Binary64 product [A; acs] [B, bcs] on the tensor cores, by integer arithmetic
// modulo small numbers (the scheme of Ozaki, Uchino and Imamura, "Ozaki scheme II: a
// GEMM-oriented emulation of floating-point matrix multiplication using an integer
// modular technique", 2025, with bf16 residues instead of 8-bit integers).
//
// GB300's FP64 pipe issues 2 DFMA per clock and SM (1.2 TFLOP/s on the whole
// chip); its tensor cores multiply bf16 at 1900 TFLOP/s.  Row i of A (column
// j of B) is scaled by the power of two above its largest element and rounded to
// an integer a' of b = 58 or 59 bits.  The exact integer C' = sum_l a'_il b'_lj is
// below half of P, the product of 17 coprime moduli up to 256 (133 bits), so it
// follows from its residues.  A residue is at most 128 in magnitude: exact in bf16,
// and 1024 products of two add up to at most 2^24, exact in the tensor cores'
// binary32 accumulators.  One bf16 product per modulus gives C' mod p (the epilogue
// reduces each accumulator modulo p), the Chinese remainder theorem C' itself, and
// C_ij = 2^(eA_i + eB_j - 2 b) C' is rounded to nearest once: all in integer and
// exact binary32 arithmetic.
//
// Accuracy.  What is lost is the rounding of a and b to b bits below their row's and
// column's scale: each term errs by at most 2^-b in units of 2^(eA_i + eB_j), so an
// element by at most k 2^-b.  With M_ij = sum_l |a_il b_lj| in the same units, an element
// is taken only where M_ij >= 1.52 2^(53 - b) sqrt(k): its error is then at most 0.66
// sqrt(k) u M_ij (u = 2^-53), plus one rounding of the result (of each panel's, when K
// takes several).  That is the bound that holds for every operand; it is no statement
// about a chain of multiply-adds on the same data.  On generic data (independent
// roundings, partial sums that grow) the errors are far below the chain's, whose
// roundings come to about 0.38 u sqrt(k / 2) times the rms of the terms' sum, at least
// 0.27 u M_ij; but where neighbours nearly cancel the chain's partial sums stay small and
// it can be the closer one (pairs that agree to 1e-3 in a row whose largest element meets
// a zero: errors of 4 to 7 times the chain's at k = 1024 to 12000, 0.1 u M_ij).  M is one
// more product (plane 17: the magnitudes as bf16, rounded towards zero), and every tile
// computes it first: each element is checked, so rows of mixed scales, graded operands
// whose large rows meet small columns, and sparse operands keep that bound.  Elements of
// rows and columns that are integers as they are need no check.  The 32 x 32 chunks that
// hold an element below the line, NaN or infinite operands or exponents outside [-440,
// 500] are left to the DFMA kernel (k_gemm_f64_bad).
//
// Those chunks cost both products: where all of them are left out (columns of A and rows
// of B graded over 16 decades, or rows below 2^-440) 128^3 takes 164 us (the FP64 pipe
// alone 135), 512^3 570 (527), 2048^3 14.63 ms (14.29), 4096^3 116.8 (110.0).
//
// The tensor cores bound it: 18 products of 2 m n k bf16 flops each.  (Exact digits
// in radix 256 instead of residues take 29 to 37 products for the same accuracy,
// a level sum in 32-bit integers per thread and a copy of every level: 8192^3 21.6
// ms, 4096^3 2.93, 2048^3 0.38 .. 0.47, 512^3 59 us.)  128 x (64 bpt)-tiles on one
// CTA or 256 x 256 tiles on a pair, one CTA per SM: warps 0 / 10 copy A / B by TMA
// into a shared-memory ring, warp 1 issues tcgen05.mma into two alternating TMEM
// accumulators, warps 2-9 reduce each accumulator modulo p and keep the residues of
// a finished modulus, one byte each, in a per-CTA scratch (coalesced, mostly L2).
//
// Measured, product kernels alone: 8192^3 on a 16 x 16 grid 949 ms on the FP64 pipe,
// 11.6 .. 15 here (with the clock); 4096^3 on an 8 x 8 grid 130 -> 1.98; 2048^3 16.3 ->
// 0.28; 1000 x 1501 x 777 2.36 -> 0.088; 512^3 0.53 -> 0.026.  Relative Frobenius error
// against the exact product, N(0,1): 4.5e-17 (DFMA 7.7e-16) at k = 512, 4.7e-17 (2.0e-15)
// at k = 4096, 7.0e-17 (4.9e-15) at k = 20000 in two panels of K.
#include <cuda.h>

#include <stdlib.h>

#include <algorithm>

#include "gemm_f64.cuh"
#include "internal.cuh"
#include "tc_ptx.cuh"

namespace abft {
namespace {

constexpr int BM = 128, BK = 64;
constexpr int kModuli = 17, kMagPlane = kModuli, kPlanes64 = kModuli + 1;
constexpr int kGroupSteps = 16;   // k-steps per accumulator: 1024 products of at most 2^14
constexpr int kMaxPanel = 16320;  // K of a pass: 255 k-steps, 16 partial residues per thread
constexpr int kMaxBits = 59;      // of an operand's integers (four 15-bit limbs hold them)
constexpr int kEpiWarps = 8;
constexpr int kWarpProdB = 2 + kEpiWarps;
constexpr int kThreads = 32 * (kWarpProdB + 1);
constexpr uint32_t kABytes = BM * BK * 2, kBoxBytes = 64 * BK * 2;
constexpr int kMaxStages = 8;
constexpr int kMinExp = -440, kMaxExp = 500;
constexpr int kCut = 1, kRefused = 2;  // operand lines that were rounded / cannot be held
constexpr int kMinK = 48;         // shorter K loops run on the FP64 pipe (plan_f64_tc)
constexpr double kMiB = 1048576.0;
constexpr double kPlaneBudget = 12288 * kMiB;
constexpr double kDeviceBytes = 284208 * kMiB;  // of a GB300's memory
constexpr int kSms = 152;  // persistent CTAs the workspace is laid out for

// Tile kinds.  One CTA: 128 rows x bpt 64-column boxes.  CTA pair (bpt = 4): 256
// x 256, one cta_group::2 MMA per K step reads 128 rows of A and 128 columns of B
// from each CTA's shared memory.
constexpr int cta_boxes(int bpt, bool pair) { return pair ? bpt / 2 : bpt; }
constexpr int stages(int boxes) { return boxes == 4 ? 4 : (boxes == 2 ? 6 : 8); }
constexpr size_t smem_bytes(int boxes) {
  return 1024 + (size_t)stages(boxes) * (kABytes + boxes * kBoxBytes) + 320;
}
static_assert(smem_bytes(4) <= 232448 && smem_bytes(2) <= 232448 && smem_bytes(1) <= 232448,
              "shared memory per CTA");

// ------------------------------------------------------------------ residues

// The moduli (pairwise coprime) and what the device needs of them.  Residues are
// signed and smallest in magnitude.  Signed limbs: x = sum_i limb_i 2^(32 i), each in
// [-2^31, 2^31).
struct Moduli {
  int p[kModuli] = {256, 255, 253, 251, 247, 241, 239, 233, 229, 227, 223, 217, 211, 199, 197,
                    193, 191};
  float pf[kModuli] = {}, inv[kModuli] = {};
  // weights of the 15-bit limbs of an integer in its residue, for B; for A times
  // (P / p)^-1 mod p, so the product's residue x_t has C' = sum_t x_t P / p_t mod P
  float ca[kModuli][4] = {}, cb[kModuli][4] = {};
  // reconstruction in groups of three moduli (the last of two): y = sum x_t g_t, the
  // product of the group's other moduli; C' = sum_j y_j P / (group's product) - n P
  int g[kModuli] = {};
  int limb[6][4] = {};  // P / (group's product)
  int frac[6] = {};     // 2^40 / (group's product)
  int P[5] = {};
};
constexpr double kLog2P = 132.95;  // P = 2^132.953

constexpr int centred(int64_t x, int p) {
  int64_t r = x % p;
  if (r < 0) r += p;
  return (int)(2 * r > p ? r - p : r);
}

constexpr Moduli make_moduli() {
  Moduli M;
  for (int t = 0; t < kModuli; ++t) {
    const int p = M.p[t];
    M.pf[t] = (float)p;
    M.inv[t] = 1.0f / (float)p;
    int64_t q = 1;  // P / p mod p
    for (int u = 0; u < kModuli; ++u)
      if (u != t) q = q * M.p[u] % p;
    int64_t w = 1;
    while (q * w % p != 1) ++w;
    int64_t c = 1;
    for (int i = 0; i < 4; ++i) {
      M.cb[t][i] = (float)centred(c, p);
      M.ca[t][i] = (float)centred(c * w, p);
      c = c * 32768 % p;
    }
    const int j0 = t / 3 * 3;
    M.g[t] = 1;
    for (int u = j0; u < j0 + 3 && u < kModuli; ++u)
      if (u != t) M.g[t] *= M.p[u];
  }
  for (int j = 0; j <= 6; ++j) {  // j = 6: P itself
    uint64_t v[6] = {1, 0, 0, 0, 0, 0};  // 32-bit limbs
    int64_t group = 1;
    for (int u = 0; u < kModuli; ++u) {
      if (u / 3 == j) {
        group *= M.p[u];
        continue;
      }
      uint64_t carry = 0;
      for (int i = 0; i < 6; ++i) {
        const uint64_t x = v[i] * (uint64_t)M.p[u] + carry;
        v[i] = x & 0xffffffffull;
        carry = x >> 32;
      }
    }
    int64_t carry = 0;
    for (int i = 0; i < 5; ++i) {
      int64_t x = (int64_t)v[i] + carry;
      carry = 0;
      if (x >= 2147483648ll) {
        x -= 4294967296ll;
        carry = 1;
      }
      if (j == 6)
        M.P[i] = (int)x;
      else if (i < 4)
        M.limb[j][i] = (int)x;
    }
    if (j < 6) M.frac[j] = (int)(((1ll << 40) + group / 2) / group);
  }
  return M;
}

// Compile-time: as instruction operands they cost nothing, where a constant bank's
// cold misses cost a small product 10 us.
constexpr Moduli kM = make_moduli();

// {p, 1 / p} where the modulus is a loop variable.
struct ModulusTable {
  float2 m[kModuli];
};
constexpr ModulusTable make_table() {
  ModulusTable T{};
  for (int t = 0; t < kModuli; ++t) {
    T.m[t].x = kM.pf[t];
    T.m[t].y = kM.inv[t];
  }
  return T;
}
__constant__ ModulusTable kModulus = make_table();

// x 2^(bits - e) rounded to the nearest integer, ties to even (|x| < 2^e, e = efield -
// 1022 with efield the biased exponent of the line's largest element; bits <= 59).
// Values whose last bit is the half (a line of elements 2^6 .. 2^7 below its largest
// one) would all err the same way if ties left zero: the error of a sum of k of them
// grew like k, where it grows like sqrt(k) now.
__device__ __forceinline__ int64_t scaled(double x, int efield, int bits, bool& cut) {
  const uint64_t b = (uint64_t)__double_as_longlong(x);
  const int E = (int)(b >> 52) & 0x7ff;
  const uint64_t m =
      ((b & 0xfffffffffffffull) | (E ? 0x10000000000000ull : 0ull)) << 10;  // below 2^63
  const int r = efield - max(E, 1) + (63 - bits);
  uint64_t v = 0;
  if (r < 64) {
    const uint64_t up = m + ((1ull << r) >> 1);
    v = up >> r;
    const uint64_t t = v << r;
    const bool c = t != m;
    cut |= c;
    v &= ~(uint64_t)(c & (t == up));  // a half, rounded up: to the even one
  } else {
    cut |= m != 0;
  }
  return (int64_t)(b >> 63 ? 0ull - v : v);
}

// |x| 2^-e as bf16, rounded towards zero (nonzero values at least 2^-60).
__device__ __forceinline__ uint32_t magnitude(double x, int efield) {
  const uint32_t hi = (uint32_t)__double2hiint(x) & 0x7fffffffu;
  if ((hi | (uint32_t)__double2loint(x)) == 0) return 0;
  const int ex = 126 - (efield - (int)(hi >> 20));  // bf16 exponent field
  return ex < 67 ? 67u << 7 : ((uint32_t)ex << 7) | ((hi >> 13) & 0x7fu);
}

constexpr float kRound = 12582912.0f;  // 1.5 2^23: x + kRound - kRound rounds x, |x| <= 2^22

// The smallest residue of the integer s (|s| <= 2^24) modulo p.
__device__ __forceinline__ float residue(float s, float p, float inv) {
  return fmaf(-(fmaf(s, inv, kRound) - kRound), p, s);
}

// The residues modulo p_t and all later moduli of four integers, from their limbs.
template <bool kA, int t>
__device__ __forceinline__ void residues4(const float (&l)[4][4], uint16_t* o, int64_t plane) {
  constexpr float c0 = kA ? kM.ca[t][0] : kM.cb[t][0], c1 = kA ? kM.ca[t][1] : kM.cb[t][1],
                  c2 = kA ? kM.ca[t][2] : kM.cb[t][2], c3 = kA ? kM.ca[t][3] : kM.cb[t][3],
                  p = kM.pf[t], inv = kM.inv[t];
  float r[4];
#pragma unroll
  for (int q = 0; q < 4; ++q)  // the sum is at most 4 2^14 2^7: exact
    r[q] = residue(fmaf(l[q][3], c3, fmaf(l[q][2], c2, fmaf(l[q][1], c1, l[q][0] * c0))), p, inv);
  // bf16 holds a residue exactly: the upper halves of the binary32 words
  *reinterpret_cast<uint2*>(o) =
      make_uint2(__byte_perm(__float_as_uint(r[0]), __float_as_uint(r[1]), 0x7632u),
                 __byte_perm(__float_as_uint(r[2]), __float_as_uint(r[3]), 0x7632u));
  if constexpr (t + 1 < kModuli) residues4<kA, t + 1>(l, o + plane, plane);
}

// Four consecutive elements of every plane, at o (planes `plane` elements apart),
// from four values with scales ef (0: a line that cannot be held, whose residues are
// zero and whose magnitudes are NaN); cut: whether any bits were cut off.
template <bool kA>
__device__ __forceinline__ void slice4(const double (&x)[4], const int (&ef)[4], int bits,
                                       uint16_t* o, int64_t plane, bool (&cut)[4]) {
  float l[4][4];  // 15-bit signed limbs of the integers
  uint32_t mag[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int f = ef[q] ? ef[q] : 1022;
    const double v = ef[q] ? x[q] : 0.0;
    // with 2^14 added in every limb but the top one, the limbs are bit fields
    const int64_t u = scaled(v, f, bits, cut[q]) + 0x100020004000ll;
    mag[q] = ef[q] ? magnitude(v, f) : 0x7fc0u;
#pragma unroll
    for (int i = 0; i < 3; ++i)  // 2^23 + field as binary32 bits, minus 2^23 + 2^14
      l[q][i] = __uint_as_float(0x4B000000u | ((uint32_t)(u >> (15 * i)) & 0x7fffu)) - 8404992.0f;
    l[q][3] = __uint_as_float(0x4B000000u | (uint32_t)((int)(u >> 45) + 32768)) - 8421376.0f;
  }
  residues4<kA, 0>(l, o, plane);
  *reinterpret_cast<uint2*>(o + kMagPlane * plane) =
      make_uint2(mag[0] | (mag[1] << 16), mag[2] | (mag[3] << 16));
}

// Four consecutive elements, zeros from element nv on.
__device__ __forceinline__ void load4(const double* p, int64_t nv, double (&x)[4]) {
  if (nv >= 4 && (reinterpret_cast<uintptr_t>(p) & 15) == 0) {
    const double2 a = *reinterpret_cast<const double2*>(p);
    const double2 b = *reinterpret_cast<const double2*>(p + 2);
    x[0] = a.x; x[1] = a.y; x[2] = b.x; x[3] = b.y;
  } else {
#pragma unroll
    for (int q = 0; q < 4; ++q) x[q] = q < nv ? p[q] : 0.0;
  }
}

// A value's key for the maximum: its high word (whose upper bits are the
// exponent), with the last bit set when any lower bit is, so that 0 means zero.
__device__ __forceinline__ uint32_t max_key(double x) {
  return ((uint32_t)__double2hiint(x) & 0x7fffffffu) | (__double2loint(x) != 0 ? 1u : 0u);
}

// The biased exponent that scales a line with that maximal key: 0 marks a line
// that the integers cannot hold (NaN, infinite, exponent outside the range).
__device__ __forceinline__ int line_field(uint32_t key) {
  const int E = (int)(key >> 20);
  if (key == 0) return 1022;
  return (E - 1022 < kMinExp || E - 1022 > kMaxExp) ? 0 : E;
}

struct SliceArgs {
  F64Args g;          // operands of this panel
  int64_t kpad;       // panel length rounded up to 64
  int bits;           // of the integers
  uint16_t* pa;       // planes of [A; acs]: [plane][rows_a][kpad]
  uint16_t* pb;       // planes of [B, bcs]: [plane][kpad][cols_b]
  int2* a_row;        // {exponent, kCut / kRefused} per row / column
  int2* b_col;
  uint32_t* cmax;     // [ceil(kpad / 256)][cols_b] maximal keys of 256 rows of B
  int* hdr;           // {status, any bad tile, arrivals of keep_step}
  int64_t rows_a, cols_b, row_cs, col_cs;
  int tpr;            // threads per row of A in the maximum pass
  int rows;           // rows of a slicing CTA
  int64_t n0, n1, n2; // CTAs: A or B data, then their checksums (see the kernels)
};

constexpr int kSliceThreads = 256;
constexpr int kMaxRows = 256;     // rows of B per partial maximum
constexpr int kSliceCols = 256;   // columns and rows of a slicing CTA
constexpr int kSliceRows = 16;    // 4 where 16 would leave SMs idle

// The maximal keys: rows of [A; acs] (tpr threads per row), columns of [B, bcs]
// (32 columns x 256 rows per CTA).  Two passes over the operands in two launches
// (here and k_f64_slice) instead of one CTA that walks a strip of columns twice:
// 512^3 31 -> 21 us, 8192^3 1.60 -> 0.82 ms with nine planes of radix-256 digits.  The
// 18 planes are 36 bytes per element: 1.09 ms at 8192^3 for 6.3 GB, 0.85 of the copy
// rate.
__device__ __forceinline__ void max_rows(const SliceArgs& a, const double* src, int64_t ld,
                                         int64_t rows, int64_t row_out, int64_t blk,
                                         uint32_t* sh) {
  const int tpr = a.tpr, q = threadIdx.x & (tpr - 1), rib = threadIdx.x / tpr;
  const int64_t r = blk * (kSliceThreads / tpr) + rib;
  const double* p = src + (r < rows ? r : 0) * ld;
  const int64_t k = r < rows ? a.g.k : 0;
  uint32_t key = 0;
#pragma unroll 4
  for (int64_t l = 4 * q; l < k; l += 4 * tpr) {
    double x[4];
    load4(p + l, k - l, x);
#pragma unroll
    for (int e = 0; e < 4; ++e) key = max(key, max_key(x[e]));
  }
  key = __reduce_max_sync(0xffffffffu, key);
  const int warp = threadIdx.x >> 5, wpr = tpr / 32;
  if ((threadIdx.x & 31) == 0) sh[warp] = key;
  __syncthreads();
  if (q == 0 && r < rows) {
    for (int w = 1; w < wpr; ++w) key = max(key, sh[warp + w]);
    const int f = line_field(key);
    a.a_row[row_out + r] = make_int2(f ? f - 1022 : kMinExp - 1, 0);
  }
}

__device__ __forceinline__ void max_cols(const SliceArgs& a, const double* src, int64_t ld,
                                         int64_t cols, int64_t col_out, int64_t blk,
                                         uint32_t* sh) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t ncj = cdiv(cols, 32), c = blk / ncj, j = blk % ncj * 32 + lane;
  const int64_t l0 = c * kMaxRows + warp * 32, l1 = min(l0 + 32, a.g.k);
  uint32_t key = 0;
  if (j < cols) {
    const double* p = src + l0 * ld + j;
#pragma unroll 8
    for (int64_t l = l0; l < l1; ++l, p += ld) key = max(key, max_key(*p));
  }
  sh[warp * 32 + lane] = key;
  __syncthreads();
  if (warp == 0 && j < cols) {
#pragma unroll
    for (int w = 1; w < kSliceThreads / 32; ++w) key = max(key, sh[w * 32 + lane]);
    a.cmax[c * a.cols_b + col_out + j] = key;
    if (c == 0) a.b_col[col_out + j] = make_int2(0, 0);
  }
}

__global__ void __launch_bounds__(kSliceThreads) k_f64_max(const SliceArgs a) {
  __shared__ uint32_t sh[kSliceThreads];
  if (blockIdx.x == 0 && threadIdx.x < 3 && (threadIdx.x > 0 || !a.g.accumulate))
    a.hdr[threadIdx.x] = 0;  // the status word covers every panel
  int64_t b = blockIdx.x;
  if (b < a.n0) return max_cols(a, a.g.B, a.g.ldb, a.g.n, 0, b, sh);
  b -= a.n0;
  if (b < a.n1) return max_cols(a, a.g.bcs, a.g.ldbcs, a.g.Cc, a.col_cs, b, sh);
  b -= a.n1;
  if (b < a.n2) return max_rows(a, a.g.A, a.g.lda, a.g.m, 0, b, sh);
  max_rows(a, a.g.acs, a.g.ldacs, a.g.R, a.row_cs, b - a.n2, sh);
}

// The residues of a.rows rows x 256 columns of A (one scale per row) or B (one per
// column): a thread takes four columns of every fourth row.
template <bool kRowsScaled>
__device__ __forceinline__ void slice_tile(const SliceArgs& a, const double* src, int64_t ld,
                                           int64_t rows, int64_t cols, int64_t prow,
                                           int64_t pcol, int64_t blk, int* sef) {
  const int tx = threadIdx.x & 63, ty = threadIdx.x >> 6, lane = threadIdx.x & 31;
  const int64_t pw = kRowsScaled ? a.kpad : cdiv(cols, 64) * 64;  // padded columns
  const int64_t ph = kRowsScaled ? rows : a.kpad;                 // padded rows
  const int64_t nbx = cdiv(pw, kSliceCols);
  const int64_t r0 = blk / nbx * a.rows, c0 = blk % nbx * kSliceCols + 4 * tx;
  const int64_t ldp = kRowsScaled ? a.kpad : a.cols_b;
  const int64_t plane = (kRowsScaled ? a.rows_a : a.kpad) * ldp;
  uint16_t* const out = kRowsScaled ? a.pa : a.pb;
  if constexpr (!kRowsScaled) {  // the columns' scales from their partial maxima
    const int64_t j = blk % nbx * kSliceCols + threadIdx.x;
    uint32_t key = 0;
    if (j < cols)
      for (int64_t c = 0; c < cdiv(a.g.k, kMaxRows); ++c)
        key = max(key, a.cmax[c * a.cols_b + pcol + j]);
    const int f = line_field(key);
    sef[threadIdx.x] = f;
    if (r0 == 0 && j < cols) a.b_col[pcol + j].x = f ? f - 1022 : 0;
    __syncthreads();
  }
  int ef[4];
  bool cut[4] = {false, false, false, false};
  if constexpr (!kRowsScaled) {
#pragma unroll
    for (int q = 0; q < 4; ++q) ef[q] = sef[4 * tx + q];
  }
  const bool in = c0 < pw;
#pragma unroll 2
  for (int i = 0; i < a.rows / 4; ++i) {
    const int64_t r = r0 + ty + 4 * i;
    if (r >= ph) break;  // the whole warp: a row belongs to one
    double x[4] = {0.0, 0.0, 0.0, 0.0};
    if (in && r < rows) load4(src + r * ld + c0, cols - c0, x);
    if constexpr (kRowsScaled) {
      const int e = a.a_row[prow + r].x;
      const int f = e < kMinExp ? 0 : e + 1022;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        ef[q] = f;
        cut[q] = false;
      }
    }
    if (in)
      slice4<kRowsScaled>(x, ef, a.bits, out + (prow + r) * ldp + pcol + c0, plane, cut);
    if constexpr (kRowsScaled) {
      const bool c = __any_sync(0xffffffffu, cut[0] | cut[1] | cut[2] | cut[3]);
      const int z = ef[0] == 0 ? kRefused : (c ? kCut : 0);
      if (lane == 0 && a.a_row[prow + r].y < z) atomicMax(&a.a_row[prow + r].y, z);
    }
  }
  if constexpr (!kRowsScaled) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      if (c0 + q >= cols) break;
      const int z = ef[q] == 0 ? kRefused : (cut[q] ? kCut : 0);
      int2* const at = a.b_col + pcol + c0 + q;
      if (at->y < z) atomicMax(&at->y, z);
    }
  }
}

__global__ void __launch_bounds__(kSliceThreads) k_f64_slice(const SliceArgs a) {
  __shared__ int sef[kSliceCols];
  int64_t b = blockIdx.x;
  if (b < a.n0) return slice_tile<false>(a, a.g.B, a.g.ldb, a.g.k, a.g.n, 0, 0, b, sef);
  b -= a.n0;
  if (b < a.n1)
    return slice_tile<false>(a, a.g.bcs, a.g.ldbcs, a.g.k, a.g.Cc, 0, a.col_cs, b, sef);
  b -= a.n1;
  if (b < a.n2) return slice_tile<true>(a, a.g.A, a.g.lda, a.g.m, a.g.k, 0, 0, b, sef);
  slice_tile<true>(a, a.g.acs, a.g.ldacs, a.g.R, a.g.k, a.row_cs, 0, b - a.n2, sef);
}

// ------------------------------------------------------------------ product

struct Maps {
  CUtensorMap a;   // (kpad, planes x rows_a): box 64 x 128
  CUtensorMap bw;  // (64, planes x kpad, column boxes): box 64 x 64 x a CTA's boxes
  CUtensorMap b1;  // (cols_b, planes x kpad): box 64 x 64
};

struct ProdArgs {
  F64Args g;
  TileGrid T;
  int nkb, bpt;                  // k-steps of a panel; boxes per tile
  int kpad, rows_a, row_cs, col_cs;
  const int2* a_row;
  const int2* b_col;
  uint8_t* bad;
  int* hdr;                      // {status, any bad tile, arrivals of keep_step}
  uint32_t* scratch;             // per CTA: [modulus][chunk][8][256 epilogue threads], four
                                 // residues of a thread's row each
  int split;                     // CTAs that share a tile's planes
  int bits;                      // of the operands' integers
  float line;                    // the magnitude that an element needs
  uint64_t wait_ns;
  int stall_test;
};

// 16 consecutive fp32 columns of this thread's TMEM lane.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16]) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// Byte u of x as a signed number.
__device__ __forceinline__ int signed_byte(uint32_t x, int u) {
  return (int)(x << (24 - 8 * u)) >> 24;
}

// Group j and all later ones: y_j P / (group's product) added to acc, in limbs, and
// y_j / (group's product) to nf, in 2^-40.
template <int j>
__device__ __forceinline__ void add_groups(const uint32_t (&x)[kModuli], int u,
                                           int64_t (&acc)[4], int64_t& nf) {
  constexpr int g0 = kM.g[3 * j], g1 = kM.g[3 * j + 1],
                g2 = 3 * j + 2 < kModuli ? kM.g[3 * j + 2 < kModuli ? 3 * j + 2 : 0] : 0,
                l0 = kM.limb[j][0], l1 = kM.limb[j][1], l2 = kM.limb[j][2], l3 = kM.limb[j][3],
                f = kM.frac[j];
  int y = signed_byte(x[3 * j], u) * g0 + signed_byte(x[3 * j + 1], u) * g1;
  if constexpr (3 * j + 2 < kModuli) y += signed_byte(x[3 * j + 2], u) * g2;
  acc[0] += (int64_t)y * l0;
  acc[1] += (int64_t)y * l1;
  acc[2] += (int64_t)y * l2;
  acc[3] += (int64_t)y * l3;
  nf += (int64_t)y * f;
  if constexpr (j + 1 < 6) add_groups<j + 1>(x, u, acc, nf);
}

// C' 2^e rounded to the nearest binary64 (ties to even; the result is a normal
// number or zero), with C' from its residues: byte u of x[t].  Integer instructions
// only: y_j of each group of three moduli, n = round(sum_j y_j / (group's product))
// in 40-bit fixed point (within 1e-4 of the exact sum; 2 |C'| < P keeps it away from
// a half by far more), C' = sum_j y_j P / (group's product) - n P in 32-bit limbs.
__device__ __forceinline__ double crt_f64(const uint32_t (&x)[kModuli], int u, int e) {
  int64_t acc[4] = {0, 0, 0, 0}, nf = 0;
  add_groups<0>(x, u, acc, nf);
  const int n = (int)((nf + (1ll << 39)) >> 40);
  constexpr int P0 = kM.P[0], P1 = kM.P[1], P2 = kM.P[2], P3 = kM.P[3], P4 = kM.P[4];
  acc[0] -= (int64_t)n * P0;
  acc[1] -= (int64_t)n * P1;
  acc[2] -= (int64_t)n * P2;
  acc[3] -= (int64_t)n * P3;
  acc[1] += acc[0] >> 32;
  acc[2] += acc[1] >> 32;
  acc[3] += acc[2] >> 32;
  const int top = (int)(acc[3] >> 32) - n * P4;  // the fifth limb
  uint32_t w[5] = {(uint32_t)acc[0], (uint32_t)acc[1], (uint32_t)acc[2], (uint32_t)acc[3],
                   (uint32_t)top};
  const bool neg = top < 0;
  if (neg) {
    uint32_t carry = 1;
#pragma unroll
    for (int i = 0; i < 5; ++i) {
      w[i] = ~w[i] + carry;
      carry = carry & (w[i] == 0 ? 1u : 0u);
    }
  }
  // the leading three words hi, mid, lo (hi: word idx, not zero) and what is below
  int idx = 4;
  uint32_t hi = w[4], mid = w[3], lo = w[2], rest = w[0] | w[1];
#pragma unroll
  for (int i = 1; i >= 0; --i)
    if (hi == 0) {
      hi = mid;
      mid = lo;
      lo = w[i];
      rest = i == 1 ? w[0] : 0u;
      --idx;
    }
  if (hi == 0) {  // below 2^64
    if ((mid | lo) == 0) return 0.0;
    idx = mid ? 1 : 0;
    hi = mid ? mid : lo;
    mid = idx ? lo : 0u;
    lo = 0u;
  }
  const int z = __clz((int)hi);
  const uint64_t t64 =
      ((uint64_t)__funnelshift_l(mid, hi, z) << 32) | __funnelshift_l(lo, mid, z);
  const uint64_t m = t64 >> 11;
  const uint32_t r = (uint32_t)t64 & 0x7ffu;
  const bool below = ((lo << z) | rest) != 0;
  const uint64_t up = (r > 0x400u || (r == 0x400u && (below || (m & 1)))) ? 1 : 0;
  const uint64_t bits = ((uint64_t)(32 * idx + 31 - z + e + 1022) << 52) + m + up;
  return __longlong_as_double((long long)(bits | (neg ? 0x8000000000000000ull : 0ull)));
}

struct TileView64 {
  bool cs_row, cs_col;
  int64_t row0, col0;     // this CTA's first row, the tile's first column, in C / E / F
  int arow, bcol;         // padded row of the A planes, column of the B planes
  int ncols, nmma;        // valid columns; the MMA's N
  int bx, nbox;           // this CTA's first column of the B planes and its boxes
  bool full;              // all boxes of a full tile (one copy)
  int64_t rlim;
};

template <bool kPair>
__device__ __forceinline__ TileView64 view_tile(const ProdArgs& p, int64_t t, int rank) {
  int ty, tx;
  p.T.decode(t, ty, tx);
  TileView64 V;
  V.cs_row = ty >= p.T.tm;
  V.cs_col = tx >= p.T.tn;
  V.row0 = (int64_t)(V.cs_row ? ty - p.T.tm : ty) * (kPair ? 2 * BM : BM) + BM * rank;
  V.col0 = (int64_t)(V.cs_col ? tx - p.T.tn : tx) * 64 * p.bpt;
  V.arow = (int)V.row0 + (V.cs_row ? p.row_cs : 0);
  V.bcol = (int)V.col0 + (V.cs_col ? p.col_cs : 0);
  V.rlim = V.cs_row ? p.g.R : p.g.m;
  V.ncols = (int)min((int64_t)64 * p.bpt, (V.cs_col ? p.g.Cc : p.g.n) - V.col0);
  // a pair's MMA takes half of its N columns from each CTA
  V.nmma = kPair ? (V.ncols + 31) / 32 * 32 : (V.ncols + 15) / 16 * 16;
  V.bx = V.bcol + (kPair ? V.nmma / 2 * rank : 0);
  V.nbox = ((kPair ? V.nmma / 2 : V.ncols) + 63) / 64;
  V.full = kPair ? V.nmma == 64 * p.bpt : V.nbox == p.bpt;
  return V;
}

// tc::keep_step before every kStepPlanes-th plane of a pair's tile.  The pairs of a wave
// share 2048 rows of A and about 2400 columns of B, 73 MB per plane at k = 8192 and 101 MB
// at 11264; left alone they drift planes apart (checksum tiles are narrower) and every one
// reads its panels from DRAM again.  11264^3 on a 22 x 22 grid: 186 to 246 GB read per
// launch -> 61, product in the step 43.8 -> 31.3 ms; 8192^3 encode + product 17.1 -> 14.7;
// 4096^3, where a plane is 37 MB, 2.88 either way.  Before every plane 11264^3 takes 31.3
// ms too and 4096^3 2.89; once per tile gains nothing (the drift is within a tile).
constexpr int kStepPlanes = 3;
constexpr int kStepCalls = (kPlanes64 + kStepPlanes - 1) / kStepPlanes;  // of a tile
// kSplit: the planes of a tile (magnitudes, then the moduli) are dealt to the p.split
// CTAs of a cluster, each takes them like a whole tile, the residues meet in the
// cluster's scratch and every CTA puts a share of the columns together: a small
// product then occupies p.split times as many SMs.
template <bool kPair, bool kSplit>
__global__ void __launch_bounds__(kThreads, 1)
    k_gemm_f64_tc(const __grid_constant__ Maps M, const ProdArgs p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  const int boxes = cta_boxes(p.bpt, kPair);  // this CTA's boxes of a full tile
  const int NS = stages(boxes);
  const uint32_t stage = kABytes + boxes * kBoxBytes;
  constexpr int kWarpsAll = kPair ? 2 * kEpiWarps : kEpiWarps;  // epilogue warps of a tile
  static_assert(!(kPair && kSplit), "pairs do not split");
  const int rank = kPair ? (int)tc::cluster_ctarank() : 0;
  const int part = kSplit ? (int)tc::cluster_ctarank() : 0, nparts = kSplit ? p.split : 1;
  const int plane0 = kPlanes64 * part / nparts, plane1 = kPlanes64 * (part + 1) / nparts;
  const bool issuer = rank == 0;  // its MMA warp issues for both CTAs of a pair
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + NS * stage);
  // full [8], empty [8], tmem full [2], tmem empty [2], drain, residues done
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * kMaxStages + 6);
  volatile int* abort = reinterpret_cast<volatile int*>(tmem_slot + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  auto full = [&](int s) { return tc::smem_addr(&bars[s]); };
  auto empty = [&](int s) { return tc::smem_addr(&bars[kMaxStages + s]); };
  auto tfull = [&](int a) { return tc::smem_addr(&bars[2 * kMaxStages + a]); };
  auto tempty = [&](int a) { return tc::smem_addr(&bars[2 * kMaxStages + 2 + a]); };
  const uint32_t drain = tc::smem_addr(&bars[2 * kMaxStages + 4]);
  const uint32_t done = tc::smem_addr(&bars[2 * kMaxStages + 5]);

  if (threadIdx.x == 0) {
    for (int s = 0; s < NS; ++s) {
      tc::mbar_init(full(s), 2);
      tc::mbar_init(empty(s), 1);
    }
    for (int a = 0; a < 2; ++a) {
      tc::mbar_init(tfull(a), 1);
      tc::mbar_init(tempty(a), kWarpsAll);
    }
    tc::mbar_init(drain, 1);
    tc::mbar_init(done, kEpiWarps * nparts);
    *abort = 0;
    tc::wait_limit_ns() = p.wait_ns;
    tc::fence_barrier_init();
    tc::prefetch_tmap(&M.a);
    tc::prefetch_tmap(&M.bw);
    tc::prefetch_tmap(&M.b1);
  }
  if (warp == 1) {
    if constexpr (kPair) {
      tc::tmem_alloc_pair(tc::smem_addr(tmem_slot), 512);
      tc::tmem_relinquish_pair();
    } else {
      tc::tmem_alloc(tc::smem_addr(tmem_slot), 512);
      tc::tmem_relinquish();
    }
  }
  tc::fence_before_sync();
  if constexpr (kPair || kSplit)
    tc::cluster_sync();
  else
    __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = *tmem_slot;
  const int64_t total = p.T.total();
  constexpr bool kCluster = kPair || kSplit;
  const int64_t tfirst = kCluster ? (int64_t)tc::cluster_id() : (int64_t)blockIdx.x;
  const int64_t tstep = kCluster ? (int64_t)tc::num_clusters() : (int64_t)gridDim.x;
  const int nkb = p.nkb;
  if (warp == 0 || warp == kWarpProdB) {
    if (tc::elect_one()) {
      const bool pA = warp == 0;
      int s = 0;
      uint32_t ph = 0;
      int64_t issued = 0;
      bool ok = true, together = true;
      for (int64_t t = tfirst; t < total && ok && !*abort; t += tstep) {
        if (p.stall_test && t == 0) continue;
        const TileView64 V = view_tile<kPair>(p, t, rank);
        // a pair's bytes (both CTAs') land on the issuer's barrier, which the
        // issuer's producers expect
        const uint32_t tx = (pA ? kABytes : (uint32_t)V.nbox * kBoxBytes) * (kPair ? 2 : 1);
        // a plane of A and of B: the magnitudes, then the residues
        for (int i = plane0; i < plane1 && ok; ++i) {
          const int plane = i == 0 ? kMagPlane : i - 1;
          if (kPair && pA && issuer && i % kStepPlanes == 0) {
            uint32_t* const arr = reinterpret_cast<uint32_t*>(p.hdr) + 2;
            if (!together)
              atomicAdd(arr, 1u);
            else  // a k-step takes about 320 ns
              together = tc::keep_step(arr, (uint32_t)tstep, total, (uint32_t)((t - tfirst) / tstep),
                                   i / kStepPlanes + 1, kStepCalls, 640ull * kStepPlanes * nkb);
          }
          const int arow = plane * p.rows_a + V.arow, brow = plane * p.kpad;
          for (int kb = 0; kb < nkb; ++kb) {
            if (!tc::wait(empty(s), ph ^ 1, abort)) { ok = false; break; }
            const uint32_t sa = tc::smem_addr(smem + s * stage);
            if (issuer) tc::mbar_arrive_expect_tx(full(s), tx);
            const uint32_t fb = kPair ? tc::mapa(full(s), 0) : full(s);
            if (pA) {
              if constexpr (kPair)
                tc::tma_load_2d_pair(sa, &M.a, fb, kb * BK, arow);
              else
                tc::tma_load_2d(sa, &M.a, fb, kb * BK, arow);
            } else if (V.full) {
              if constexpr (kPair)
                tc::tma_load_3d_pair(sa + kABytes, &M.bw, fb, 0, brow + kb * BK, V.bx / 64);
              else
                tc::tma_load_3d(sa + kABytes, &M.bw, fb, 0, brow + kb * BK, V.bx / 64);
            } else {
              for (int b = 0; b < V.nbox; ++b) {
                if constexpr (kPair)
                  tc::tma_load_2d_pair(sa + kABytes + b * kBoxBytes, &M.b1, fb, V.bx + 64 * b,
                                       brow + kb * BK);
                else
                  tc::tma_load_2d(sa + kABytes + b * kBoxBytes, &M.b1, fb, V.bx + 64 * b,
                                  brow + kb * BK);
              }
            }
            ++issued;
            if (++s == NS) { s = 0; ph ^= 1; }
          }
        }
      }
      // no copies left in flight (bounded): a pair's complete on the issuer's
      // barriers, so its CTAs wait until the MMAs have consumed the stages
      for (int q = 0; q < NS && issued > 0; ++q, --issued) {
        if (--s < 0) { s = NS - 1; ph ^= 1; }
        const uint64_t t0 = tc::globaltimer();
        const uint32_t bar = kPair ? empty(s) : full(s);
        while (!tc::mbar_try_wait(bar, ph) && tc::globaltimer() - t0 < tc::wait_limit_ns()) {
        }
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    if (issuer && tc::elect_one()) {
      int s = 0, acc = 0;
      uint32_t ph = 0, aph = 0;
      bool ok = true;
      for (int64_t t = tfirst; t < total && ok && !*abort; t += tstep) {
        const TileView64 V = view_tile<kPair>(p, t, rank);
        const uint32_t idesc = tc::idesc_bf16(kPair ? 2 * BM : BM, V.nmma, 1);
        // nk k-steps in accumulators of g each
        auto level = [&](int nk, int g) {
          for (int k0 = 0; k0 < nk; k0 += g) {
            if (!tc::wait(tempty(acc), aph ^ 1, abort)) return false;
            tc::fence_after_sync();
            const uint32_t d = tmem + acc * 256;
            const int k1 = min(k0 + g, nk);
            for (int kb = k0; kb < k1; ++kb) {
              if (!tc::wait(full(s), ph, abort)) return false;
              tc::fence_after_sync();
              const uint32_t sa = tc::smem_addr(smem + s * stage), sb = sa + kABytes;
              tc::mma4_f16<kPair, 2, 128>(d, tc::sdesc_sw128(sa, 16, 1024),
                                          tc::sdesc_sw128(sb, kBoxBytes, 1024), idesc, kb > k0);
              tc::commit_x<kPair>(empty(s));
              if (++s == NS) { s = 0; ph ^= 1; }
            }
            tc::commit_x<kPair>(tfull(acc));
            if (++acc == 2) { acc = 0; aph ^= 1; }
          }
          return true;
        };
        for (int i = plane0; i < plane1 && ok; ++i)
          ok = level(nkb, i == 0 ? nkb : kGroupSteps);  // magnitudes: one accumulator
      }
      // every MMA has completed before TMEM is freed
      if constexpr (kPair)
        tc::commit_pair(drain, 1);
      else
        tc::commit(drain);
      const uint64_t t0 = tc::globaltimer();
      while (!tc::mbar_try_wait(drain, 0) && tc::globaltimer() - t0 < tc::wait_limit_ns()) {
      }
    }
    __syncwarp();
  } else {
    // epilogue: TMEM lane quarter q = warp % 4, column half (warp - 2) / 4
    const int q = warp & 3, half = (warp - 2) >> 2, ew = warp - 2, et = ew * 32 + lane;
    const int nch = p.bpt, c_lo = half * 32 * nch;  // 32-column chunks per warp
    // a cluster's scratch alternates between two slots (one while others still read the
    // other)
    const int64_t slot = (int64_t)kModuli * nch * 8 * 256;
    uint32_t* scr = p.scratch + (kSplit ? 2 * tfirst : (int64_t)blockIdx.x) * slot + et;
    uint32_t par = 0;
    int acc = 0;
    uint32_t aph = 0;
    bool ok = true;
    const uint32_t lanes = (uint32_t)(q * 32) << 16;
    // the same answer in every lane, and the warp converged after it
    auto wait_all = [&](uint32_t bar, uint32_t ph) {
      return __all_sync(0xffffffffu, tc::wait(bar, ph, abort)) != 0;
    };
    auto release = [&]() {
      tc::fence_before_sync();
      __syncwarp();
      if (lane == 0) {
        if constexpr (kPair)
          tc::mbar_arrive_cluster(tc::mapa(tempty(acc), 0));
        else
          tc::mbar_arrive(tempty(acc));
      }
      if (++acc == 2) { acc = 0; aph ^= 1; }
    };
    for (int64_t t = tfirst; t < total && ok; t += tstep) {
      const TileView64 V = view_tile<kPair>(p, t, rank);
      const int64_t row = V.row0 + 32 * q + lane;
      const bool rv = row < V.rlim;
      const int2 ri = rv ? p.a_row[V.arow + 32 * q + lane] : make_int2(0, 0);
      const int c_hi = min(c_lo + 32 * nch, V.ncols);  // this warp's valid columns
      // ---- magnitudes: the chunks with an element below the line are left out
      uint8_t* const bad =
          p.bad + (t * (kPair ? 8 : 4) + 4 * rank + q) * (2 * p.bpt) + half * nch;
      uint32_t leave = 0;  // bit ci: chunk ci
      if (plane0 == 0) {
        if (!wait_all(tfull(acc), aph)) { ok = false; break; }
        tc::fence_after_sync();
        const bool cut_rows = __any_sync(0xffffffffu, ri.y != 0);
        for (int ci = 0; ci < nch; ++ci) {
          const int c = c_lo + 32 * ci;
          if (c >= c_hi) break;
          const bool cut = cut_rows | __any_sync(0xffffffffu, c + lane < c_hi &&
                                                                  p.b_col[V.bcol + c + lane].y != 0);
          bool low = false;
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            float v[16];
            tmem_ld16(tmem + lanes + acc * 256 + c + 16 * h, v);
#pragma unroll
            for (int u = 0; u < 16; ++u)  // NaN is below the line
              low |= c + 16 * h + u < c_hi && v[u] != 0.0f && !(v[u] >= p.line);
          }
          // zero: every term is zero; nothing cut: the integers are exact
          if (__any_sync(0xffffffffu, low && rv) && cut) leave |= 1u << ci;
        }
        release();
        if (lane < nch) bad[lane] = (uint8_t)((leave >> lane) & 1);
        if (leave && lane == 0) atomicExch(&p.hdr[1], 1);
      }
      // ---- residues
      for (int t = max(plane0, 1) - 1; t < plane1 - 1; ++t) {
        const float pm = kModulus.m[t].x, inv = kModulus.m[t].y;
        float sum[4][32];
#pragma unroll
        for (int ci = 0; ci < 4; ++ci)
#pragma unroll
          for (int u = 0; u < 32; ++u) sum[ci][u] = 0.0f;
        for (int k0 = 0; k0 < nkb; k0 += kGroupSteps) {
          if (!wait_all(tfull(acc), aph)) { ok = false; break; }
          tc::fence_after_sync();
          const uint32_t base = tmem + lanes + acc * 256 + c_lo;
#pragma unroll
          for (int ci = 0; ci < 4; ++ci) {
            if (ci < nch && c_lo + 32 * ci < c_hi) {
#pragma unroll
              for (int h = 0; h < 2; ++h) {
                float v[16];
                tmem_ld16(base + 32 * ci + 16 * h, v);
#pragma unroll
                for (int u = 0; u < 16; ++u) sum[ci][16 * h + u] += residue(v[u], pm, inv);
              }
            }
          }
          release();
        }
        if (!ok) break;
#pragma unroll
        for (int ci = 0; ci < 4; ++ci)
          if (ci < nch && c_lo + 32 * ci < c_hi) {
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              uint32_t r[4];  // the residue is the low byte
#pragma unroll
              for (int u = 0; u < 4; ++u)
                r[u] = __float_as_uint(residue(sum[ci][4 * j + u], pm, inv) + kRound);
              scr[(int64_t)((t * nch + ci) * 8 + j) * 256] = __byte_perm(
                  __byte_perm(r[0], r[1], 0x0040u), __byte_perm(r[2], r[3], 0x0040u), 0x5410u);
            }
          }
      }
      if (!ok) break;
      if constexpr (kSplit) {  // every CTA's residues and the left-out chunks are written
        __syncwarp();
        if (lane == 0) {
          __threadfence();
          for (int r = 0; r < nparts; ++r) tc::mbar_arrive_cluster(tc::mapa(done, r));
        }
        if (!__all_sync(0xffffffffu, tc::wait_cluster(done, par, abort))) { ok = false; break; }
        leave = __ballot_sync(0xffffffffu, lane < nch && __ldcg(&bad[lane]) != 0);
      }
      // ---- the residues together, rounded once; the next four columns' residues are
      // in flight while these are put together
      double* const dst = (V.cs_row ? p.g.E : (V.cs_col ? p.g.F : p.g.C)) +
                          row * (V.cs_row ? p.g.lde : (V.cs_col ? p.g.ldf : p.g.ldc)) + V.col0;
      const int ncj0 = (min(c_hi, c_lo + 32 * nch) - c_lo + 3) / 4;  // groups of four columns
      const int first = ncj0 * part / nparts, ncj = ncj0 * (part + 1) / nparts;
      uint32_t x[kModuli], y[kModuli];
      auto fetch = [&](int cj) {
#pragma unroll
        for (int t = 0; t < kModuli; ++t) y[t] = __ldcg(&scr[(int64_t)(t * nch * 8 + cj) * 256]);
      };
      if (first < ncj) fetch(first);
#pragma unroll 1
      for (int cj = first; cj < ncj; ++cj) {
#pragma unroll
        for (int t = 0; t < kModuli; ++t) x[t] = y[t];
        if (cj + 1 < ncj) fetch(cj + 1);
        if (!rv || ((leave >> (cj >> 3)) & 1)) continue;
        const int c = c_lo + 4 * cj;
        double o[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int eb = c + u < c_hi ? p.b_col[V.bcol + c + u].x : 0;
          o[u] = crt_f64(x, u, ri.x + eb - 2 * p.bits);
        }
        double* const d = dst + c;
        if (p.g.accumulate) {
#pragma unroll
          for (int u = 0; u < 4; ++u)
            if (c + u < c_hi) o[u] += d[u];
        }
        if (c + 4 <= c_hi && (reinterpret_cast<uintptr_t>(d) & 15) == 0) {
          *reinterpret_cast<double2*>(d) = make_double2(o[0], o[1]);
          *reinterpret_cast<double2*>(d + 2) = make_double2(o[2], o[3]);
        } else {
#pragma unroll
          for (int u = 0; u < 4; ++u)
            if (c + u < c_hi) d[u] = o[u];
        }
      }
      __syncwarp();
      if constexpr (kSplit) {
        scr += par ? -slot : slot;
        par ^= 1;
      }
    }
  }

  tc::fence_before_sync();
  // a cluster: no CTA frees TMEM or exits while another may still signal its barriers
  // or (pairs) the issuer's MMAs read its shared memory
  if constexpr (kCluster)
    tc::cluster_sync();
  else
    __syncthreads();
  if (threadIdx.x == 0 && *abort) atomicExch(&p.hdr[0], 1);
  if (warp == 1) {
    tc::fence_after_sync();
    if constexpr (kPair)
      tc::tmem_dealloc_pair(tmem, 512);
    else
      tc::tmem_dealloc(tmem, 512);
  }
  if constexpr (kPair) tc::cluster_sync();
}

size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

TileGrid tile_grid(int64_t m, int64_t n, int64_t R, int64_t Cc, int bpt, bool pair) {
  const int bm = pair ? 2 * BM : BM;
  return TileGrid{(int)cdiv(m, bm), (int)cdiv(n, 64 * bpt), (int)cdiv(R, bm),
                  (int)cdiv(Cc, 64 * bpt), 2048 / bm};
}

}  // namespace

// Clusters of `split` CTAs that run at once (of six: 23, since a cluster stays within a
// GPC; the others with the same margin).
static int64_t split_workers(int split) {
  return split == 1 ? kSms : (split == 2 ? 74 : (split == 3 ? 46 : 22));
}

bool plan_f64_tc(const abft_desc& d, int64_t R, int64_t Cc, F64TcRegions* rg, size_t* bytes) {
  // 128^3: 136 us on the FP64 pipe (one 64 x 64 tile's chain of k), 32 here; below,
  // both are bound by latency and the FP64 pipe needs one launch instead of four
  // (1024 x 1024 x 64: 134 and 64 us, 100000 x 3 x 300: 3.34 and 0.65 ms).  A K loop is
  // padded to 64: from k = 48 on every shape measured is faster here (FP64 pipe / here,
  // plain products: 2048 x 2048 x 48 342 / 138 us, 64 x 65536 x 48 342 / 309, 2^20 x 1 x 48
  // 5.82 / 3.86 ms), at 32 some are slower (2048 x 2048 231 / 138 us, 64 x 65536 231 / 306)
  // and at 16 and below all are (2048 x 2048 x 16 119 / 136, 64 x 65536 x 2 119 / 493: with
  // so few terms many elements fail the magnitude check and run on both).
  if (d.k < kMinK || (double)d.m * (double)d.n * (double)d.k < 2097152.0) return false;
  F64TcRegions& r = *rg;
  r.row_cs = cdiv(d.m, 2 * BM) * 2 * BM;
  r.rows_a = r.row_cs + cdiv(R, 2 * BM) * 2 * BM;
  r.col_cs = cdiv(d.n, 256) * 256;
  r.cols_b = r.col_cs + cdiv(Cc, 256) * 256;
  // Panels of K: the planes take at most kPlaneBudget, five times what the operands and
  // the result take (36 bytes per element of A and B instead of 8, before padding) and
  // 256 MiB, and half of what these and the checksums leave of the device.  A product that has no room for
  // a panel of one k-step runs on the FP64 pipe: short K under very long sides, whose
  // planes are mostly padding, and operands that nearly fill the device.
  const int64_t per_k = (r.rows_a + r.cols_b) * kPlanes64 * 2;
  const double held = 8.0 * ((double)d.m * d.k + (double)d.k * d.n + (double)d.m * d.n);
  const double sums = 8.0 * ((double)R * (d.n + d.k) + (double)Cc * (d.m + d.k));
  const double budget =
      std::min({kPlaneBudget, 5.0 * held + 256 * kMiB, 0.5 * (kDeviceBytes - held - sums)});
  if (budget < (double)per_k * BK) return false;
  const int64_t fit = (int64_t)(budget / (double)per_k) / BK * BK;
  r.kp = std::min<int64_t>({cdiv(d.k, BK) * BK, kMaxPanel, fit});
  // Tile kind: clocks per k-step times waves.  The copies bind the one-CTA tiles
  // (L2 delivers about 75 bytes per clock and SM; a k-step of four, two, one boxes
  // is 48, 32, 24 KiB: 640, 420, 360 clocks at 4096^3, where the MMAs take 512,
  // 256, 192); a pair's CTAs copy 32 KiB per 512-clock k-step (590).  Whole steps
  // with pairs / four / two / one boxes: 512^3 241 / 237 / 190 / 170 us, 1000 x 1501
  // x 777 313 / 327 / 265 / 300, 2048 chain 1.32 / 1.16 / 1.25 / 1.58 ms, 4096^3
  // 3.03 / 3.11 / 3.24 / 4.61, 8192^3 encode + product 16.7 / 17.0 / 19.8 / 28.4.  The
  // model was fitted there; elsewhere (18 shapes from 256^3 to 8192^2 x 1024, ragged and
  // narrow ones, each kind and split forced in turn) its choice is within 1 % of the best
  // but for 4000 x 4000 x 500 (pairs 616 us, four boxes 586) and 6000 x 6000 x 2000 (four
  // boxes 2437, pairs 2343).
  // Few tiles leave SMs idle: their planes are split over clusters of 2, 3 or 6 CTAs
  // (the residues are put together in about 8000 clocks per box).  512^3 step with one /
  // two / three / six CTAs per tile of one box 171 / 157 / 149 / 156 us, of two boxes 193 /
  // 164 / 158 / 155; 1000 x 1501 x 777 with two boxes 259 / 261 / 273 / 281, four 322 / 250 /
  // 275 / 266.
  struct Kind {
    int bpt;
    bool pair;
    int clocks;
  };
  const Kind kinds[] = {{4, true, 590}, {4, false, 640}, {2, false, 420}, {1, false, 360}};
  const int64_t nkb = cdiv(std::min(d.k, r.kp), BK);
  double best = 0;
  for (const Kind& kd : kinds)
    for (int split : {1, 2, 3, 6}) {
      if (kd.pair && split > 1) continue;
      const int64_t t = tile_grid(d.m, d.n, R, Cc, kd.bpt, kd.pair).total();
      const int64_t workers = kd.pair ? kSms / 2 : split_workers(split);
      if (split > 1 && t > workers) continue;
      const double cost = ((double)kd.clocks * nkb * kPlanes64 + 8000.0 * kd.bpt) / split *
                          cdiv(t, workers);
      if (best == 0 || cost < best) {
        best = cost;
        r.bpt = kd.bpt;
        r.pair = kd.pair;
        r.split = split;
      }
    }
  const int64_t tiles = tile_grid(d.m, d.n, R, Cc, r.bpt, r.pair).total();
  const int64_t ctas = std::min<int64_t>(r.pair ? 2 * tiles : tiles, kSms);
  size_t off = 0;
  auto region = [&](size_t b) {
    const size_t o = off;
    off = align256(off + b);
    return o;
  };
  r.a_planes = region((size_t)kPlanes64 * r.rows_a * r.kp * 2);
  r.b_planes = region((size_t)kPlanes64 * r.cols_b * r.kp * 2);
  r.a_row = region(sizeof(int2) * r.rows_a);
  r.b_col = region(sizeof(int2) * r.cols_b);
  r.cmax = region(sizeof(uint32_t) * cdiv(r.kp, kMaxRows) * r.cols_b);
  r.bad = region((size_t)tiles * (r.pair ? 8 : 4) * 2 * r.bpt);
  r.scratch = region((size_t)ctas * (r.split > 1 ? 2 : 1) * kModuli * r.bpt * 8 * 256 *
                     sizeof(uint32_t));
  *bytes = off;
  return true;
}

cudaError_t launch_gemm_f64_tc(const Plan& P, const F64Args& g, void* ws, cudaStream_t st) {
  const F64TcRegions& r = P.f64tc;
  char* w = static_cast<char*>(ws) + P.f64tc_base;
  int* hdr = reinterpret_cast<int*>(static_cast<char*>(ws) + P.f64tc_hdr);
  const TileGrid T = tile_grid(g.m, g.n, g.R, g.Cc, r.bpt, r.pair);
  const char* stall = getenv("ABFT_TEST_STALL_PRODUCER");
  const auto kernel = r.pair      ? k_gemm_f64_tc<true, false>
                      : r.split > 1 ? k_gemm_f64_tc<false, true>
                                    : k_gemm_f64_tc<false, false>;
  const int boxes = cta_boxes(r.bpt, r.pair);
  const size_t smem = smem_bytes(boxes);
  cudaError_t e =
      cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  for (int64_t k0 = 0; k0 < g.k && e == cudaSuccess; k0 += r.kp) {
    F64Args gp = g;
    gp.k = std::min(r.kp, g.k - k0);
    gp.A += k0;
    gp.B += k0 * g.ldb;
    if (g.R) gp.acs += k0;
    if (g.Cc) gp.bcs += k0 * g.ldbcs;
    gp.accumulate = k0 > 0;
    const int64_t kpad = cdiv(gp.k, BK) * BK;

    SliceArgs a{};
    a.g = gp;
    a.kpad = kpad;
    // 2 k 2^(2 bits) < P
    const int bits = std::min(kMaxBits, (int)floor((kLog2P - 1 - log2((double)gp.k)) / 2));
    a.bits = bits;
    a.pa = reinterpret_cast<uint16_t*>(w + r.a_planes);
    a.pb = reinterpret_cast<uint16_t*>(w + r.b_planes);
    a.a_row = reinterpret_cast<int2*>(w + r.a_row);
    a.b_col = reinterpret_cast<int2*>(w + r.b_col);
    a.hdr = hdr;
    a.rows_a = r.rows_a; a.cols_b = r.cols_b; a.row_cs = r.row_cs; a.col_cs = r.col_cs;
    a.cmax = reinterpret_cast<uint32_t*>(w + r.cmax);
    a.tpr = 32;
    while (a.tpr < kSliceThreads && a.tpr * 8 < kpad) a.tpr *= 2;
    const int rpc = kSliceThreads / a.tpr;
    const int64_t nch = cdiv(gp.k, kMaxRows);
    a.n0 = cdiv(g.n, 32) * nch;
    a.n1 = cdiv(g.Cc, 32) * nch;
    a.n2 = cdiv(g.m, rpc);
    k_f64_max<<<(unsigned)(a.n0 + a.n1 + a.n2 + cdiv(g.R, rpc)), kSliceThreads, 0, st>>>(a);
    auto tiles = [&](int64_t rows, int64_t cols) {
      return cdiv(rows, a.rows) * cdiv(cdiv(cols, BK) * BK, kSliceCols);
    };
    a.rows = kSliceRows;
    if (tiles(kpad, g.n) + tiles(g.m, kpad) < 8 * num_sms()) a.rows = 4;
    a.n0 = tiles(kpad, g.n);
    a.n1 = tiles(kpad, g.Cc);
    a.n2 = tiles(g.m, kpad);
    k_f64_slice<<<(unsigned)(a.n0 + a.n1 + a.n2 + tiles(g.R, kpad)), kSliceThreads, 0, st>>>(a);
    if ((e = cudaGetLastError()) != cudaSuccess) break;

    Maps M;
    e = make_bf16_map(&M.a, a.pa, kPlanes64 * r.rows_a, kpad, kpad, BK, BM);
    if (e == cudaSuccess)
      e = make_bf16_map_boxes(&M.bw, a.pb, kPlanes64 * kpad, r.cols_b, r.cols_b, boxes);
    if (e == cudaSuccess)
      e = make_bf16_map(&M.b1, a.pb, kPlanes64 * kpad, r.cols_b, r.cols_b, BK, BK);
    if (e != cudaSuccess) break;
    ProdArgs p{};
    p.g = gp;
    p.T = T;
    p.nkb = (int)(kpad / BK);
    p.bpt = r.bpt;
    p.kpad = (int)kpad; p.rows_a = (int)r.rows_a; p.row_cs = (int)r.row_cs;
    p.col_cs = (int)r.col_cs;
    p.a_row = a.a_row;
    p.b_col = a.b_col;
    p.bad = reinterpret_cast<uint8_t*>(w + r.bad);
    p.hdr = hdr;
    p.scratch = reinterpret_cast<uint32_t*>(w + r.scratch);
    p.bits = bits;
    p.line = (float)(1.52 * ldexp(1.0, 53 - bits) * sqrt((double)gp.k));
    p.stall_test = stall && stall[0] == '1';
    p.wait_ns = p.stall_test ? 200000000ull : tc::kWaitLimitNs;
    const int per = r.pair ? 2 : r.split;  // CTAs per worker
    const int workers =
        per > 1 ? max_clusters(reinterpret_cast<const void*>(kernel), smem, per, kThreads)
                : num_sms();
    p.split = r.split;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = per;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.gridDim =
        dim3((unsigned)(per * std::min<int64_t>({T.total(), kSms / per, workers})), 1, 1);
    cfg.blockDim = dim3(kThreads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = per > 1 ? 1 : 0;
    if ((e = cudaLaunchKernelEx(&cfg, kernel, M, p)) != cudaSuccess) break;
    e = launch_gemm_f64_bad(gp, T, r.pair ? 4 : 2, r.bpt, hdr + 1, p.bad, st);
    count_launches(3);
  }
  return e;
}

}  // namespace abft
