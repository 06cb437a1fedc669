// Checksum encoding for binary64 operands (section 2.1; the encoded operands
// of Eq. (1)) in two launches: k_enc64 streams A and B (each CTA takes a unit of
// one of five passes), k_enc64_norms forms the threshold norms from what it
// left.  Every sum has a fixed order, so the results do not depend on scheduling.
//
// Bound: the FP64 pipe (2 results per clock and SM).  Per element of A: e sum, w
// sum, row square, block checksum; per element of B: e sum, w sum, column square
// -- so the passes avoid every other binary64 instruction (weights come from a
// table instead of conversions, the warp sums of four rows of B share one
// transposing butterfly, the row squares run in a pass of their own whose lanes
// add 1 / 32 of a row before they meet: one reduction per 32 x 32 elements would
// cost as much as the squares).  The passes read A three times and B twice, which
// HBM has room for.  Small problems are bound by latency instead: a verify block's
// rows are split into 64-row segments over the warps of a CTA and eight rows of
// loads are in flight per thread.  Measured, both launches against the eight kernels
// before them: 512^3 902 -> 21 us, 2048^3 557 -> 66, 4096^3 on an 8 x 8 grid 1152 -> 252,
// 8192^3 on a 16 x 16 grid 2604 -> 935 (FP64 pipe: 850).

#include <algorithm>

#include "internal.cuh"

namespace abft {
namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kSegRows = 64;    // rows per segment of a verify block (A column sums)
constexpr int kSqRows = 256;    // rows per column-square partial of B
constexpr int kRowsB = 4;       // rows of B per warp in the row-checksum pass

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

struct EncArgs {
  const double* A;
  const double* B;
  int64_t lda, ldb, m, n, k;
  int vb_r, vb_c, er, ec;
  int64_t nvr, nvc, Cc;
  double* acs;     // 2 nvr rows of k: e^T A_I, w^T A_I
  double* S;       // f bs rows of k: block checksums
  double* bcs;     // k rows of Cc: B_J e, B_J w
  double* nArow;
  double* colsq;   // [ceil(k / 256)][n] partial column squares of B
  int p, f;
  int64_t bs;
  double* car_a;   // cleared: a fresh encode carries no deviation
  double* car_b;
  int32_t* status; // tensor-core product: its status word, cleared
  int wpu;         // warps that share a verify block's rows
  // CTAs of the passes, in this order (0: the pass is not wanted)
  int64_t n_acols, n_brows, n_ablk, n_bsq, n_arows;
};

// Column checksums of A: unit = 32 columns x one verify block, its rows in
// wpu contiguous parts, one per warp; acs[2I] = e^T A_I, acs[2I+1] = w^T A_I.
// Blocks of up to 64 rows are summed in row order by one warp.
__device__ __forceinline__ void enc_acols(const EncArgs& a, int64_t blk, double* sh,
                                          const double* wtab) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t nck = cdiv(a.k, 32), u = blk * (kWarps / a.wpu) + warp / a.wpu;
  const int part = warp % a.wpu;
  const bool uv = u < a.nvr * nck;
  const int64_t I = uv ? u / nck : 0, l = (uv ? u % nck : 0) * 32 + lane;
  const int64_t i0 = I * a.vb_r, i1 = min(i0 + (int64_t)a.vb_r, a.m);
  const int64_t len = max((int64_t)kSegRows, cdiv(a.vb_r, a.wpu));  // rows of a part
  const int64_t b0 = i0 + part * len, b1 = min(b0 + len, i1);
  const double sc = scalbn(1.0, -a.er);
  double se = 0.0, sw = 0.0;
  if (uv && l < a.k) {
    for (int64_t s0 = b0; s0 < b1; s0 += kSegRows) {
      const int nr = (int)min((int64_t)kSegRows, b1 - s0);
      const double* q = a.A + s0 * a.lda + l;
      double e = 0.0, w = 0.0;
      int t = 0;
      for (; t + 8 <= nr; t += 8) {
        double x[8];
#pragma unroll
        for (int r = 0; r < 8; ++r) x[r] = q[(t + r) * a.lda];
#pragma unroll
        for (int r = 0; r < 8; ++r) {
          e += x[r];
          w = fma(wtab[t + r], x[r], w);
        }
      }
      for (; t < nr; ++t) {
        const double x = q[t * a.lda];
        e += x;
        w = fma(wtab[t], x, w);
      }
      sw += w;
      if (s0 > i0) sw = fma((double)(s0 - i0) * sc, e, sw);  // (0 Inf would be NaN)
      se += e;
    }
  }
  if (a.wpu > 1) {
    sh[warp * 64 + lane] = se;
    sh[warp * 64 + 32 + lane] = sw;
    __syncthreads();
    if (part == 0)
      for (int w = warp + 1; w < warp + a.wpu; ++w) {
        se += sh[w * 64 + lane];
        sw += sh[w * 64 + 32 + lane];
      }
  }
  if (part == 0 && uv && l < a.k) {
    a.acs[(2 * I) * a.k + l] = se;
    a.acs[(2 * I + 1) * a.k + l] = sw;
  }
}

// Row checksums of B: a warp takes kRowsB rows x one verify block,
// bcs[l][2J] = B_J e, bcs[l][2J+1] = B_J w.
__device__ __forceinline__ void enc_brows(const EncArgs& a, int64_t blk) {
  const int lane = threadIdx.x & 31;
  const int64_t u = blk * kWarps + (threadIdx.x >> 5);
  const int64_t l0 = u / a.nvc * kRowsB, J = u % a.nvc;
  if (l0 >= a.k) return;
  const int64_t j0 = J * a.vb_c;
  const int len = (int)(min(j0 + (int64_t)a.vb_c, a.n) - j0);
  const int nr = (int)min((int64_t)kRowsB, a.k - l0);
  const double* q = a.B + l0 * a.ldb + j0;
  double v[2 * kRowsB];  // e sums, then w sums
#pragma unroll
  for (int r = 0; r < 2 * kRowsB; ++r) v[r] = 0.0;
  const double sc = scalbn(1.0, -a.ec), step = 32.0 * sc;
  double w = (double)(lane + 1) * sc;
#pragma unroll 4
  for (int t = lane; t < len; t += 32) {
#pragma unroll
    for (int r = 0; r < kRowsB; ++r) {
      const double x = r < nr ? q[r * a.ldb + t] : 0.0;
      v[r] += x;
      v[kRowsB + r] = fma(w, x, v[kRowsB + r]);
    }
    w += step;
  }
  // sums over the lanes, eight values at once: lane l ends with value l / 4
#pragma unroll
  for (int s = 16, h = kRowsB; h >= 1; s >>= 1, h >>= 1) {
    const bool upper = (lane & s) != 0;
#pragma unroll
    for (int i = 0; i < h; ++i) {
      const double send = upper ? v[i] : v[i + h];
      v[i] = (upper ? v[i + h] : v[i]) + __shfl_xor_sync(0xffffffffu, send, s);
    }
  }
  v[0] += __shfl_xor_sync(0xffffffffu, v[0], 2);
  v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
  const int idx = lane >> 2, r = idx % kRowsB, c = idx / kRowsB;
  if ((lane & 3) == 0 && r < nr)
    a.bcs[(l0 + r) * a.Cc + 2 * J + c] = v[0];
}

// Block checksum rows: row c bs + t of S = sum_I c_{c,I} A[I bs + t] (c < f).
__device__ __forceinline__ void enc_ablk(const EncArgs& a, int64_t blk, double* sh) {
  const int64_t nck = cdiv(a.k, kThreads), ct = blk / nck;
  const int64_t l = blk % nck * kThreads + threadIdx.x;
  const int c = (int)(ct / a.bs);
  const double* q = a.A + (ct - c * a.bs) * a.lda + l;
  const int64_t step = a.bs * a.lda;
  double s = 0.0;
  if (c == 0) {  // coefficients 1
    if (l < a.k) {
#pragma unroll 8
      for (int I = 0; I < a.p; ++I) s += q[I * step];
    }
  } else {
    for (int I0 = 0; I0 < a.p; I0 += kThreads) {  // the coefficients of 256 blocks at a time
      __syncthreads();
      if (I0 + (int)threadIdx.x < a.p) sh[threadIdx.x] = block_coef(c, I0 + threadIdx.x, a.p);
      __syncthreads();
      if (l < a.k) {
        const int n = min(kThreads, a.p - I0);
#pragma unroll 8
        for (int I = 0; I < n; ++I) s += sh[I] * q[(I0 + I) * step];
      }
    }
  }
  if (l < a.k) a.S[ct * a.k + l] = s;
}

// Partial column squares of B: 32 columns x 256 rows, 32 rows per warp.
__device__ __forceinline__ void enc_bsq(const EncArgs& a, int64_t blk, double* sh) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t ncj = cdiv(a.n, 32), c = blk / ncj, j = blk % ncj * 32 + lane;
  const int64_t l0 = c * kSqRows + warp * 32, l1 = min(l0 + 32, a.k);
  double s = 0.0;
  if (j < a.n) {
    const double* q = a.B + l0 * a.ldb + j;
#pragma unroll 8
    for (int64_t l = l0; l < l1; ++l, q += a.ldb) s = fma(*q, *q, s);
  }
  sh[warp * 32 + lane] = s;
  __syncthreads();
  if (warp == 0 && j < a.n) {
    for (int w = 1; w < kWarps; ++w) s += sh[w * 32 + lane];
    a.colsq[c * a.n + j] = s;
  }
}

// ||A_{i,:}||_2, one warp per row.
__device__ __forceinline__ void enc_arows(const EncArgs& a, int64_t blk) {
  const int64_t i = blk * kWarps + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (i >= a.m) return;
  const double* q = a.A + i * a.lda;
  double s[2] = {0.0, 0.0};
  int64_t l = lane;
#pragma unroll 4
  for (; l + 32 < a.k; l += 64) {
    const double x = q[l], y = q[l + 32];
    s[0] = fma(x, x, s[0]);
    s[1] = fma(y, y, s[1]);
  }
  if (l < a.k) s[0] = fma(q[l], q[l], s[0]);
  const double t = warp_sum(s[0] + s[1]);
  if (lane == 0) a.nArow[i] = sqrt(t);
}

__global__ void __launch_bounds__(kThreads) k_enc64(const EncArgs a) {
  __shared__ double sh[kWarps * 64];
  __shared__ double wtab[kSegRows];
  if (blockIdx.x == 0) {
    for (int64_t x = threadIdx.x; x < 2 * a.nvr; x += kThreads) a.car_a[x] = 0.0;
    for (int64_t x = threadIdx.x; x < 2 * a.nvc; x += kThreads) a.car_b[x] = 0.0;
    if (a.status && threadIdx.x < 2) a.status[threadIdx.x] = 0;
  }
  int64_t b = blockIdx.x;
  if (b < a.n_acols) {
    // weights at most 1: a weighted term never exceeds its element
    if (threadIdx.x < kSegRows)
      wtab[threadIdx.x] = (double)(threadIdx.x + 1) * scalbn(1.0, -a.er);
    __syncthreads();
    return enc_acols(a, b, sh, wtab);
  }
  b -= a.n_acols;
  if (b < a.n_brows) return enc_brows(a, b);
  b -= a.n_brows;
  if (b < a.n_ablk) return enc_ablk(a, b, sh);
  b -= a.n_ablk;
  if (b < a.n_bsq) return enc_bsq(a, b, sh);
  enc_arows(a, b - a.n_bsq);
}

// Threshold norms, one CTA per verify block: nblk[4I] = sqrt(sum_{t in I} v_t^2),
// nblk[4I+1] = sqrt(sum (w_t v_t)^2) with v the line norms of the block, and
// nblk[4I+2], nblk[4I+3] the norms of its two checksum vectors.  CTAs 0 .. nvr-1:
// row blocks of A; then the column blocks of B; then the column norms nBcol from their
// partial squares, 512 columns per CTA (a square root is some twenty instructions of
// the FP64 pipe, 16 clocks each per warp, so they are spread over CTAs of their own).
constexpr int kNormThreads = 512;
__global__ void __launch_bounds__(kNormThreads) k_enc64_norms(const EncArgs a, double* nAblk,
                                                              double* nBcol, double* nBblk) {
  __shared__ double sh[4][kNormThreads / 32];
  const int64_t nch = cdiv(a.k, kSqRows);
  auto column_square = [&](int64_t j) {
    double v = 0.0;
#pragma unroll 8
    for (int64_t c = 0; c < nch; ++c) v += a.colsq[c * a.n + j];
    return v;
  };
  if (blockIdx.x >= a.nvr + a.nvc) {
    const int64_t j = (blockIdx.x - a.nvr - a.nvc) * kNormThreads + threadIdx.x;
    if (j < a.n) nBcol[j] = sqrt(column_square(j));
    return;
  }
  const bool rows = blockIdx.x < a.nvr;
  const int64_t I = rows ? blockIdx.x : blockIdx.x - a.nvr;
  const int vb = rows ? a.vb_r : a.vb_c;
  const int64_t t0 = I * vb;
  const int len = (int)(min(t0 + (int64_t)vb, rows ? a.m : a.n) - t0);
  const double sc = scalbn(1.0, rows ? -a.er : -a.ec);
  double s[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 4
  for (int64_t l = threadIdx.x; l < a.k; l += kNormThreads) {
    double e, w;
    if (rows) {
      e = a.acs[(2 * I) * a.k + l];
      w = a.acs[(2 * I + 1) * a.k + l];
    } else {
      const double2 x = *reinterpret_cast<const double2*>(a.bcs + l * a.Cc + 2 * I);
      e = x.x;
      w = x.y;
    }
    s[2] = fma(e, e, s[2]);
    s[3] = fma(w, w, s[3]);
  }
  for (int t = threadIdx.x; t < len; t += kNormThreads) {
    double v2;
    if (rows) {
      const double v = a.nArow[t0 + t];
      v2 = v * v;
    } else {
      v2 = column_square(t0 + t);
    }
    const double w = (double)(t + 1) * sc;
    s[0] += v2;
    s[1] = fma(w * w, v2, s[1]);
  }
  // the four sums together, in a transposing butterfly (lane l: sum l / 8), the warps'
  // in shared memory, one warp per sum
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 16, h = 2; h >= 1; o >>= 1, h >>= 1) {
    const bool upper = (lane & o) != 0;
#pragma unroll
    for (int i = 0; i < h; ++i) {
      const double send = upper ? s[i] : s[i + h];
      s[i] = (upper ? s[i + h] : s[i]) + __shfl_xor_sync(0xffffffffu, send, o);
    }
  }
#pragma unroll
  for (int o = 4; o >= 1; o >>= 1) s[0] += __shfl_xor_sync(0xffffffffu, s[0], o);
  if ((lane & 7) == 0) sh[lane >> 3][warp] = s[0];
  __syncthreads();
  if (warp < 4) {
    const double t = warp_sum(lane < kNormThreads / 32 ? sh[warp][lane] : 0.0);
    if (lane == 0) ((rows ? nAblk : nBblk) + 4 * I)[warp] = sqrt(t);
  }
}

// ---------------------------------------------------------------- chained calls
// A chained product (section 3.2: stacked calls do not recompute checksums)
// takes its encoded rows of A / columns of B from an earlier product's
// expected checksums; k_carry bounds their deviation from the stored operand.

// Deviation bound of checksums carried out of an earlier product: its
// deviation per line stays within that product's unscaled threshold, so the
// largest one of verify block I is at most
//   car[2I+c] = max_t nvec[t] * (f1 * nblk[4I+c] + f2 * nblk[4I+2+c] + car_prev[2I+c]),
// nvec the earlier product's column norms of B (row side: row norms of A).
// One CTA.
__global__ void __launch_bounds__(kThreads) k_carry(const double* __restrict__ nvec, int64_t len,
                                                    const double* __restrict__ nblk,
                                                    const double* __restrict__ car_prev,
                                                    int64_t nvb, double f1, double f2,
                                                    double* __restrict__ car) {
  __shared__ double sh[kThreads / 32];
  __shared__ double s_mx;
  double mx = 0.0;
  for (int64_t t = threadIdx.x; t < len; t += kThreads) mx = fmax(mx, nvec[t]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = mx;
  __syncthreads();
  if (threadIdx.x == 0) {
    double v = 0.0;
    for (int w = 0; w < kThreads / 32; ++w) v = fmax(v, sh[w]);
    s_mx = v;
  }
  __syncthreads();
  mx = s_mx;
  for (int64_t x = threadIdx.x; x < 2 * nvb; x += kThreads) {
    const int64_t I = x >> 1, c = x & 1;
    car[x] = mx * (f1 * nblk[4 * I + c] + f2 * nblk[4 * I + 2 + c] + car_prev[x]);
  }
}

// The encode's launches, with the column-square partials of B at `part` (the
// workspace scratch, or the static array of abft_encode_noalloc).  rows / cols:
// form the checksum rows of A / columns of B (otherwise they are in ws already).
cudaError_t encode_f64_into(const Plan& P, const double* A, const double* B, void* ws,
                            double* part, bool rows, bool cols, cudaStream_t st) {
  const abft_desc& d = P.d;
  char* w = static_cast<char*>(ws);
  auto at = [&](size_t off) { return reinterpret_cast<double*>(w + off); };
  if (d.k == 0) {  // empty inner dimension: all checksums and norms are zero
    cudaMemsetAsync(at(P.L.nArow), 0, sizeof(double) * d.m, st);
    cudaMemsetAsync(at(P.L.nAblk), 0, sizeof(double) * 4 * P.nvr, st);
    cudaMemsetAsync(at(P.L.nBcol), 0, sizeof(double) * d.n, st);
    cudaMemsetAsync(at(P.L.nBblk), 0, sizeof(double) * 4 * P.nvc, st);
    cudaMemsetAsync(at(P.L.car_a), 0, sizeof(double) * 2 * P.nvr, st);
    cudaMemsetAsync(at(P.L.car_b), 0, sizeof(double) * 2 * P.nvc, st);
    return cudaGetLastError();
  }
  EncArgs a{};
  a.A = A; a.B = B;
  a.lda = d.lda; a.ldb = d.ldb; a.m = d.m; a.n = d.n; a.k = d.k;
  a.vb_r = d.vb_rows; a.vb_c = d.vb_cols; a.er = P.er; a.ec = P.ec;
  a.nvr = P.nvr; a.nvc = P.nvc; a.Cc = P.Cc;
  a.acs = at(P.L.acs);
  a.S = a.acs + 2 * P.nvr * d.k;
  a.bcs = at(P.L.bcs);
  a.nArow = at(P.L.nArow);
  a.colsq = part;
  a.p = d.grid_p; a.f = P.f; a.bs = P.bs;
  a.car_a = at(P.L.car_a);
  a.car_b = at(P.L.car_b);
  a.status = P.tc64 ? reinterpret_cast<int32_t*>(w + P.f64tc_hdr) : nullptr;
  a.wpu = 1;
  while (a.wpu < kWarps && a.wpu * kSegRows < d.vb_rows) a.wpu *= 2;
  a.n_acols = rows ? cdiv(P.nvr * cdiv(d.k, 32), kWarps / a.wpu) : 0;
  a.n_brows = cols ? cdiv(P.nvc * cdiv(d.k, kRowsB), kWarps) : 0;
  a.n_ablk = rows && P.bs > 0 ? P.f * P.bs * cdiv(d.k, kThreads) : 0;
  a.n_bsq = cdiv(d.n, 32) * cdiv(d.k, kSqRows);
  a.n_arows = cdiv(d.m, kWarps);
  k_enc64<<<(unsigned)(a.n_acols + a.n_brows + a.n_ablk + a.n_bsq + a.n_arows), kThreads, 0, st>>>(
      a);
  k_enc64_norms<<<(unsigned)(P.nvr + P.nvc + cdiv(d.n, kNormThreads)), kNormThreads, 0, st>>>(
      a, at(P.L.nAblk), at(P.L.nBcol), at(P.L.nBblk));
  count_launches(2);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_encode_f64(const Plan& P, const double* A, const double* B, void* ws,
                              cudaStream_t st) {
  return encode_f64_into(P, A, B, ws, scratch_view(P, ws).part, true, true, st);
}

// ---------------------------------------------------------------------------
// Encode without a workspace scratch region (abft_encode_noalloc).
//
// The encode's per-chunk partial sums normally live in the scratch part of the
// caller's workspace.  For callers that cannot allocate device memory, this
// variant keeps them in the file-scope array below instead.  The array is
// created by the CUDA runtime when this module is loaded on a device and stays
// resident on every device that loads the library until the process exits.
// Every call shares it; every slot a call reads is first written by the same
// call, so nothing needs clearing, but calls that overlap on the GPU race on
// it.
constexpr size_t kStaticEncodePartBytes = size_t(8) << 20;  // 8 MiB
static __device__ __align__(256) double g_encode_part[kStaticEncodePartBytes / sizeof(double)];

size_t static_encode_part_bytes() { return kStaticEncodePartBytes; }

// In host code the array's name is only a stand-in, not a device address:
// the address on the current device is looked up with cudaGetSymbolAddress on
// every call (it is not cached, so a device reset or a new context cannot
// leave a stale pointer behind).
cudaError_t launch_encode_f64_noalloc(const Plan& P, const double* A, const double* B, void* ws,
                                      cudaStream_t st) {
  void* part = nullptr;
  const cudaError_t e = cudaGetSymbolAddress(&part, g_encode_part);
  if (e != cudaSuccess) return e;
  return encode_f64_into(P, A, B, ws, static_cast<double*>(part), true, true, st);
}

// Deviation bounds of the checksums carried out of an earlier product PL
// (workspace wsL): its column checksum rows (one pair per row verify block)
// and its row checksum columns (one pair per column verify block).
cudaError_t launch_carry_rows(const Plan& PL, const void* wsL, double* car, cudaStream_t st) {
  const char* wl = static_cast<const char*>(wsL);
  k_carry<<<1, kThreads, 0, st>>>(reinterpret_cast<const double*>(wl + PL.L.nBcol), PL.d.n,
                                  reinterpret_cast<const double*>(wl + PL.L.nAblk),
                                  reinterpret_cast<const double*>(wl + PL.L.car_a), PL.nvr,
                                  PL.f1_col, PL.f2_col, car);
  return cudaGetLastError();
}
cudaError_t launch_carry_cols(const Plan& PR, const void* wsR, double* car, cudaStream_t st) {
  const char* wr = static_cast<const char*>(wsR);
  k_carry<<<1, kThreads, 0, st>>>(reinterpret_cast<const double*>(wr + PR.L.nArow), PR.d.m,
                                  reinterpret_cast<const double*>(wr + PR.L.nBblk),
                                  reinterpret_cast<const double*>(wr + PR.L.car_b), PR.nvc,
                                  PR.f1_row, PR.f2_row, car);
  return cudaGetLastError();
}

cudaError_t launch_encode_f64_chained(const Plan& P, const double* A, const double* B, void* ws,
                                      const Plan* PL, const void* wsL, const Plan* PR,
                                      const void* wsR, cudaStream_t st) {
  const abft_desc& d = P.d;
  if (d.k == 0) return launch_encode_f64(P, A, B, ws, st);  // nothing to carry: zero norms
  char* w = static_cast<char*>(ws);
  cudaError_t e = cudaSuccess;
  if (PL)  // rows of A: the earlier product's E (verify rows, then block checksum rows)
    e = cudaMemcpyAsync(w + P.L.acs, static_cast<const char*>(wsL) + PL->L.E,
                        sizeof(double) * (size_t)P.R * d.k, cudaMemcpyDeviceToDevice, st);
  if (PR && e == cudaSuccess)  // columns of B: the earlier product's F (k x Cc)
    e = cudaMemcpyAsync(w + P.L.bcs, static_cast<const char*>(wsR) + PR->L.F,
                        sizeof(double) * (size_t)d.k * P.Cc, cudaMemcpyDeviceToDevice, st);
  if (e == cudaSuccess)
    e = encode_f64_into(P, A, B, ws, scratch_view(P, ws).part, !PL, !PR, st);
  if (PL && e == cudaSuccess) {
    e = launch_carry_rows(*PL, wsL, reinterpret_cast<double*>(w + P.L.car_a), st);
    count_launches(1);
  }
  if (PR && e == cudaSuccess) {
    e = launch_carry_cols(*PR, wsR, reinterpret_cast<double*>(w + P.L.car_b), st);
    count_launches(1);
  }
  return e;
}

}  // namespace abft
