// Binary64 ABFT product (Eq. (1)): [A; acs] [B, bcs] on the FP64 FMA pipe, for
// products below 128^3 or with k < 48, products whose planes have no room
// (plan_f64_tc), checksum-free products without a workspace and the chunks that the product on the tensor cores (gemm_f64_tc.cu) leaves out.
//
// On GB300 the FP64 FMA pipe issues 2 DFMA per clock per SM (measured
// 1.20 TFLOP/s over 152 SMs); mma.sync f64 runs slower (1.05 TFLOP/s) and
// tcgen05 has no f64 kind, so the kernel is a shared-memory tiled DFMA GEMM
// whose only job is to keep that pipe busy.  A 64x64 tile per 256-thread CTA,
// 4x4 outputs per thread, BK = 16 with a register-prefetched double buffer.
// Memory traffic is ~(1/64 + 1/64) words per FMA, far below HBM and L2
// bandwidth at this FMA rate.
//
// Tiles are scheduled as one 1-D grid in a grouped order (TileGrid): data tiles,
// whole tiles of checksum rows (acs, writing E) and checksum columns (bcs,
// writing F); the corner (acs x bcs) is not computed.  Each output element is one
// FMA chain over k in increasing order.
#include <algorithm>

#include "gemm_f64.cuh"
#include "internal.cuh"

namespace abft {
namespace {

constexpr int BM = 64, BN = 64, BK = 16, kThreads = 256;

constexpr int GROUP_M = 16;  // tile rows per raster group

// The BM x BN tile at (row0, col0) of the data (cs_row = cs_col = false), of the
// checksum rows (cs_row) or of the checksum columns (cs_col); bit 2 r + c of mask:
// write its 32 x 32 quarter (r, c).
__device__ __forceinline__ void tile_f64(const F64Args& g, bool cs_row, bool cs_col, int64_t row0,
                                         int64_t col0, int mask) {
  // Source and destination of this tile.
  const double* Asrc = cs_row ? g.acs : g.A;
  const int64_t ldA = cs_row ? g.ldacs : g.lda, rlim = cs_row ? g.R : g.m;
  const double* Bsrc = cs_col ? g.bcs : g.B;
  const int64_t ldB = cs_col ? g.ldbcs : g.ldb, clim = cs_col ? g.Cc : g.n;
  double* Dst = cs_row ? g.E : (cs_col ? g.F : g.C);
  const int64_t ldD = cs_row ? g.lde : (cs_col ? g.ldf : g.ldc);

  __shared__ double As[2][BK][BM + 2];
  __shared__ double Bs[2][BK][BN];

  const int tid = threadIdx.x;
  const int tx = tid & 15, ty = tid >> 4;
  double acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int64_t row = row0 + ty + 16 * i;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int64_t col = col0 + tx + 16 * j;
      acc[i][j] = (g.accumulate && row < rlim && col < clim) ? Dst[row * ldD + col] : 0.0;
    }
  }

  double ra[4], rb[4];
  auto load = [&](int64_t k0) {
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int idx = e * kThreads + tid;
      const int r = idx >> 4, c = idx & 15;
      const int64_t row = row0 + r, kk = k0 + c;
      ra[e] = (row < rlim && kk < g.k) ? Asrc[row * ldA + kk] : 0.0;
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int idx = e * kThreads + tid;
      const int r = idx >> 6, c = idx & 63;
      const int64_t kk = k0 + r, col = col0 + c;
      rb[e] = (kk < g.k && col < clim) ? Bsrc[kk * ldB + col] : 0.0;
    }
  };
  auto store = [&](int buf) {
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int idx = e * kThreads + tid;
      As[buf][idx & 15][idx >> 4] = ra[e];
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int idx = e * kThreads + tid;
      Bs[buf][idx >> 6][idx & 63] = rb[e];
    }
  };

  const int64_t nk = cdiv(g.k, BK);
  load(0);
  store(0);
  __syncthreads();
  int buf = 0;
  for (int64_t kt = 0; kt < nk; ++kt) {
    if (kt + 1 < nk) load((kt + 1) * BK);
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      double a[4], b[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = As[buf][kk][ty + 16 * i];
#pragma unroll
      for (int j = 0; j < 4; ++j) b[j] = Bs[buf][kk][tx + 16 * j];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
    }
    if (kt + 1 < nk) store(buf ^ 1);
    __syncthreads();
    buf ^= 1;
  }

#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int64_t row = row0 + ty + 16 * i;
    if (row >= rlim) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int64_t col = col0 + tx + 16 * j;
      if (col < clim && (mask >> ((i >> 1) * 2 + (j >> 1)) & 1)) Dst[row * ldD + col] = acc[i][j];
    }
  }
}

__global__ void __launch_bounds__(kThreads, 2) k_gemm_f64(const F64Args g, const TileGrid T) {
  int ty, tx;
  T.decode(blockIdx.x, ty, tx);
  const bool cs_row = ty >= T.tm, cs_col = tx >= T.tn;
  tile_f64(g, cs_row, cs_col, (int64_t)(cs_row ? ty - T.tm : ty) * BM,
           (int64_t)(cs_col ? tx - T.tn : tx) * BN, 15);
}

// The 32 x 32 chunks that the product on the tensor cores left out (tiles of 64 hpt x
// 64 bpt; bad: per tile [chunk row][chunk column]), each with the BM x BN tile it is
// a quarter of.
__global__ void __launch_bounds__(kThreads, 2)
    k_gemm_f64_bad(const F64Args g, const TileGrid T, int hpt, int bpt, const int* any,
                   const uint8_t* bad) {
  if (*any == 0) return;
  const int64_t total = T.total() * hpt * bpt;
  for (int64_t u = blockIdx.x; u < total; u += gridDim.x) {
    const int64_t t = u / (hpt * bpt);
    const int s = (int)(u - t * hpt * bpt), sr = s % hpt, sc = s / hpt;
    const uint8_t* const b = bad + t * (4 * hpt * bpt) + 2 * sr * (2 * bpt) + 2 * sc;
    const int mask = (b[0] ? 1 : 0) | (b[1] ? 2 : 0) | (b[2 * bpt] ? 4 : 0) |
                     (b[2 * bpt + 1] ? 8 : 0);
    if (!mask) continue;
    int ty, tx;
    T.decode(t, ty, tx);
    const bool cs_row = ty >= T.tm, cs_col = tx >= T.tn;
    const int64_t row0 = ((int64_t)(cs_row ? ty - T.tm : ty) * hpt + sr) * BM;
    const int64_t col0 = ((int64_t)(cs_col ? tx - T.tn : tx) * bpt + sc) * BN;
    if (row0 >= (cs_row ? g.R : g.m) || col0 >= (cs_col ? g.Cc : g.n)) continue;
    __syncthreads();  // the previous tile's shared memory has been read
    tile_f64(g, cs_row, cs_col, row0, col0, mask);
  }
}

}  // namespace

cudaError_t launch_gemm_f64_bad(const F64Args& g, const TileGrid& tiles, int hpt, int bpt,
                                const int* any, const uint8_t* bad, cudaStream_t st) {
  const int64_t total = tiles.total() * hpt * bpt;
  const unsigned grid = (unsigned)std::min<int64_t>(total, 2 * num_sms());
  k_gemm_f64_bad<<<grid, kThreads, 0, st>>>(g, tiles, hpt, bpt, any, bad);
  count_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_gemm_f64(const Plan& P, const double* A, const double* B, double* C, void* ws,
                            bool checksums, cudaStream_t st) {
  const abft_desc& d = P.d;
  if (d.m == 0 || d.n == 0) return cudaSuccess;
  F64Args g{};
  g.A = A; g.B = B; g.C = C;
  g.lda = d.lda; g.ldb = d.ldb; g.ldc = d.ldc;
  g.m = d.m; g.n = d.n; g.k = d.k;
  if (checksums) {
    char* w = static_cast<char*>(ws);
    g.acs = reinterpret_cast<const double*>(w + P.L.acs);
    g.bcs = reinterpret_cast<const double*>(w + P.L.bcs);
    g.E = reinterpret_cast<double*>(w + P.L.E);
    g.F = reinterpret_cast<double*>(w + P.L.F);
    g.R = P.R;
    g.Cc = P.Cc;
    g.ldacs = d.k;
    g.ldbcs = g.ldf = P.Cc;
    g.lde = d.n;
  }
  if (P.tc64 && ws) return launch_gemm_f64_tc(P, g, ws, st);
  const TileGrid T{(int)cdiv(d.m, BM), (int)cdiv(d.n, BN), (int)cdiv(g.R, BM), (int)cdiv(g.Cc, BN),
                   GROUP_M};
  k_gemm_f64<<<(unsigned)T.total(), kThreads, 0, st>>>(g, T);
  count_launches(1);
  return cudaGetLastError();
}

}  // namespace abft
