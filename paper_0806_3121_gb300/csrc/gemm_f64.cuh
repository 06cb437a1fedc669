// Shared by the two binary64 products: the DFMA kernel (gemm_f64.cu) and the
// product on the tensor cores (gemm_f64_tc.cu).
#pragma once

#include "internal.cuh"

namespace abft {

// Linear tile index -> (tile row, tile column), tile rows >= tm being checksum
// rows and tile columns >= tn checksum columns.  Groups of `group` data tile
// rows run column by column; checksum tile rows are dealt round-robin to the
// groups and checksum tile columns follow each group's data columns, so
// consecutive CTAs share the A and B panels in L2.
struct TileGrid {
  int tm, tn;  // data tiles along rows / columns
  int tr, tc;  // checksum tiles along rows / columns (0 for the plain product)
  int group;
  __host__ __device__ int64_t total() const {
    return (int64_t)tm * tn + (int64_t)tr * tn + (int64_t)tm * tc;
  }
  __device__ __forceinline__ void decode(int64_t t, int& ty, int& tx) const {
    const int64_t ngr = (tm + group - 1) / group;
    int64_t off = 0;
    for (int64_t G = 0; G < ngr; ++G) {
      const int64_t gd = min((int64_t)group, (int64_t)tm - G * group);
      const int64_t nr = G < tr ? (tr - G + ngr - 1) / ngr : 0;
      const int64_t part1 = (gd + nr) * tn, part2 = gd * tc;
      if (t < off + part1 + part2) {
        int64_t u = t - off;
        if (u < part1) {
          const int64_t ri = u % (gd + nr);
          tx = (int)(u / (gd + nr));
          ty = ri < gd ? (int)(G * group + ri) : (int)(tm + G + (ri - gd) * ngr);
        } else {
          u -= part1;
          tx = (int)(tn + u / gd);
          ty = (int)(G * group + u % gd);
        }
        return;
      }
      off += part1 + part2;
    }
    ty = tx = 0;  // not reached for t inside the product
  }
};

// One binary64 product [A; acs] [B, bcs] without its corner.
struct F64Args {
  const double* A;
  const double* B;
  const double* acs;
  const double* bcs;
  double* C;
  double* E;
  double* F;
  int64_t lda, ldb, ldc, ldacs, ldbcs, lde, ldf;
  int64_t m, n, k, R, Cc;
  int accumulate;  // 1: add to C, E, F (a later panel of K) instead of writing them
};

// The DFMA kernel on the 32 x 32 chunks of the tiles (64 hpt x 64 bpt) of the product
// on the tensor cores whose byte in `bad` is set; returns at once when *any is zero.
cudaError_t launch_gemm_f64_bad(const F64Args& g, const TileGrid& tiles, int hpt, int bpt,
                                const int* any, const uint8_t* bad, cudaStream_t st);

// The product on the tensor cores in the workspace regions of P.f64tc.
cudaError_t launch_gemm_f64_tc(const Plan& P, const F64Args& g, void* ws, cudaStream_t st);

}  // namespace abft
