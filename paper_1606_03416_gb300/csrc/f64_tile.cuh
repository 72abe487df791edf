// Tiles of the FP64 products on the CUDA cores (f64_kernels.cu, realign.cu).
#pragma once
#include <cstdint>

namespace dg {
namespace f64tile {

constexpr int T = 64;        // columns of a tile (and rows, in the products over states)
constexpr int TR = 16;       // rows of a tile
constexpr int BK = 16;       // contraction slice
constexpr int TP = T + 1;    // padded shared-memory rows
constexpr int TRP = TR + 1;
constexpr int NT = 128;      // threads per CTA: 8 column lanes x 16 rows

// acc[j] += sum_q a(q) Bs[q][tx + 8 j] for j < JN, a(q) = As[q][row]. A count
// of its own per JN, not a predicate per group: a multiply-add that is
// predicated off takes its turn in the FP64 pipe all the same (n = 40 columns:
// 0.67 TFLOP/s with predicates).
template <int JN, int P>
__device__ __forceinline__ void fma_cols(const double (&As)[BK][P], const double (&Bs)[BK][TP], double (&acc)[8],
                                         int kn, int tx, int row) {
#pragma unroll 4
  for (int q = 0; q < kn; ++q) {
    const double a = As[q][row];
#pragma unroll
    for (int j = 0; j < JN; ++j) acc[j] = fma(a, Bs[q][tx + 8 * j], acc[j]);
  }
}

// The slice's kn <= 16 terms for the first jn <= 8 column groups of one row.
template <int P>
__device__ __forceinline__ void fma_slice(const double (&As)[BK][P], const double (&Bs)[BK][TP], double (&acc)[8],
                                          int kn, int jn, int tx, int row) {
  if (kn == BK && jn == 8) {
#pragma unroll
    for (int q = 0; q < BK; ++q) {
      const double a = As[q][row];
#pragma unroll
      for (int j = 0; j < 8; ++j) acc[j] = fma(a, Bs[q][tx + 8 * j], acc[j]);
    }
    return;
  }
  switch (jn) {
    case 8: fma_cols<8>(As, Bs, acc, kn, tx, row); break;
    case 7: fma_cols<7>(As, Bs, acc, kn, tx, row); break;
    case 6: fma_cols<6>(As, Bs, acc, kn, tx, row); break;
    case 5: fma_cols<5>(As, Bs, acc, kn, tx, row); break;
    case 4: fma_cols<4>(As, Bs, acc, kn, tx, row); break;
    case 3: fma_cols<3>(As, Bs, acc, kn, tx, row); break;
    case 2: fma_cols<2>(As, Bs, acc, kn, tx, row); break;
    case 1: fma_cols<1>(As, Bs, acc, kn, tx, row); break;
    default: break;
  }
}

// The 64 x 64 products over states: acc[i][j] += As[q][row[i]] Bs[q][tx + 8 j]
// for the row groups i and column groups j < lim[i] of this warp.
__device__ __forceinline__ void fma_outer(const double (&As)[BK][TP], const double (&Bs)[BK][TP],
                                          double (&acc)[4][8], int kn, const int (&lim)[4], int tx,
                                          const int (&row)[4]) {
  if (kn == BK && lim[0] == 8 && lim[1] == 8 && lim[2] == 8 && lim[3] == 8) {
#pragma unroll 4
    for (int q = 0; q < BK; ++q) {
      double b[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) b[j] = Bs[q][tx + 8 * j];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const double a = As[q][row[i]];
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[i][j] = fma(a, b[j], acc[i][j]);
      }
    }
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i) fma_slice(As, Bs, acc[i], kn, lim[i], tx, row[i]);
  }
}

// Column groups of eight that reach into [0, n).
__device__ __forceinline__ int groups8(int64_t n) { return n >= T ? 8 : (n <= 0 ? 0 : (int)((n + 7) >> 3)); }

}  // namespace f64tile
}  // namespace dg
