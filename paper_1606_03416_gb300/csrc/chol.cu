// Cholesky factor of the Gram matrix and its inverse from dense products
// (Alg. 1 step 3: S = U^T U, Y_hat = Y U^{-1}). The paper names the Cholesky
// factorisation, next to the eigensolve, as the part of the subspace problem
// to move onto dense matrix products (Conclusion); here it is a recursive
// blocked factorisation whose work is four products per level.
//
// Row-major lower view: S = L L^T with L = U^T lower, and what the step needs
// is L^{-1} = U^{-T} (Y_hat^T = L^{-1} Y^T). For the leading block split
// S = [S11, .; S21, S22] (n1 + n2 rows):
//   L11, L11^{-1}  from the block S11 (recursively),
//   L21 = S21 L11^{-T},
//   S22 <- S22 - L21 L21^T          (lower triangle only),
//   L22, L22^{-1}  from the updated S22 (recursively),
//   (L^{-1})21 = -L22^{-1} (L21 L11^{-1}),
// (Golub and Van Loan, Matrix Computations, 4th ed., Sec. 4.2 for the block
// Cholesky; the block form of the triangular inverse is the one of Sec. 3.1).
// Blocks of at most 64 rows are factored and inverted by one CTA (k_chol_leaf).
// Products with every side at least 512 run from exact BF16 slices on the
// tensor cores (sliced.cu), smaller ones on the FP64 cores in 8 x 8 tiles over
// the whole GPU (k_small_product). S is first equilibrated by powers of two
// (see k_scale_by_powers). Order 2999: 17.0 ms with a register-resident
// column-by-column leaf (0.18 ms each) and split 32 x 32 tiles, now 7.3 ms.
#include <algorithm>
#include <cmath>

#include "ctx.h"

namespace dg {

namespace {

// Rows of a block factored by one CTA. A leaf runs on one SM at two FP64
// multiply-adds per clock and the leaves are serial; smaller leaves would add a
// level of products (four launches per block) for what they save.
constexpr int kLeaf = 64;
constexpr int kB = 8;              // tile of the leaf
constexpr int kLP = kLeaf + 1;     // padded row
constexpr int64_t kSliced = 512;   // smallest product side run from slices
constexpr int kLeafWarps = 8;
constexpr int kLeafSmem = 2 * kLeaf * kLP * (int)sizeof(double);

// 1 / sqrt(p) for p > 0: the FP32 reciprocal square root of p's leading 24 bits
// (relative error below 2^-21) and one third-order step y (1 + e/2 + 3 e^2/8),
// e = 1 - p y^2 (Taylor's series of (1 - e)^{-1/2}), which leaves an error of the
// order e^3 < 2^-62 and rounding; p outside FP32's range through the library's
// rsqrt. The conversions are integer operations: a dependent FP64 operation,
// conversions and comparisons included, takes ~150 clocks here, and this chain
// is what a pivot costs.
__device__ __forceinline__ double inv_sqrt(double p) {
  const int hi = __double2hiint(p), lo = __double2loint(p), ex = hi >> 20;
  if (ex < 1023 - 100 || ex > 1023 + 100) return rsqrt(p);
  const float pf = __int_as_float(((ex - 1023 + 127) << 23) | ((hi & 0xfffff) << 3) | (int)((unsigned)lo >> 29));
  const int yi = __float_as_int(rsqrtf(pf));
  const double y = __hiloint2double((((yi >> 23) - 127 + 1023) << 20) | ((yi >> 3) & 0xfffff), (yi & 7) << 29);
  const double e = fma(-p * y, y, 1.0);
  return fma(fma(0.375, e, 0.5), y * e, y);
}

// One 8 x 8 tile product per warp: acc[u] += sum_q A[r][q] B(q, c + u), lane = (row
// r = lane / 4, columns c = 2 (lane mod 4) and c + 1); NT: B(q, c) = B[c][q].
template <bool NT>
__device__ __forceinline__ void tile_mul(const double* A, const double* B, double (&acc)[2], int r, int c) {
#pragma unroll
  for (int q = 0; q < kB; ++q) {
    const double a = A[r * kLP + q];
    acc[0] = fma(a, NT ? B[c * kLP + q] : B[q * kLP + c], acc[0]);
    acc[1] = fma(a, NT ? B[(c + 1) * kLP + q] : B[q * kLP + c + 1], acc[1]);
  }
}

// One CTA factors the n x n block (n <= 64) whose lower triangle is at A (lda)
// and writes L^{-1} (lower, strict upper zero) to Li (ldl); A is left as it was.
// Blocked by 8 x 8 tiles in shared memory (rows past n as the identity):
// for each block column p
//   1. warp 0 factors and inverts the diagonal tile in registers (8 dependent
//      pivots); meanwhile the other warps apply column p - 1 to the tiles right
//      of column p and form M_pj = sum_k L_pk W_kj, j < p, for the inverse W;
//   2. all warps: L_ip = A_ip L_pp^{-T} below, W_pj = -L_pp^{-1} M_pj to the left;
//   3. all warps: column p + 1 gets its update from column p.
// What bounds it: the FP64 pipe (2 multiply-adds per clock on one SM, ~40 us for
// the ~230 tile products and the pivots) and the chain of 64 pivots, which runs
// beside step 1's products. A pivot that is not positive and finite stops the
// block: *info = col0 + j + 1 (1-based column of the whole matrix) if *info was 0.
__global__ void __launch_bounds__(32 * kLeafWarps, 1) k_chol_leaf(const double* __restrict__ A, int64_t lda,
                                                                  double* __restrict__ Li, int64_t ldl, int n,
                                                                  int64_t col0, int* __restrict__ info) {
  extern __shared__ double sm_leaf[];
  double* L = sm_leaf;                // A, then L below the diagonal tiles
  double* W = sm_leaf + kLeaf * kLP;  // M, then W = L^{-1}
  __shared__ int failed;
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const int r = lane >> 2, c = 2 * (lane & 3);
  const int nb = (n + kB - 1) / kB;
  for (int e = t; e < kLeaf * kLeaf; e += 32 * kLeafWarps) {
    const int i = e / kLeaf, k = e % kLeaf;
    L[i * kLP + k] = (i < n && k <= i) ? A[(int64_t)i * lda + k] : (i == k ? 1.0 : 0.0);
    W[i * kLP + k] = 0.0;
  }
  if (t == 0) failed = 0;
  __syncthreads();
  auto at = [](double* X, int i, int j) { return X + (kB * i) * kLP + kB * j; };
  auto sub_nt = [&](int i, int j, int p) {  // A_ij -= L_ip L_jp^T
    double acc[2] = {0.0, 0.0};
    tile_mul<true>(at(L, i, p), at(L, j, p), acc, r, c);
    double* o = at(L, i, j) + r * kLP + c;
    o[0] -= acc[0];
    o[1] -= acc[1];
  };
  for (int p = 0; p < nb; ++p) {
    if (warp == 0) {
      // diagonal tile: a = its entries, w = the rows of the identity under the same row operations
      double* d = at(L, p, p) + r * kLP + c;
      double a[2] = {d[0], d[1]}, w[2] = {r == c ? 1.0 : 0.0, r == c + 1 ? 1.0 : 0.0};
#pragma unroll
      for (int j = 0; j < kB; ++j) {
        const double cj = (j & 1) ? a[1] : a[0];  // column j of the tile, held by lanes 4 i + j / 2
        const double pv = __shfl_sync(0xffffffffu, cj, 4 * j + j / 2);
        const int hi = __double2hiint(pv);
        if ((unsigned)hi >= 0x7ff00000u || (hi | __double2loint(pv)) == 0) {  // not positive and finite; the same in every lane
          if (lane == 0) {
            failed = 1;
            atomicCAS(info, 0, (int)(col0 + kB * p + j + 1));
          }
          break;
        }
        const double y = inv_sqrt(pv);
        const double lr = __shfl_sync(0xffffffffu, cj, 4 * r + j / 2) * y;        // L_rj
        const double l0 = __shfl_sync(0xffffffffu, cj, 4 * c + j / 2) * y;        // L_cj
        const double l1 = __shfl_sync(0xffffffffu, cj, 4 * (c + 1) + j / 2) * y;  // L_c+1,j
        const double w0 = __shfl_sync(0xffffffffu, w[0], 4 * j + (lane & 3)) * y;  // row j of W, divided
        const double w1 = __shfl_sync(0xffffffffu, w[1], 4 * j + (lane & 3)) * y;
        if (r > j) {
          if (c > j) a[0] = fma(-lr, l0, a[0]);
          if (c + 1 > j) a[1] = fma(-lr, l1, a[1]);
          w[0] = fma(-lr, w0, w[0]);
          w[1] = fma(-lr, w1, w[1]);
        } else if (r == j) {
          w[0] = w0;
          w[1] = w1;
        }
      }
      double* o = at(W, p, p) + r * kLP + c;
      o[0] = w[0];
      o[1] = w[1];
    } else {
      // tiles (i, j), p < j <= i, lose L_i,p-1 L_j,p-1^T; M_pj for j < p
      int k = 0;
      if (p > 0) {
        for (int j = 0; j < p; ++j, ++k) {
          if (k % (kLeafWarps - 1) != warp - 1) continue;
          double acc[2] = {0.0, 0.0};
          for (int q = j; q < p; ++q) tile_mul<false>(at(L, p, q), at(W, q, j), acc, r, c);
          double* o = at(W, p, j) + r * kLP + c;
          o[0] = acc[0];
          o[1] = acc[1];
        }
        for (int i = nb - 1; i > p; --i)
          for (int j = p + 1; j <= i; ++j, ++k)
            if (k % (kLeafWarps - 1) == warp - 1) sub_nt(i, j, p - 1);
      }
    }
    __syncthreads();
    if (failed) return;
    // L_ip for i > p, W_pj for j < p: one tile per warp in place (nb - 1 <= 7 tiles)
    if (warp < nb - 1) {
      double acc[2] = {0.0, 0.0};
      double* o;
      if (warp < p) {
        o = at(W, p, warp);
        tile_mul<false>(at(W, p, p), o, acc, r, c);
        acc[0] = -acc[0];
        acc[1] = -acc[1];
      } else {
        o = at(L, warp + 1, p);
        tile_mul<true>(o, at(W, p, p), acc, r, c);
      }
      __syncwarp();
      o[r * kLP + c] = acc[0];
      o[r * kLP + c + 1] = acc[1];
    }
    __syncthreads();
    if (p + 1 + warp < nb) sub_nt(p + 1 + warp, p + 1, p);
    __syncthreads();
  }
  for (int e = t; e < n * kLeaf; e += 32 * kLeafWarps) {
    const int i = e / kLeaf, k = e % kLeaf;
    if (k < n) Li[(int64_t)i * ldl + k] = k <= i ? W[i * kLP + k] : 0.0;
  }
}

// The four small products of a level, FP64 on the CUDA cores, one 8 x 8 output
// tile per 64-thread CTA (one SM does two multiply-adds per clock, so even a
// 64-row block's product needs many CTAs; a tile's operands come from L2):
//   kL21:  C[r, c] = sum_{k <= c} X[r, k] Z[c, k]     (Z = L11^{-1}, lower)
//   kS22:  C[r, c] -= sum_k X[r, k] X[c, k], c <= r
//   kLL:   C[r, c] = sum_{k >= c} X[r, k] Z[k, c]     (Z = L11^{-1}, lower)
//   kLi21: C[r, c] = -sum_{k <= r} X[r, k] Z[k, c]    (X = L22^{-1}, lower)
// Each sums its terms in order of k over the range its triangle leaves.
enum SmallKind { kL21, kS22, kLL, kLi21 };

template <int KIND>
__global__ void __launch_bounds__(64) k_small_product(const double* __restrict__ X, int64_t ldx,
                                                      const double* __restrict__ Z, int64_t ldz, double* C,
                                                      int64_t ldc, int rows, int cols, int K) {
  constexpr int KC = 64;
  constexpr bool ZT = KIND == kL21 || KIND == kS22;
  const int r0 = blockIdx.y * 8, c0 = blockIdx.x * 8;
  if (KIND == kS22 && c0 > r0 + 7) return;
  __shared__ double Xs[8][KC + 1], Zs[8][KC + 1];  // Zs[c][k]
  const int t = threadIdx.x, r = t >> 3, c = t & 7;
  const int kb = KIND == kLL ? c0 : 0;
  const int ke = KIND == kL21 ? min(K, c0 + 8) : (KIND == kLi21 ? min(K, r0 + 8) : K);
  double acc = 0.0;
  for (int k0 = kb; k0 < ke; k0 += KC) {
    const int kn = min(KC, ke - k0);
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      Xs[u][t] = (t < kn && r0 + u < rows) ? X[(int64_t)(r0 + u) * ldx + k0 + t] : 0.0;
      if (ZT) {
        Zs[u][t] = (t < kn && c0 + u < cols) ? Z[(int64_t)(c0 + u) * ldz + k0 + t] : 0.0;
      } else {
        const int k = r + 8 * u;
        Zs[c][k] = (k < kn && c0 + c < cols) ? Z[(int64_t)(k0 + k) * ldz + c0 + c] : 0.0;
      }
    }
    __syncthreads();
    if (kn == KC) {
#pragma unroll 16
      for (int k = 0; k < KC; ++k) acc = fma(Xs[r][k], Zs[c][k], acc);
    } else {
      for (int k = 0; k < kn; ++k) acc = fma(Xs[r][k], Zs[c][k], acc);
    }
    __syncthreads();
  }
  const int i = r0 + r, j = c0 + c;
  if (i >= rows || j >= cols) return;
  double* o = C + (int64_t)i * ldc + j;
  if (KIND == kS22) {
    if (j <= i) *o -= acc;
  } else {
    *o = KIND == kLi21 ? -acc : acc;
  }
}

// Exact equilibration: d_i = 2^{-round(log2(S_ii) / 2)} (1 for a diagonal
// entry that is not positive and finite, which the factorisation then
// rejects), and the lower triangle of S scaled to d_i S_ij d_j, whose
// diagonal lies in [1/2, 2]. Powers of two change no bits, and the factor of
// the scaled matrix is D L, so L^{-1} = (D L)^{-1} D. The slices of a product
// share one exponent per row, so without this a matrix whose diagonal spans
// many orders keeps fewer significant bits in the rows' smaller entries.
__global__ void k_diagonal_powers(const double* __restrict__ S, int64_t lda, int64_t n, double* __restrict__ d) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const double sii = S[i * lda + i];
    d[i] = (sii > 0.0 && isfinite(sii)) ? ldexp(1.0, -(int)rint(0.5 * log2(sii))) : 1.0;
  }
}

__global__ void k_scale_by_powers(double* __restrict__ S, int64_t lda, int64_t n, const double* __restrict__ d) {
  for (int64_t i = blockIdx.y; i < n; i += gridDim.y) {
    const double di = d[i];
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j <= i; j += (int64_t)gridDim.x * blockDim.x)
      S[i * lda + j] *= di * d[j];
  }
}

// S[i, j] = Li[i, j] d_j on the lower triangle (L^{-1} = (D L)^{-1} D).
__global__ void k_unscale_inverse(const double* __restrict__ Li, int64_t n, const double* __restrict__ d,
                                  double* __restrict__ S, int64_t lda) {
  const int64_t tot = n * n;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < tot; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = e / n, j = e % n;
    if (j <= i) S[i * lda + j] = Li[e] * d[j];
  }
}

unsigned grid_2d(int64_t tot) { return (unsigned)std::max<int64_t>(1, std::min<int64_t>((tot + 255) / 256, 152 * 16)); }

struct Chol {
  dgchefsi_ctx* ctx;
  double* A;     // the matrix (lower triangle; its Schur complements on return)
  int64_t lda;
  double* Li;    // L^{-1}, n x n, row stride n (strict upper zero)
  double* Lw;    // L below the leaves, n x n, row stride n
  double* T;     // scratch, n x n, row stride n
  int64_t n;
  int* info;     // device
  int* bad;      // device non-finite flag of the sliced products
  int slices;
  cudaStream_t st;

  template <int KIND>
  dgchefsi_status small(const double* X, int64_t ldx, const double* Z, int64_t ldz, double* C, int64_t ldc,
                        int64_t rows, int64_t cols, int64_t K) {
    k_small_product<KIND><<<dim3((unsigned)((cols + 7) / 8), (unsigned)((rows + 7) / 8)), 64, 0, st>>>(
        X, ldx, Z, ldz, C, ldc, (int)rows, (int)cols, (int)K);
    count_launch();
    DG_CUDA(cudaGetLastError());
    return DGCHEFSI_OK;
  }

  // The diagonal block at (i0, i0) of m rows, its Schur complement applied.
  dgchefsi_status block(int64_t i0, int64_t m) {
    double* a = A + i0 * lda + i0;
    double* li = Li + i0 * n + i0;
    if (m <= kLeaf) {
      k_chol_leaf<<<1, 32 * kLeafWarps, kLeafSmem, st>>>(a, lda, li, n, (int)m, i0, info);
      count_launch();
      DG_CUDA(cudaGetLastError());
      return DGCHEFSI_OK;
    }
    // split on a multiple of the leaf (of 256 once blocks are large), near the middle
    const int64_t q = m >= 1024 ? 256 : kLeaf;
    const int64_t m1 = std::max<int64_t>(q, (m / 2 + q / 2) / q * q);
    const int64_t m2 = m - m1;
    const bool sliced = std::min(m1, m2) >= kSliced;
    DG_TRY(block(i0, m1));
    double* a21 = a + m1 * lda;
    double* a22 = a21 + m1;
    double* l21 = Lw + (i0 + m1) * n + i0;
    double* li11 = li;
    double* li21 = li + m1 * n;
    double* li22 = li21 + m1;
    // L21 = S21 L11^{-T};  S22 -= L21 L21^T (lower)
    if (sliced) {
      DG_TRY(sliced_gemm(ctx, true, false, m2, m1, m1, a21, lda, li11, n, l21, n, slices, bad));
      DG_TRY(sliced_gemm(ctx, true, false, m2, m2, m1, l21, n, l21, n, a22, lda, slices, bad, m2, true));
    } else {
      DG_TRY(small<kL21>(a21, lda, li11, n, l21, n, m2, m1, m1));
      DG_TRY(small<kS22>(l21, n, l21, n, a22, lda, m2, m2, m1));
    }
    DG_TRY(block(i0 + m1, m2));
    // (L^{-1})21 = -L22^{-1} (L21 L11^{-1})
    if (sliced) {
      DG_TRY(sliced_gemm(ctx, false, false, m2, m1, m1, l21, n, li11, n, T, n, slices, bad));
      DG_TRY(sliced_gemm(ctx, false, true, m2, m1, m2, li22, n, T, n, li21, n, slices, bad, 0, false, true));
    } else {
      DG_TRY(small<kLL>(l21, n, li11, n, T, n, m2, m1, m1));
      DG_TRY(small<kLi21>(li22, n, T, n, li21, n, m2, m1, m2));
    }
    return DGCHEFSI_OK;
  }
};

}  // namespace

dgchefsi_status cholesky_inverse(dgchefsi_ctx* ctx, double* S, int64_t n, int64_t lda, int* info, int* bad) {
  if (n <= 0) return DGCHEFSI_OK;
  const size_t nn = (size_t)n * (size_t)n;
  DG_TRY(ensure(ctx, ctx->ws_chol, sizeof(double) * (3 * nn + (size_t)n), "Cholesky workspace"));
  double* Li = static_cast<double*>(ctx->ws_chol.p);
  double* d = Li + 3 * nn;
  Chol c{ctx, S, lda, Li, Li + nn, Li + 2 * nn, n, info, bad, std::max(ctx->products_slices, 10), ctx->stream};
  DG_CUDA(cudaFuncSetAttribute(k_chol_leaf, cudaFuncAttributeMaxDynamicSharedMemorySize, kLeafSmem));
  DG_CUDA(cudaMemsetAsync(Li, 0, sizeof(double) * nn, c.st));
  k_diagonal_powers<<<grid_2d(n), 256, 0, c.st>>>(S, lda, n, d);
  k_scale_by_powers<<<dim3((unsigned)std::min<int64_t>((n + 255) / 256, 64), (unsigned)std::min<int64_t>(n, 65535)),
                      256, 0, c.st>>>(S, lda, n, d);
  count_launch(2);
  DG_CUDA(cudaGetLastError());
  // the sliced products are only enqueued; their one status check is at the end
  DG_TRY(pair_products_begin(ctx));
  ctx->pairs_deferred = true;
  const dgchefsi_status run = c.block(0, n);
  ctx->pairs_deferred = false;
  if (run != DGCHEFSI_OK) return run;
  // L^{-1} into the lower triangle of S (its strict upper part is left unspecified)
  k_unscale_inverse<<<grid_2d((int64_t)nn), 256, 0, c.st>>>(Li, n, d, S, lda);
  count_launch();
  DG_CUDA(cudaGetLastError());
  return pair_products_status(ctx);
}

}  // namespace dg
