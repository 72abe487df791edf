// FP64 kernels of the CheFSI cycle: block-sparse mat-vec with the Chebyshev
// recurrence fused into its epilogue (Alg. 1 step 2, Eq. matvec_3), the
// Lanczos vector operations (Alg. 1 step 1), the dense FP64 products of the
// subspace problem (Alg. 1 steps 3-5), the Fermi level and occupations, and the
// diagonal density blocks (Eq. densitymatrix).
//
// GB300 executes FP64 only on the CUDA-core DFMA pipe (tcgen05 has no FP64
// kind), two multiply-adds per clock and SM, so these kernels are ALU-bound by
// a wide margin and what a tile costs is the multiply-adds it issues, padding
// included. So the tiles are small (16 rows x up to 64 columns, 128 threads,
// one row x eight columns each; 64 x 64 for the products over states), a warp
// skips the 8-column groups and 4-row groups that lie outside the result, and
// the contraction runs to its own end, not to a multiple of a slice. A small
// tile also spreads a small problem evenly over the SMs; operands re-read for
// it come from L2 at a few bytes per clock. Operands are staged through shared
// memory in 16-deep slices.
// Measured, before (64 x 64 or 64 x 32 tiles, 256 threads) and now: H X at n_K =
// 40, 300 states 3.28 -> 1.47 ms (1.13 TFLOP/s), n_K = 64 and 4096 states 371 ms
// both (1.25); Gram matrix of 401 states of 12096 rows 12.7 -> 2.0 ms; density
// blocks at n_K = 64, 4096 states 16.9 -> 9.6 ms; pattern blocks at n_K = 40
// 3.75 -> 1.57 ms.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cooperative_groups.h>

#include "f64_tile.cuh"
#include "internal.h"

namespace dg {

static std::atomic<int64_t> g_launches{0};
void count_launch(int n) { g_launches.fetch_add(n, std::memory_order_relaxed); }
int64_t launch_count() { return g_launches.load(std::memory_order_relaxed); }

namespace {

using namespace f64tile;

// One Chebyshev step on a (16 states) x (64 rows of element K) tile:
// out = alpha * (sum_{K'} H_KK' in_K' - c in_K) - beta * prev_K.
__global__ void __launch_bounds__(NT) k_filter_step_f64(HView h, const double* __restrict__ in, int64_t ld,
                                                        const double* prev, double* out, int64_t ldo,
                                                        int64_t Ns, double alpha, double c, double beta,
                                                        const double* __restrict__ coef, int step) {
  if (coef) {  // coefficients in device memory ([c, alpha_0, beta_0, alpha_1, ...]; graph replays)
    c = coef[0];
    alpha = coef[1 + 2 * step];
    beta = coef[2 + 2 * step];
  }
  const int K = blockIdx.y;
  const int nK = h.nb[K];
  const int j0 = blockIdx.z * T;
  if (j0 >= nK) return;
  const int64_t s0 = (int64_t)blockIdx.x * TR;
  __shared__ double As[BK][TRP];
  __shared__ double Bs[BK][TP];
  const int tid = threadIdx.x, tx = tid & 7, ty = tid >> 3;
  const int jn = groups8(nK - j0);
  const bool live = s0 + (ty & ~3) < Ns;  // this warp's four states
  double acc[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) acc[j] = 0.0;
  const int64_t offK = h.off[K];
  const int64_t e_end = h.row_ptr[K + 1];
  const int kk = tid & 15, rr = tid >> 4;
  for (int64_t e = h.row_ptr[K]; e < e_end; ++e) {
    const int Kp = h.col[e];
    const int nKp = h.nb[Kp];
    const int64_t offKp = h.off[Kp];
    const double* blk = h.vals + h.blk_off[e];
    for (int k0 = 0; k0 < nKp; k0 += BK) {
      const bool kin = (k0 + kk) < nKp;
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int r = rr + 8 * i;
        As[kk][r] = (kin && s0 + r < Ns) ? in[(s0 + r) * ld + offKp + k0 + kk] : 0.0;
      }
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int r = rr + 8 * i;
        if (i < jn) Bs[kk][r] = (kin && j0 + r < nK) ? blk[(int64_t)(j0 + r) * nKp + k0 + kk] : 0.0;
      }
      __syncthreads();
      if (live) fma_slice(As, Bs, acc, min(BK, nKp - k0), jn, tx, ty);
      __syncthreads();
    }
  }
  const int64_t s = s0 + ty;
  if (s >= Ns) return;
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const int jj = j0 + tx + 8 * j;
    if (jj >= nK) continue;
    const int64_t idx = s * ldo + offK + jj;
    double r = alpha * (acc[j] - c * in[s * ld + offK + jj]);
    if (beta != 0.0) r -= beta * prev[idx];
    out[idx] = r;
  }
}

// Row `row` of H times x, by one warp (the sum in every lane). The lanes fetch
// the descriptors of up to 32 neighbour blocks at once, so that the loads of
// the blocks' rows, not a chain of descriptor loads per block, are in flight.
// (x is no __restrict__ pointer: the Lanczos kernel reads what other CTAs wrote.)
__device__ __forceinline__ double warp_row_product(const HView& h, const double* x, int64_t row) {
  const int lane = threadIdx.x & 31;
  int lo = 0, hi = h.M;  // find K with off[K] <= row < off[K+1]
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (h.off[mid] <= row) lo = mid; else hi = mid;
  }
  const int K = lo;
  const int j = (int)(row - h.off[K]);
  double sum = 0.0;
  const int64_t e1 = h.row_ptr[K + 1];
  for (int64_t e0 = h.row_ptr[K]; e0 < e1; e0 += 32) {
    const int cnt = e1 - e0 < 32 ? (int)(e1 - e0) : 32;
    int n = 0;
    const double *brow = nullptr, *xs = nullptr;
    if (lane < cnt) {
      const int Kp = h.col[e0 + lane];
      n = h.nb[Kp];
      brow = h.vals + h.blk_off[e0 + lane] + (int64_t)j * n;
      xs = x + h.off[Kp];
    }
    for (int q0 = 0; q0 < cnt; q0 += 4) {  // four blocks' loads, then their multiply-adds
      double bv[4][2], xv[4][2];
      int nq[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int q = min(q0 + u, cnt - 1);
        nq[u] = __shfl_sync(0xffffffffu, n, q);
        const double* bq = reinterpret_cast<const double*>(__shfl_sync(0xffffffffu, reinterpret_cast<unsigned long long>(brow), q));
        const double* xq = reinterpret_cast<const double*>(__shfl_sync(0xffffffffu, reinterpret_cast<unsigned long long>(xs), q));
        if (q0 + u >= cnt) nq[u] = 0;
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          const bool in = lane + 32 * c < nq[u];
          bv[u][c] = in ? bq[lane + 32 * c] : 0.0;
          xv[u][c] = in ? xq[lane + 32 * c] : 0.0;
        }
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (nq[u] > 0) sum = fma(bv[u][0], xv[u][0], sum);
        if (nq[u] > 32) sum = fma(bv[u][1], xv[u][1], sum);
      }
    }
    if (__any_sync(0xffffffffu, n > 64))  // elements of more than 64 functions: the rest of their rows
      for (int q = 0; q < cnt; ++q) {
        const int nq = __shfl_sync(0xffffffffu, n, q);
        const double* bq = reinterpret_cast<const double*>(__shfl_sync(0xffffffffu, reinterpret_cast<unsigned long long>(brow), q));
        const double* xq = reinterpret_cast<const double*>(__shfl_sync(0xffffffffu, reinterpret_cast<unsigned long long>(xs), q));
        for (int jp = lane + 64; jp < nq; jp += 32) sum = fma(bq[jp], xq[jp], sum);
      }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  return sum;
}

// y = H x: one warp per row of H.
__global__ void k_spmv_f64(HView h, const double* __restrict__ x, double* __restrict__ y) {
  const int64_t row = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (row >= h.N) return;
  const double sum = warp_row_product(h, x, row);
  if ((threadIdx.x & 31) == 0) y[row] = sum;
}

__device__ __forceinline__ double block_sum(double v, double* red) {
  const int tid = threadIdx.x;
  red[tid] = v;
  __syncthreads();
  for (int s = blockDim.x >> 1; s > 0; s >>= 1) {
    if (tid < s) red[tid] += red[tid + s];
    __syncthreads();
  }
  const double r = red[0];
  __syncthreads();
  return r;
}

__global__ void k_dots_f64(const double* __restrict__ V, int64_t ldv, const double* __restrict__ w, int64_t n,
                           double* __restrict__ out) {
  __shared__ double red[256];
  const double* v = V + (int64_t)blockIdx.x * ldv;
  double s = 0.0;
  for (int64_t i = threadIdx.x; i < n; i += blockDim.x) s = fma(v[i], w[i], s);
  const double t = block_sum(s, red);
  if (threadIdx.x == 0) out[blockIdx.x] = t;
}

__global__ void k_sub_combination_f64(double* __restrict__ w, const double* __restrict__ V, int64_t ldv,
                                      const double* __restrict__ coef, int nv, int64_t n) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    double acc = 0.0;
    for (int l = 0; l < nv; ++l) acc = fma(coef[l], V[(int64_t)l * ldv + i], acc);
    w[i] -= acc;
  }
}

__global__ void k_axpby_f64(double a, const double* __restrict__ x, double b, const double* y, double* yo, int64_t n) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    yo[i] = a * x[i] + b * y[i];
}

// All k Lanczos steps with full re-orthogonalisation in one cooperative launch
// (a step by launches: ~8 of them and two host round trips, 65 us on a 256-row
// H). Each CTA owns a range of rows of every vector; what crosses CTAs are the
// dot products: each CTA writes its part to `part` (entry l of CTA b at l * grid
// + b), and after a grid barrier every CTA adds the parts in the same order, so
// all hold the same bits. Per step: w = H v_j - beta v_{j-1}, alpha = v_j . w |
// w -= alpha v_j, c = V^T w | w -= V c, beta = |w| | v_{j+1} = w / beta, with a
// barrier at each bar. V: k + 1 vectors, w: one. out: [0] |v0|, [1] steps taken,
// [2 + 2 j] alpha_j, [3 + 2 j] beta_j. Stops after a zero or non-finite beta.
// Bound by the row products (0.45 GB and 57 M multiply-adds per step on the
// 8x8x8 H, ~0.1 ms of the FP64 pipe) or, on small H, by the barriers.
// FP64 adds are few and far between: one warp adds the parts, takes the root and
// the reciprocal for its CTA (a warp's FP64 instruction takes 16 clocks of the
// SM whatever its lanes do, ~150 until its result can be used).
constexpr int LZ_THREADS = 1024;

__device__ __forceinline__ double lz_warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Sum of entry l's parts, by one warp.
__device__ __forceinline__ double lz_total(const double* part, int l) {
  double v = 0.0;
  for (int b = threadIdx.x & 31; b < (int)gridDim.x; b += 32) v += __ldcg(part + (int64_t)l * gridDim.x + b);
  return lz_warp_sum(v);
}

__global__ void __launch_bounds__(LZ_THREADS, 1) k_lanczos_f64(HView h, const double* __restrict__ v0, int k, double* V,
                                                               double* w, double* part, double* out) {
  namespace cg = cooperative_groups;
  cg::grid_group grid = cg::this_grid();
  __shared__ double red[LZ_THREADS / 32], coef[LZ_MAX_STEPS], tot[2];
  const int64_t N = h.N;
  const int64_t r0 = N * blockIdx.x / gridDim.x, r1 = N * (blockIdx.x + 1) / gridDim.x;
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31, nt = blockDim.x, nw = nt >> 5;
  const bool first = blockIdx.x == 0 && t == 0;
  // tot[0] = the total of a dot product of which v is this thread's part, or its
  // root and tot[1] the reciprocal of that
  auto all_sum = [&](double v, bool root) {
    v = lz_warp_sum(v);
    if (lane == 0) red[warp] = v;
    __syncthreads();
    if (warp == 0) {
      const double p = lz_warp_sum(lane < nw ? red[lane] : 0.0);
      if (lane == 0) __stcg(part + blockIdx.x, p);
    }
    grid.sync();
    if (warp == 0) {
      double s = lz_total(part, 0);
      if (root) s = sqrt(s);
      if (lane == 0) {
        tot[0] = s;
        if (root) tot[1] = 1.0 / s;
      }
    }
    __syncthreads();
  };
  double s = 0.0;
  for (int64_t i = r0 + t; i < r1; i += nt) s = fma(v0[i], v0[i], s);
  all_sum(s, true);
  const double nrm = tot[0];
  if (first) {
    out[0] = nrm;
    out[1] = 0.0;
  }
  if (!(nrm > 0.0) || !isfinite(nrm)) return;  // the same in every CTA
  double inv = tot[1], beta = 0.0;
  for (int64_t i = r0 + t; i < r1; i += nt) V[i] = v0[i] * inv;
  for (int j = 0; j < k; ++j) {
    const double* vj = V + (int64_t)j * N;
    grid.sync();  // v_j complete, and the parts of the last total read
    s = 0.0;
    for (int64_t i = r0 + warp; i < r1; i += nw) {
      double y = warp_row_product(h, vj, i);
      if (lane == 0) {
        if (j > 0) y -= beta * vj[i - N];
        w[i] = y;
        s = fma(vj[i], y, s);
      }
    }
    all_sum(s, false);
    const double alpha = tot[0];
    for (int64_t i = r0 + t; i < r1; i += nt) w[i] -= alpha * vj[i];
    __syncthreads();
    for (int l = warp; l <= j; l += nw) {  // parts 1 .. j + 1: entry 0 may still be read
      double c = 0.0;
      for (int64_t i = r0 + lane; i < r1; i += 32) c = fma(V[(int64_t)l * N + i], w[i], c);
      c = lz_warp_sum(c);
      if (lane == 0) __stcg(part + (int64_t)(l + 1) * gridDim.x + blockIdx.x, c);
    }
    grid.sync();
    for (int l = warp; l <= j; l += nw) {
      const double c = lz_total(part, l + 1);
      if (lane == 0) coef[l] = c;
    }
    __syncthreads();
    s = 0.0;
    for (int64_t i = r0 + t; i < r1; i += nt) {
      double acc = 0.0;
      for (int l = 0; l <= j; ++l) acc = fma(coef[l], V[(int64_t)l * N + i], acc);
      const double x = w[i] - acc;
      w[i] = x;
      s = fma(x, x, s);
    }
    all_sum(s, true);
    beta = tot[0];
    inv = tot[1];
    if (first) {
      out[1] = j + 1;
      out[2 + 2 * j] = alpha;
      out[3 + 2 * j] = beta;
    }
    if (j == k - 1 || beta == 0.0 || !isfinite(alpha) || !isfinite(beta)) return;  // the same in every CTA
    for (int64_t i = r0 + t; i < r1; i += nt) V[(int64_t)(j + 1) * N + i] = w[i] * inv;
  }
}

// What a product split along its contraction does with part z's result:
// written as the whole one (part 0), to the z-th block of the buffer of parts
// (another kernel adds these in order), or added to the parts before it.
enum PartTo { kWrite, kBuffer, kAdd };

// C[i,j] = sum_r A[i,r] B[j,r]; lower_only: the entries j <= i, mirrored. Part z =
// z0 + blockIdx.z sums kc terms; in a buffer (C + z * rows * cols, added by
// k_sum_parts_f64) all parts run at once: a product of few tiles and many terms (a
// Gram matrix of a few hundred states) fills the GPU.
__global__ void __launch_bounds__(NT) k_gemm_nt_f64(const double* __restrict__ A, int64_t lda,
                                                    const double* __restrict__ B, int64_t ldb, double* C,
                                                    int64_t ldc, int64_t rows, int64_t cols, int64_t K, int64_t kc,
                                                    int lower_only, int z0, PartTo to) {
  const int64_t nrt = (rows + TR - 1) / TR;
  const int64_t i0 = (blockIdx.x % nrt) * TR, j0 = (blockIdx.x / nrt) * T;
  if (lower_only && j0 > i0 + TR - 1) return;
  __shared__ double As[BK][TRP];
  __shared__ double Bs[BK][TP];
  const int tid = threadIdx.x, tx = tid & 7, ty = tid >> 3;
  const int jn = groups8((lower_only && i0 + TR < cols ? i0 + TR : cols) - j0);
  const bool live = i0 + (ty & ~3) < rows;
  double acc[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) acc[j] = 0.0;
  const int kk = tid & 15, rr = tid >> 4;
  const int64_t z = z0 + (int64_t)blockIdx.z, kb = z * kc, ke = kb + kc < K ? kb + kc : K;
  for (int64_t k0 = kb; k0 < ke; k0 += BK) {
    const bool kin = (k0 + kk) < ke;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int r = rr + 8 * i;
      As[kk][r] = (kin && i0 + r < rows) ? A[(i0 + r) * lda + k0 + kk] : 0.0;
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int r = rr + 8 * i;
      if (i < jn) Bs[kk][r] = (kin && j0 + r < cols) ? B[(j0 + r) * ldb + k0 + kk] : 0.0;
    }
    __syncthreads();
    if (live) fma_slice(As, Bs, acc, (int)(ke - k0 < BK ? ke - k0 : BK), jn, tx, ty);
    __syncthreads();
  }
  const int64_t ii = i0 + ty;
  if (ii >= rows) return;
  const bool part = to == kBuffer;
  double* c = C + (part ? z * rows * cols : 0);
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const int64_t jj = j0 + tx + 8 * j;
    if (jj >= cols || (lower_only && jj > ii)) continue;
    double* o = c + ii * (part ? cols : ldc) + jj;
    const double v = to == kAdd ? *o + acc[j] : acc[j];
    *o = v;
    if (lower_only && !part) c[jj * ldc + ii] = v;
  }
}

// C[i,j] = sum_z P[z][i,j], z ascending (P: parts x rows x cols); lower_only:
// the entries j <= i, mirrored.
__global__ void k_sum_parts_f64(const double* __restrict__ P, int parts, int64_t rows, int64_t cols,
                                double* __restrict__ C, int64_t ldc, int lower_only) {
  const int64_t tot = rows * cols;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < tot; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = e / cols, j = e - i * cols;
    if (lower_only && j > i) continue;
    double sum = P[e];
    for (int z = 1; z < parts; ++z) sum += P[(int64_t)z * tot + e];
    C[i * ldc + j] = sum;
    if (lower_only) C[j * ldc + i] = sum;
  }
}

__global__ void k_symmetrise_f64(double* C, int64_t n, int64_t ldc) {
  const int64_t i = (int64_t)blockIdx.y * blockDim.y + threadIdx.y;
  const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n || j >= n || j <= i) return;
  const double v = 0.5 * (C[i * ldc + j] + C[j * ldc + i]);
  C[i * ldc + j] = v;
  C[j * ldc + i] = v;
}

// C[i,r] = sum_l A[i,l] B[l,r]
__global__ void __launch_bounds__(NT) k_gemm_nn_f64(const double* __restrict__ A, int64_t lda,
                                                    const double* __restrict__ B, int64_t ldb,
                                                    double* __restrict__ C, int64_t ldc, int64_t rows,
                                                    int64_t cols, int64_t K, int a_lower) {
  const int64_t nrt = (rows + TR - 1) / TR;
  const int64_t i0 = (blockIdx.x % nrt) * TR, r0 = (blockIdx.x / nrt) * T;
  __shared__ double As[BK][TRP];
  __shared__ double Bs[BK][TP];
  const int tid = threadIdx.x, tx = tid & 7, ty = tid >> 3;
  const int jn = groups8(cols - r0);
  const bool live = i0 + (ty & ~3) < rows;
  double acc[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) acc[j] = 0.0;
  const int kk = tid & 15, rr = tid >> 4, cc = tid & 63;
  const int64_t kend = a_lower && i0 + TR < K ? i0 + TR : K;
  for (int64_t k0 = 0; k0 < kend; k0 += BK) {
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int r = rr + 8 * i;
      const int64_t l = k0 + kk, row = i0 + r;
      As[kk][r] = (l < K && row < rows && (!a_lower || l <= row)) ? A[row * lda + l] : 0.0;
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int kq = (tid >> 6) + 2 * i;
      const int64_t l = k0 + kq;
      Bs[kq][cc] = (l < K && r0 + cc < cols) ? B[l * ldb + r0 + cc] : 0.0;
    }
    __syncthreads();
    if (live) fma_slice(As, Bs, acc, (int)(kend - k0 < BK ? kend - k0 : BK), jn, tx, ty);
    __syncthreads();
  }
  const int64_t ii = i0 + ty;
  if (ii >= rows) return;
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const int64_t q = r0 + tx + 8 * j;
    if (q < cols) C[ii * ldc + q] = acc[j];
  }
}

// P_K[j, j'] = sum_i f_i X[i, off_K + j] X[i, off_K + j'] for j' <= j, mirrored
// (P_K is symmetric: half the multiply-adds). blockIdx.y: pair of 64-wide
// chunks of the element, chunk of j >= chunk of j'. Part z = z0 + blockIdx.z
// sums `sc` states; in a buffer (P + z * total, laid out like P, added by
// k_density_sum_f64) all parts run at once, so that few elements still fill the
// GPU and many fill it evenly.
__global__ void __launch_bounds__(NT) k_density_f64(HView h, const int64_t* __restrict__ poff,
                                                    const double* __restrict__ X, int64_t Ns, int64_t ld,
                                                    const double* __restrict__ f, int64_t sc, double* __restrict__ P,
                                                    int z0, PartTo to) {
  const int K = blockIdx.x;
  const int nK = h.nb[K];
  int ca = 0, cb = blockIdx.y;  // chunks of j and j': row ca of the lower triangle of chunk pairs
  while (cb > ca) cb -= ++ca;
  const int j0 = ca * T, jp0 = cb * T;
  if (j0 >= nK) return;
  const int64_t offK = h.off[K];
  __shared__ double As[BK][TP];
  __shared__ double Bs[BK][TP];
  const int tid = threadIdx.x, tx = tid & 7, ty = tid >> 3;
  int lim[4], row[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    // the warps take the four-row groups of a 16-row band forwards and backwards
    // in turn: below the diagonal later rows are longer, and each warp has its
    // own part of the FP64 pipe
    const int r4 = 16 * i + ((i & 1) ? 12 - (ty & ~3) : (ty & ~3));
    row[i] = r4 + (ty & 3);
    lim[i] = j0 + r4 < nK ? groups8(min(nK, j0 + r4 + 4) - jp0) : 0;
  }
  double acc[4][8];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 8; ++j) acc[i][j] = 0.0;
  const int cc = tid & 63;
  const int64_t z = z0 + (int64_t)blockIdx.z, sb = z * sc, se = sb + sc < Ns ? sb + sc : Ns;
  for (int64_t i0 = sb; i0 < se; i0 += BK) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int kk = (tid >> 6) + 2 * i;
      const int64_t s = i0 + kk;
      double v = 0.0, w = 0.0;
      if (s < se) {
        const double* xr = X + s * ld + offK;
        if (j0 + cc < nK) v = f[s] * xr[j0 + cc];
        if (jp0 + cc < nK) w = xr[jp0 + cc];
      }
      As[kk][cc] = v;
      Bs[kk][cc] = w;
    }
    __syncthreads();
    fma_outer(As, Bs, acc, (int)(se - i0 < BK ? se - i0 : BK), lim, tx, row);
    __syncthreads();
  }
  const bool part = to == kBuffer;
  double* PK = P + poff[K] + (part ? z * poff[h.M] : 0);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int jj = j0 + row[i];
    if (jj >= nK) continue;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int jq = jp0 + tx + 8 * j;
      if (jq > jj) continue;
      double* o = PK + (int64_t)jj * nK + jq;
      const double v = to == kAdd ? *o + acc[i][j] : acc[i][j];
      *o = v;
      if (!part) PK[(int64_t)jq * nK + jj] = v;
    }
  }
}

// P = the sum of the parts, z ascending, lower triangles mirrored. One CTA per element.
__global__ void k_density_sum_f64(HView h, const int64_t* __restrict__ poff, const double* __restrict__ part,
                                  int parts, double* __restrict__ P) {
  const int K = blockIdx.x;
  const int nK = h.nb[K];
  const int64_t total = poff[h.M];
  const double* p = part + poff[K];
  double* PK = P + poff[K];
  for (int e = threadIdx.x; e < nK * nK; e += blockDim.x) {
    const int j = e / nK, q = e - j * nK;
    if (q > j) continue;
    double sum = p[e];
    for (int z = 1; z < parts; ++z) sum += p[(int64_t)z * total + e];
    PK[e] = sum;
    PK[(int64_t)q * nK + j] = sum;
  }
}

__device__ __forceinline__ double fermi(double x) {
  if (x > 0.0) {
    const double e = exp(-x);
    return e / (1.0 + e);
  }
  return 1.0 / (1.0 + exp(x));
}

// Fermi level by bisection and occupations, by one cluster of up to 8 CTAs of
// 256 threads. Each CTA sums the occupations of its share of the states; the
// parts meet through distributed shared memory in one order, so every CTA takes
// the same branch. Bound by the FP64 exponentials of ~45 halvings (one SM does
// two multiply-adds per clock: 1.71 ms for 4096 states on one CTA that took the
// exponential of every state), so a state further than 45 kT from the level
// counts as 0 or 1, off by e^-45 < 2^-64, in the halvings.
constexpr int OCC_CTAS = 8;
__global__ void __launch_bounds__(256) k_occupations_f64(const double* __restrict__ lam, int64_t Ns, double Ne,
                                                        double kT, double* __restrict__ f, double* __restrict__ mu_out) {
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  const int nct = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  __shared__ double red[256], part[2];
  double vmin = INFINITY, vmax = -INFINITY;
  for (int64_t i = threadIdx.x; i < Ns; i += blockDim.x) {
    vmin = fmin(vmin, lam[i]);
    vmax = fmax(vmax, lam[i]);
  }
  red[threadIdx.x] = vmin;
  __syncthreads();
  for (int s = 128; s > 0; s >>= 1) {
    if (threadIdx.x < s) red[threadIdx.x] = fmin(red[threadIdx.x], red[threadIdx.x + s]);
    __syncthreads();
  }
  double lo = red[0] - 50.0 * kT;
  __syncthreads();
  red[threadIdx.x] = vmax;
  __syncthreads();
  for (int s = 128; s > 0; s >>= 1) {
    if (threadIdx.x < s) red[threadIdx.x] = fmax(red[threadIdx.x], red[threadIdx.x + s]);
    __syncthreads();
  }
  double hi = red[0] + 50.0 * kT;
  __syncthreads();
  const double tol = 1e-13 * Ne;
  // Ns states off by e^-45 each are below tol / 100 unless almost nothing is occupied
  const double far = Ne >= 1e-4 * (double)Ns ? 45.0 * kT : INFINITY;
  double mu = 0.5 * (lo + hi);
  const int64_t first = (int64_t)rank * blockDim.x + threadIdx.x, step = (int64_t)nct * blockDim.x;
  for (int it = 0; it < 200; ++it) {
    mu = 0.5 * (lo + hi);
    double s = 0.0;
    for (int64_t i = first; i < Ns; i += step) {
      const double x = lam[i] - mu;
      if (x < -far)
        s += 1.0;
      else if (!(x > far))
        s += fermi(x / kT);
    }
    s = block_sum(s, red);
    if (threadIdx.x == 0) part[it & 1] = s;  // the other buffer may still be read
    cl.sync();
    double total = 0.0;
    for (int c = 0; c < nct; ++c) total += *cl.map_shared_rank(&part[it & 1], c);
    const double count = 2.0 * total;
    if (fabs(count - Ne) <= tol) break;
    if (count < Ne) lo = mu; else hi = mu;
  }
  for (int64_t i = first; i < Ns; i += step) f[i] = fermi((lam[i] - mu) / kT);
  if (rank == 0 && threadIdx.x == 0) *mu_out = mu;
  cl.sync();  // no CTA leaves while another reads its part
}

__global__ void k_shift_diag_f64(double* A, int64_t n, double coef) {
  __shared__ double red[256];
  double t = 0.0;
  for (int64_t i = threadIdx.x; i < n; i += blockDim.x) t += A[i * n + i];
  red[threadIdx.x] = t;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
    __syncthreads();
  }
  const double sft = coef * red[0];
  for (int64_t i = threadIdx.x; i < n; i += blockDim.x) A[i * n + i] += sft;
}

__global__ void k_zero_strict_upper_f64(double* A, int64_t n, int64_t lda) {
  const int64_t i = (int64_t)blockIdx.y * blockDim.y + threadIdx.y;
  const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n && j < n && j > i) A[i * lda + j] = 0.0;
}

__global__ void k_check_finite_f64(const double* __restrict__ x, int64_t n, int* flag) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    if (!isfinite(x[i])) atomicOr(flag, 1);
}


// G_e += alpha * sum_s w_s A[s, off_K + j] B[s, off_K' + j'] for every stored
// block e = (K, K') (w may be null: unit weights). DIAG (A = B, G zero, alpha 1): the
// blocks with K = K' are formed as k_density_f64 does, in parts of diag_len states
// added in order, the entries j' <= j mirrored, so that they have its bits.
template <bool DIAG>
__global__ void __launch_bounds__(NT) k_block_outer_f64(HView h, const int32_t* __restrict__ blk_row,
                                                        const double* __restrict__ A, int64_t lda,
                                                        const double* __restrict__ B, int64_t ldb,
                                                        const double* __restrict__ w, double alpha, int64_t Ns,
                                                        double* __restrict__ G, int64_t diag_len) {
  const int64_t e = blockIdx.x;
  const int K = blk_row[e], Kp = h.col[e];
  const bool diag = DIAG && K == Kp;
  const int nK = h.nb[K], nKp = h.nb[Kp];
  const int j0 = blockIdx.y * T, jp0 = blockIdx.z * T;
  if (j0 >= nK || jp0 >= nKp || (diag && jp0 > j0)) return;
  const int64_t offK = h.off[K], offKp = h.off[Kp];
  __shared__ double As[BK][TP];
  __shared__ double Bs[BK][TP];
  const int tid = threadIdx.x, tx = tid & 7, ty = tid >> 3;
  int lim[4], row[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    row[i] = ty + 16 * i;
    const int r4 = j0 + 16 * i + (ty & ~3);
    lim[i] = r4 < nK ? groups8((diag ? min(nK, r4 + 4) : nKp) - jp0) : 0;
  }
  double acc[4][8];
  const int cc = tid & 63;
  double* Ge = G + h.blk_off[e];
  const int64_t len = DIAG && diag ? diag_len : Ns;
  for (int64_t sb = 0; sb < Ns; sb += len) {
    const int64_t se = sb + len < Ns ? sb + len : Ns;
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 8; ++j) acc[i][j] = 0.0;
    for (int64_t i0 = sb; i0 < se; i0 += BK) {
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int kk = (tid >> 6) + 2 * i;
        const int64_t s = i0 + kk;
        double v = 0.0, u = 0.0;
        if (s < se) {
          if (j0 + cc < nK) v = (w ? w[s] : 1.0) * A[s * lda + offK + j0 + cc];
          if (jp0 + cc < nKp) u = B[s * ldb + offKp + jp0 + cc];
        }
        As[kk][cc] = v;
        Bs[kk][cc] = u;
      }
      __syncthreads();
      fma_outer(As, Bs, acc, (int)(se - i0 < BK ? se - i0 : BK), lim, tx, row);
      __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int jj = j0 + row[i];
      if (jj >= nK) continue;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int jq = jp0 + tx + 8 * j;
        if (jq >= nKp || (diag && jq > jj)) continue;
        double* o = Ge + (int64_t)jj * nKp + jq;
        const double v = DIAG ? (sb == 0 ? acc[i][j] : *o + acc[i][j]) : *o + alpha * acc[i][j];
        *o = v;
        if (diag) Ge[(int64_t)jq * nKp + jj] = v;
      }
    }
  }
}

// C[i,r] = sum_l A[l,i] B[l,r]  (A: K x rows, B: K x cols, both row-major)
__global__ void __launch_bounds__(NT) k_gemm_tn_f64(const double* __restrict__ A, int64_t lda,
                                                    const double* __restrict__ B, int64_t ldb,
                                                    double* __restrict__ C, int64_t ldc, int64_t rows,
                                                    int64_t cols, int64_t K) {
  const int64_t nrt = (rows + TR - 1) / TR;
  const int64_t i0 = (blockIdx.x % nrt) * TR, r0 = (blockIdx.x / nrt) * T;
  __shared__ double As[BK][TRP];
  __shared__ double Bs[BK][TP];
  const int tid = threadIdx.x, tx = tid & 7, ty = tid >> 3;
  const int jn = groups8(cols - r0);
  const bool live = i0 + (ty & ~3) < rows;
  double acc[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) acc[j] = 0.0;
  const int ar = tid & 15, ak = tid >> 4, cc = tid & 63;
  for (int64_t k0 = 0; k0 < K; k0 += BK) {
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int64_t l = k0 + ak + 8 * i;
      As[ak + 8 * i][ar] = (l < K && i0 + ar < rows) ? A[l * lda + i0 + ar] : 0.0;
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int kq = (tid >> 6) + 2 * i;
      const int64_t l = k0 + kq;
      Bs[kq][cc] = (l < K && r0 + cc < cols) ? B[l * ldb + r0 + cc] : 0.0;
    }
    __syncthreads();
    if (live) fma_slice(As, Bs, acc, (int)(K - k0 < BK ? K - k0 : BK), jn, tx, ty);
    __syncthreads();
  }
  const int64_t ii = i0 + ty;
  if (ii >= rows) return;
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const int64_t q = r0 + tx + 8 * j;
    if (q < cols) C[ii * ldc + q] = acc[j];
  }
}

// out[i, r] = scale * g[i] * (HX[i, r] - lam[i] * X[i, r]) for r < n
__global__ void k_scaled_residual_f64(const double* __restrict__ HX, const double* __restrict__ X, int64_t ld,
                                      const double* __restrict__ lam, const double* __restrict__ g, double scale,
                                      int64_t Ns, int64_t n, double* __restrict__ out, int64_t ldo) {
  const int64_t i = blockIdx.y;
  if (i >= Ns) return;
  const double gi = scale * g[i], li = lam[i];
  for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < n; r += (int64_t)gridDim.x * blockDim.x)
    out[i * ldo + r] = gi * (HX[i * ld + r] - li * X[i * ld + r]);
}

inline unsigned cdiv(int64_t a, int64_t b) { return (unsigned)((a + b - 1) / b); }
inline unsigned stream_grid(int64_t n) {
  int64_t g = (n + 255) / 256;
  if (g > 152 * 16) g = 152 * 16;
  return (unsigned)(g < 1 ? 1 : g);
}

}  // namespace

cudaError_t filter_step_f64(const HView& h, const double* in, int64_t ld_in, const double* prev, double* out,
                            int64_t ld_out, int64_t Ns, double alpha, double c, double beta, cudaStream_t s) {
  if (Ns == 0) return cudaSuccess;
  k_filter_step_f64<<<dim3(cdiv(Ns, TR), (unsigned)h.M, cdiv(h.max_nb, T)), NT, 0, s>>>(
      h, in, ld_in, prev, out, ld_out, Ns, alpha, c, beta, nullptr, 0);
  count_launch();
  return cudaGetLastError();
}

cudaError_t filter_step_f64_dev(const HView& h, const double* in, int64_t ld_in, const double* prev, double* out,
                                int64_t ld_out, int64_t Ns, const double* coef, int step, cudaStream_t s) {
  if (Ns <= 0) return cudaSuccess;
  k_filter_step_f64<<<dim3(cdiv(Ns, TR), (unsigned)h.M, cdiv(h.max_nb, T)), NT, 0, s>>>(
      h, in, ld_in, prev, out, ld_out, Ns, 0.0, 0.0, 0.0, coef, step);
  count_launch();
  return cudaGetLastError();
}

// FP64 issue-rate probe: 8 independent DFMA chains per thread, nothing read
// from memory; the store happens only if the result hits a value it cannot
// take, which keeps the chains live without memory traffic.
__global__ void __launch_bounds__(256) k_dfma_rate(int64_t iters, double x, double* __restrict__ sink) {
  double a[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) a[i] = 1.0 + 1e-3 * (threadIdx.x + i);
  const double y = -0.5 * x;
  for (int64_t n = 0; n < iters; ++n) {
#pragma unroll
    for (int i = 0; i < 8; ++i) a[i] = fma(a[i], x, y);
  }
  double t = 0.0;
#pragma unroll
  for (int i = 0; i < 8; ++i) t += a[i];
  if (t == 1234.5678) sink[0] = t;
}

cudaError_t dfma_rate(int64_t iters, int blocks, double* sink, cudaStream_t s) {
  k_dfma_rate<<<blocks, 256, 0, s>>>(iters, 0.999999, sink);
  count_launch();
  return cudaGetLastError();
}

cudaError_t preload_lanczos_kernels() {
  // cudaFuncGetAttributes loads a kernel's module on a lazily loading runtime,
  // so a later launch of these kernels allocates no device memory for code.
  cudaFuncAttributes a;
  cudaError_t e;
  if ((e = cudaFuncGetAttributes(&a, k_spmv_f64)) != cudaSuccess) return e;
  if ((e = cudaFuncGetAttributes(&a, k_dots_f64)) != cudaSuccess) return e;
  if ((e = cudaFuncGetAttributes(&a, k_sub_combination_f64)) != cudaSuccess) return e;
  return cudaFuncGetAttributes(&a, k_axpby_f64);
}

cudaError_t spmv_f64(const HView& h, const double* x, double* y, cudaStream_t s) {
  const int64_t threads = h.N * 32;
  k_spmv_f64<<<cdiv(threads, 256), 256, 0, s>>>(h, x, y);
  count_launch();
  return cudaGetLastError();
}

cudaError_t lanczos_f64(const HView& h, const double* v0, int k, double* V, double* w, double* part, int64_t nnz,
                        double* out, cudaStream_t s) {
  // one CTA per 8 rows (or 16 K entries of H), at most one per SM; a warp per row
  // while there are few, else 1024 threads for the loads in flight
  int64_t g = std::min<int64_t>(std::max<int64_t>(nnz / 16384, h.N / 8) + 1, LZ_MAX_CTAS);
  int dev = 0, nsm = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  g = std::max<int64_t>(1, std::min<int64_t>(g, nsm));
  HView hv = h;
  void* args[] = {&hv, &v0, &k, &V, &w, &part, &out};
  const unsigned threads = h.N / g <= 8 ? 256 : LZ_THREADS;
  e = cudaLaunchCooperativeKernel((const void*)k_lanczos_f64, dim3((unsigned)g), dim3(threads), args, 0, s);
  count_launch();
  return e;
}

cudaError_t dots_f64(const double* V, int64_t ldv, int nv, const double* w, int64_t n, double* out, cudaStream_t s) {
  if (nv <= 0) return cudaSuccess;
  k_dots_f64<<<nv, 256, 0, s>>>(V, ldv, w, n, out);
  count_launch();
  return cudaGetLastError();
}

cudaError_t sub_combination_f64(double* w, const double* V, int64_t ldv, const double* coef, int nv, int64_t n,
                                cudaStream_t s) {
  if (nv <= 0) return cudaSuccess;
  k_sub_combination_f64<<<stream_grid(n), 256, 0, s>>>(w, V, ldv, coef, nv, n);
  count_launch();
  return cudaGetLastError();
}

cudaError_t axpby_f64(double a, const double* x, double b, const double* y, double* y_out, int64_t n,
                      cudaStream_t s) {
  k_axpby_f64<<<stream_grid(n), 256, 0, s>>>(a, x, b, y, y_out, n);
  count_launch();
  return cudaGetLastError();
}

// CTAs at which a product no longer gains from more parts: 16 per SM, so that an
// uneven last round, or tiles of uneven work, cost a few percent.
static constexpr int64_t kFillCtas = 16 * 152;

// Parts of at least 64 of n terms, as many as give kFillCtas CTAs (of `ctas` a
// part) and as `most` allows: their number and their length, a multiple of BK.
struct Split {
  int64_t np, len;
};
static Split split_of(int64_t n, int64_t ctas, int64_t most) {
  int64_t np = std::min((kFillCtas + ctas - 1) / ctas, std::min(n / 64, most));
  np = std::max<int64_t>(1, std::min<int64_t>(np, 65535));
  const int64_t len = std::max<int64_t>(BK, ((n + np - 1) / np + BK - 1) / BK * BK);
  return {std::max<int64_t>(1, (n + len - 1) / len), len};
}

static Split gemm_nt_split(int64_t rows, int64_t cols, int64_t K, bool lower_only, int64_t doubles) {
  const int64_t tiles = (int64_t)cdiv(rows, TR) * cdiv(cols, T);
  return split_of(K, lower_only ? (tiles + 1) / 2 : tiles, doubles / std::max<int64_t>(rows * cols, 1));
}

static Split density_split(const HView& h, int64_t total, int64_t Ns, int64_t doubles) {
  const int64_t chunks = cdiv(h.max_nb, T);
  return split_of(Ns, h.M * (chunks * (chunks + 1) / 2), doubles / total);
}

int64_t gemm_nt_parts(int64_t rows, int64_t cols, int64_t K, bool lower_only, int64_t doubles) {
  return rows == 0 || cols == 0 ? 1 : gemm_nt_split(rows, cols, K, lower_only, doubles).np;
}

int64_t density_parts(const HView& h, int64_t total, int64_t Ns, int64_t doubles, int64_t* len) {
  const Split sp = density_split(h, total, Ns, doubles);
  *len = sp.len;
  return sp.np;
}

cudaError_t gemm_nt_f64(const double* A, int64_t lda, const double* B, int64_t ldb, double* C, int64_t ldc,
                        int64_t rows, int64_t cols, int64_t K, bool lower_only, bool symmetrise, const Parts& parts,
                        cudaStream_t s) {
  if (rows == 0 || cols == 0) return cudaSuccess;
  const unsigned tiles = cdiv(rows, TR) * cdiv(cols, T);
  const Split sp = gemm_nt_split(rows, cols, K, lower_only, parts.doubles);
  const int lower = lower_only ? 1 : 0;
  if (sp.np > 1 && parts.p) {
    k_gemm_nt_f64<<<dim3(tiles, 1, (unsigned)sp.np), NT, 0, s>>>(A, lda, B, ldb, parts.p, ldc, rows, cols, K, sp.len,
                                                                lower, 0, kBuffer);
    k_sum_parts_f64<<<stream_grid(rows * cols), 256, 0, s>>>(parts.p, (int)sp.np, rows, cols, C, ldc, lower);
    count_launch(2);
  } else {
    for (int z = 0; z < (int)sp.np; ++z)
      k_gemm_nt_f64<<<tiles, NT, 0, s>>>(A, lda, B, ldb, C, ldc, rows, cols, K, sp.len, lower, z, z == 0 ? kWrite : kAdd);
    count_launch((int)sp.np);
  }
  if (symmetrise && rows == cols) {
    dim3 b2(32, 8), g2(cdiv(rows, 32), cdiv(rows, 8));
    k_symmetrise_f64<<<g2, b2, 0, s>>>(C, rows, ldc);
    count_launch();
  }
  return cudaGetLastError();
}

cudaError_t gemm_nn_f64(const double* A, int64_t lda, const double* B, int64_t ldb, double* C, int64_t ldc,
                        int64_t rows, int64_t cols, int64_t K, bool a_lower, cudaStream_t s) {
  if (rows == 0 || cols == 0) return cudaSuccess;
  const int64_t tiles = (int64_t)cdiv(rows, TR) * cdiv(cols, T);
  k_gemm_nn_f64<<<(unsigned)tiles, NT, 0, s>>>(A, lda, B, ldb, C, ldc, rows, cols, K, a_lower ? 1 : 0);
  count_launch();
  return cudaGetLastError();
}

cudaError_t density_f64(const HView& h, const int64_t* poff, int64_t total, const double* X, int64_t Ns, int64_t ld,
                        const double* f, double* P, const Parts& parts, cudaStream_t s) {
  const int64_t chunks = cdiv(h.max_nb, T), pairs = chunks * (chunks + 1) / 2;
  const Split sp = density_split(h, total, Ns, parts.doubles);
  if (sp.np > 1 && parts.p) {
    k_density_f64<<<dim3((unsigned)h.M, (unsigned)pairs, (unsigned)sp.np), NT, 0, s>>>(h, poff, X, Ns, ld, f, sp.len,
                                                                                      parts.p, 0, kBuffer);
    k_density_sum_f64<<<(unsigned)h.M, 256, 0, s>>>(h, poff, parts.p, (int)sp.np, P);
    count_launch(2);
  } else {
    for (int z = 0; z < (int)sp.np; ++z)
      k_density_f64<<<dim3((unsigned)h.M, (unsigned)pairs), NT, 0, s>>>(h, poff, X, Ns, ld, f, sp.len, P, z,
                                                                       z == 0 ? kWrite : kAdd);
    count_launch((int)sp.np);
  }
  return cudaGetLastError();
}

cudaError_t occupations_f64(const double* ritz, int64_t Ns, double Ne, double kT, double* f, double* mu,
                            cudaStream_t s) {
  // one CTA per 256 states up to a cluster of 8
  const unsigned ctas = (unsigned)std::max<int64_t>(1, std::min<int64_t>(OCC_CTAS, (Ns + 255) / 256));
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr = {};
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = ctas;
  attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
  cfg.gridDim = dim3(ctas);
  cfg.blockDim = dim3(256);
  cfg.stream = s;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, k_occupations_f64, ritz, Ns, Ne, kT, f, mu);
  count_launch();
  return e;
}

cudaError_t shift_diagonal_by_trace_f64(double* A, int64_t n, double coef, cudaStream_t s) {
  k_shift_diag_f64<<<1, 256, 0, s>>>(A, n, coef);
  count_launch();
  return cudaGetLastError();
}

cudaError_t zero_strict_upper_f64(double* A, int64_t n, int64_t lda, cudaStream_t s) {
  dim3 b(32, 8), g(cdiv(n, 32), cdiv(n, 8));
  k_zero_strict_upper_f64<<<g, b, 0, s>>>(A, n, lda);
  count_launch();
  return cudaGetLastError();
}


cudaError_t block_outer_f64(const HView& h, const int32_t* blk_row, int64_t nnzb, const double* A, int64_t lda,
                            const double* B, int64_t ldb, const double* w, double alpha, int64_t Ns, double* G,
                            int64_t diag_len, cudaStream_t s) {
  if (nnzb == 0) return cudaSuccess;
  dim3 grid((unsigned)nnzb, cdiv(h.max_nb, T), cdiv(h.max_nb, T));
  if (diag_len > 0)
    k_block_outer_f64<true><<<grid, NT, 0, s>>>(h, blk_row, A, lda, B, ldb, w, alpha, Ns, G, diag_len);
  else
    k_block_outer_f64<false><<<grid, NT, 0, s>>>(h, blk_row, A, lda, B, ldb, w, alpha, Ns, G, 0);
  count_launch();
  return cudaGetLastError();
}

cudaError_t gemm_tn_f64(const double* A, int64_t lda, const double* B, int64_t ldb, double* C, int64_t ldc,
                        int64_t rows, int64_t cols, int64_t K, cudaStream_t s) {
  if (rows == 0 || cols == 0) return cudaSuccess;
  const int64_t tiles = (int64_t)cdiv(rows, TR) * cdiv(cols, T);
  k_gemm_tn_f64<<<(unsigned)tiles, NT, 0, s>>>(A, lda, B, ldb, C, ldc, rows, cols, K);
  count_launch();
  return cudaGetLastError();
}

cudaError_t scaled_residual_f64(const double* HX, const double* X, int64_t ld, const double* lam, const double* g,
                                double scale, int64_t Ns, int64_t n, double* out, int64_t ldo, cudaStream_t s) {
  if (Ns == 0) return cudaSuccess;
  dim3 grid(cdiv(n, 256) > 64 ? 64 : cdiv(n, 256), (unsigned)Ns);
  k_scaled_residual_f64<<<grid, 256, 0, s>>>(HX, X, ld, lam, g, scale, Ns, n, out, ldo);
  count_launch();
  return cudaGetLastError();
}

cudaError_t check_finite_f64(const double* x, int64_t n, int* flag, cudaStream_t s) {
  k_check_finite_f64<<<stream_grid(n), 256, 0, s>>>(x, n, flag);
  count_launch();
  return cudaGetLastError();
}

}  // namespace dg
