// Steps around the cycle: re-alignment of the coefficient block to the next
// SCF step's basis (Sec. III.B.3, Eq. basis_rotation_3) and density-matrix
// blocks on all of H's pattern (Eq. densitymatrix for neighbouring elements).
//
// Re-alignment, per element K with old size q = J_K^i, new size p = J_K^{i+1}
// and R_K sample points:
//   T_K = (V_K^{i+1})^T V_K^{i}                      (p x q, k_overlap_f64)
//   X_new[s, K, j'] = sum_j T_K[j', j] X_old[s, K, j] (k_realign_f64)
// i.e. the paper's two products, the small one first (R_K p q + N_s p q
// multiply-adds instead of R_K N_s (p + q)). Both in FP64 on the DFMA pipe.
#include <algorithm>
#include <vector>

#include "ctx.h"
#include "f64_tile.cuh"

namespace dg {
namespace {

using namespace f64tile;

constexpr int SG = 64;  // states per CTA of k_realign_f64

// T_K = Vn_K^T Vo_K for every element; Vn_K (R x p), Vo_K (R x q) row-major.
// 16 new x 64 old basis functions per CTA.
__global__ void __launch_bounds__(NT) k_overlap_f64(const int32_t* __restrict__ nb_new, const int32_t* __restrict__ nb_old,
                                                    const int32_t* __restrict__ nr, const int64_t* __restrict__ vn_off,
                                                    const int64_t* __restrict__ vo_off, const int64_t* __restrict__ t_off,
                                                    const double* __restrict__ Vn, const double* __restrict__ Vo,
                                                    double* __restrict__ Tk) {
  const int K = blockIdx.x;
  const int p = nb_new[K], q = nb_old[K], R = nr[K];
  const int j0 = blockIdx.y * TR, i0 = blockIdx.z * T;
  if (j0 >= p || i0 >= q) return;
  __shared__ double As[BK][TRP];
  __shared__ double Bs[BK][TP];
  const int tid = threadIdx.x, tx = tid & 7, ty = tid >> 3;
  const int jn = groups8(q - i0);
  const bool live = j0 + (ty & ~3) < p;
  const double* vn = Vn + vn_off[K];
  const double* vo = Vo + vo_off[K];
  double acc[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) acc[j] = 0.0;
  const int ar = tid & 15, ak = tid >> 4, cc = tid & 63;
  for (int r0 = 0; r0 < R; r0 += BK) {
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int r = r0 + ak + 8 * i;
      As[ak + 8 * i][ar] = (r < R && j0 + ar < p) ? vn[(int64_t)r * p + j0 + ar] : 0.0;
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int kq = (tid >> 6) + 2 * i, r = r0 + kq;
      Bs[kq][cc] = (r < R && i0 + cc < q) ? vo[(int64_t)r * q + i0 + cc] : 0.0;
    }
    __syncthreads();
    if (live) fma_slice(As, Bs, acc, min(BK, R - r0), jn, tx, ty);
    __syncthreads();
  }
  double* t = Tk + t_off[K];
  const int jj = j0 + ty;
  if (jj >= p) return;
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const int i = i0 + tx + 8 * j;
    if (i < q) t[(int64_t)jj * q + i] = acc[j];
  }
}

// Y[s, on_K + j'] = sum_j X[s, oo_K + j] T_K[j', j]; 16 states x 64 new columns per CTA.
__global__ void __launch_bounds__(NT) k_realign_f64(const int32_t* __restrict__ nb_new, const int32_t* __restrict__ nb_old,
                                                    const int64_t* __restrict__ off_new, const int64_t* __restrict__ off_old,
                                                    const int64_t* __restrict__ t_off, const double* __restrict__ Tk,
                                                    const double* __restrict__ X, int64_t ldx, double* __restrict__ Y,
                                                    int64_t ldy, int64_t Ns) {
  const int K = blockIdx.x;
  const int p = nb_new[K], q = nb_old[K];
  const int64_t s0 = (int64_t)blockIdx.y * SG;  // SG states per CTA, TR at a time
  const int jp0 = blockIdx.z * T;
  if (s0 >= Ns || jp0 >= p) return;
  __shared__ double As[BK][TRP];
  __shared__ double Bs[BK][TP];
  const int tid = threadIdx.x, tx = tid & 7, ty = tid >> 3;
  const int jn = groups8(p - jp0);
  const double* t = Tk + t_off[K];
  const int64_t oo = off_old[K], on = off_new[K];
  const int kk = tid & 15, rr = tid >> 4;
  for (int64_t sb = s0; sb < Ns && sb < s0 + SG; sb += TR) {
    const bool live = sb + (ty & ~3) < Ns;
    double acc[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) acc[j] = 0.0;
    for (int k0 = 0; k0 < q; k0 += BK) {
      const bool kin = k0 + kk < q;
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int r = rr + 8 * i;
        As[kk][r] = (kin && sb + r < Ns) ? X[(sb + r) * ldx + oo + k0 + kk] : 0.0;
      }
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int r = rr + 8 * i;
        if (i < jn) Bs[kk][r] = (kin && jp0 + r < p) ? t[(int64_t)(jp0 + r) * q + k0 + kk] : 0.0;
      }
      __syncthreads();
      if (live) fma_slice(As, Bs, acc, min(BK, q - k0), jn, tx, ty);
      __syncthreads();
    }
    const int64_t s = sb + ty;
    if (s < Ns) {
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int jp = jp0 + tx + 8 * j;
        if (jp < p) Y[s * ldy + on + jp] = acc[j];
      }
    }
  }
}

}  // namespace
}  // namespace dg

using namespace dg;

extern "C" dgchefsi_status dgchefsi_realign(dgchefsi_ctx* ctx, const int32_t* nb_old, const int32_t* nr,
                                            const double* V_old, const double* V_new, const double* X_old, int64_t Ns,
                                            int64_t ld_old, double* X_new, int64_t ld) {
  clear_error();
  if (!ctx) return set_error(DGCHEFSI_ERR_ARG, "null context");
  if (!nb_old || !nr || !V_old || !V_new || !X_old || !X_new) return set_error(DGCHEFSI_ERR_ARG, "null pointer");
  if (Ns < 1) return set_error(DGCHEFSI_ERR_ARG, "Ns < 1");
  const int M = ctx->M;
  std::vector<int64_t> off_old(M + 1, 0), vo(M + 1, 0), vn(M + 1, 0), to(M + 1, 0);
  int max_old = 0;
  for (int K = 0; K < M; ++K) {
    const int q = nb_old[K], p = ctx->nb_h[K], R = nr[K];
    if (q < 1 || q > 256) return set_error(DGCHEFSI_ERR_ARG, "nb_old[%d] = %d outside 1..256", K, q);
    if (R < 1) return set_error(DGCHEFSI_ERR_ARG, "nr[%d] = %d < 1", K, R);
    off_old[K + 1] = off_old[K] + q;
    vo[K + 1] = vo[K] + (int64_t)R * q;
    vn[K + 1] = vn[K] + (int64_t)R * p;
    to[K + 1] = to[K] + (int64_t)p * q;
    max_old = std::max(max_old, q);
  }
  if (ld_old < off_old[M]) return set_error(DGCHEFSI_ERR_ARG, "ld_old < sum of old element sizes");
  if (ld < ctx->N) return set_error(DGCHEFSI_ERR_ARG, "ld < N");
  // the two blocks must not overlap
  const char* a0 = reinterpret_cast<const char*>(X_old);
  const char* a1 = a0 + sizeof(double) * ((size_t)(Ns - 1) * ld_old + off_old[M]);
  const char* b0 = reinterpret_cast<const char*>(X_new);
  const char* b1 = b0 + sizeof(double) * ((size_t)(Ns - 1) * ld + ctx->N);
  if (a0 < b1 && b0 < a1) return set_error(DGCHEFSI_ERR_ARG, "X_new overlaps X_old");
  cudaStream_t s = ctx->stream;
  // device copies of the per-element tables (4 x [M+1] int64, 2 x [M] int32) and T
  const size_t tab = sizeof(int64_t) * 4 * (size_t)(M + 1) + sizeof(int32_t) * 2 * (size_t)M;
  const size_t tab_al = (tab + 255) / 256 * 256;
  DG_TRY(ensure(ctx, ctx->ws_realign, tab_al + sizeof(double) * (size_t)std::max<int64_t>(to[M], 1), "re-alignment tables"));
  std::vector<char> host(tab);
  char* hp = host.data();
  auto put = [&](const void* src, size_t n) {
    std::copy(static_cast<const char*>(src), static_cast<const char*>(src) + n, hp);
    hp += n;
  };
  put(off_old.data(), sizeof(int64_t) * (M + 1));
  put(vo.data(), sizeof(int64_t) * (M + 1));
  put(vn.data(), sizeof(int64_t) * (M + 1));
  put(to.data(), sizeof(int64_t) * (M + 1));
  put(nb_old, sizeof(int32_t) * M);
  put(nr, sizeof(int32_t) * M);
  char* dbase = static_cast<char*>(ctx->ws_realign.p);
  DG_CUDA(cudaMemcpyAsync(dbase, host.data(), tab, cudaMemcpyHostToDevice, s));
  const int64_t* d_off_old = reinterpret_cast<const int64_t*>(dbase);
  const int64_t* d_vo = d_off_old + (M + 1);
  const int64_t* d_vn = d_vo + (M + 1);
  const int64_t* d_to = d_vn + (M + 1);
  const int32_t* d_nb_old = reinterpret_cast<const int32_t*>(d_to + (M + 1));
  const int32_t* d_nr = d_nb_old + M;
  double* Tk = reinterpret_cast<double*>(dbase + tab_al);
  const unsigned tp = (unsigned)((ctx->max_nb + TR - 1) / TR), tq = (unsigned)((max_old + T - 1) / T);
  k_overlap_f64<<<dim3((unsigned)M, tp, tq), NT, 0, s>>>(ctx->nb_d, d_nb_old, d_nr, d_vn, d_vo, d_to, V_new, V_old, Tk);
  count_launch();
  DG_CUDA(cudaGetLastError());
  const int64_t st = (Ns + SG - 1) / SG;
  if (st > 65535) return set_error(DGCHEFSI_ERR_UNSUPPORTED, "Ns too large for one launch");
  k_realign_f64<<<dim3((unsigned)M, (unsigned)st, (unsigned)((ctx->max_nb + T - 1) / T)), NT, 0, s>>>(
      ctx->nb_d, d_nb_old, ctx->off_d, d_off_old, d_to, Tk, X_old, ld_old, X_new, ld, Ns);
  count_launch();
  DG_CUDA(cudaGetLastError());
  // the host table must outlive the asynchronous copy from pageable memory
  DG_CUDA(cudaStreamSynchronize(s));
  return DGCHEFSI_OK;
}

extern "C" dgchefsi_status dgchefsi_density_pattern(dgchefsi_ctx* ctx, const double* X, int64_t Ns, int64_t ld,
                                                    const double* f, double* P) {
  clear_error();
  if (!ctx) return set_error(DGCHEFSI_ERR_ARG, "null context");
  if (!X || !f || !P) return set_error(DGCHEFSI_ERR_ARG, "null pointer");
  if (Ns < 1) return set_error(DGCHEFSI_ERR_ARG, "Ns < 1");
  if (ld < ctx->N) return set_error(DGCHEFSI_ERR_ARG, "ld < N");
  cudaStream_t s = ctx->stream;
  DG_CUDA(cudaMemsetAsync(P, 0, sizeof(double) * (size_t)ctx->n_values, s));
  // the diagonal blocks with the bits of dgchefsi_density_blocks
  int64_t len = 0;
  density_parts(ctx->view(), ctx->poff_h[ctx->M], Ns, (int64_t)(kPartsBytes / sizeof(double)), &len);
  DG_CUDA(block_outer_f64(ctx->view(), ctx->blk_row_d, ctx->nnzb, X, ld, X, ld, f, 1.0, Ns, P, len, s));
  return DGCHEFSI_OK;
}
