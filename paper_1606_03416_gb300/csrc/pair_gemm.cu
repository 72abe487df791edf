// Slice-pair products of the FP64-from-BF16-slices GEMM (the Ozaki scheme of
// sliced.cu; Alg. 1 steps 3-5) on pairs of SMs: tcgen05 with cta_group::2.
//
// The digits of a slice are integers of magnitude at most 256 (9 bits, exact
// in BF16), so a product summed over 256 terms is an integer of magnitude at
// most 2^24: the tensor core's FP32 accumulation returns it exactly. The
// accumulator is drained every 256 terms (four 64-wide K slices), or every 512
// to 4096 where the digits' norms say that no partial sum can pass 2^24 there
// (Cauchy-Schwarz; the splitting kernel leaves the largest norms; digits of
// Gaussian-like entries allow 512, pairs with a leading digit 1024 and more),
// and the sums go on in INT32 registers of the epilogue warps, over the whole 4096-long K
// chunk and over all pairs (i, j) of one weight t = i + j (up to 7 pairs:
// 7 * 2^16 * 4096 < 2^31). So one INT32 slab per weight leaves the kernel
// where one FP32 slab per pair would with an accumulator that had to hold the
// whole chunk (6-bit digits: 10 slices, 55 pairs and 55 slabs for the 60 bits
// that 7 slices, 28 pairs and 7 slabs give here).
//
// One CTA pair (a cluster of two) computes a 256 x 256 tile of one weight at
// a time: each CTA stages its own 128 rows of A_i and its own 128 rows of B_j
// (32 KB per 64-wide K slice), the first CTA of the pair issues
// 256 x 256 x 16 MMAs that read both CTAs' halves, and each CTA's tensor
// memory holds its 128 rows of the tile. Per SM that is 8 KB of operands per
// 128-clock MMA, half of what a single-SM 128 x 256 tile reads, which leaves
// shared-memory bandwidth for the TMA refills. The kernel is persistent over
// (weight group, tile) units, the tiles of one group back to back and the
// largest groups first, so that the units in flight read the same slices from
// L2 and the last wave is of the shortest units; the tensor maps of all slices
// sit in device memory, so one launch covers every pair of a chunk.
//
// What bounds it: the tensor pipe (32 MMAs = 4096 clocks per 512 terms). The
// drain of those 128 x 256 sums runs beside the next terms in the other
// accumulator: ~2150 clocks, because the float-to-int conversion runs at 16 per
// clock and SM; the extra commit and the hand-over cost the tensor pipe a few
// hundred clocks each, so the fewer the better. Tensor rate of the 28 pairs at
// 4096^2 x 16384: 990 TFLOP/s with 256 terms per accumulator (the drain sets
// the time), 1510 with 512, 1660 with the norms' choice for Gaussian entries,
// 1710 without any drain: 9.3 ms, where 55 pairs of 6-bit digits took ~16.
//
// BLOCKS = true multiplies the block-sparse H: the A rows of a tile are the H
// rows of a group of elements (four of up to 64 functions, two per CTA), its K
// slices the group's neighbour list, its B rows states. Elements that do not
// couple to a slice's element multiply a zero tile there, 21 of 48 slices for a
// 2 x 2 x 1 group of a 27-point stencil.
//
// Roles per CTA (576 threads): warp 0 lane 0 loads its halves with TMA into a
// 6-slot ring and signals the first CTA's "full" barrier (its expect-tx counts
// both CTAs' bytes); warp 1 lane 0 of the first CTA issues the MMAs, frees
// ring slots in both CTAs and announces finished accumulators to both
// (multicast commits); warps 2-17 drain their CTA's accumulator
// (double-buffered, 2 x 256 columns; 64 columns of 32 rows each) and report to
// the first CTA's "empty" accumulator barrier. Every wait is bounded; on
// expiry the CTA records an error word and both CTAs still meet at the final
// cluster barrier.
#include <algorithm>
#include <cstring>
#include <vector>

#include "tc_kernel.cuh"

namespace dg {
namespace {

constexpr int PG_EPI_WARPS = 16;
constexpr int PG_THREADS = 32 * (2 + PG_EPI_WARPS);
constexpr int PG_HALF = 128 * SLICE_BYTES;  // 128 rows x 64 BF16 of one operand
constexpr int PG_STAGE = 2 * PG_HALF;       // A half + B half per CTA
constexpr int PG_STAGES = 6;

struct PairJob {
  const CUtensorMap* maps;  // device, 64-byte aligned: [s] maps of A_i, then [s] maps of B_j
  const int32_t* group;     // [ngroups + 1] first pair of each group; a group's pairs have one weight i + j
  const int32_t* pair_i;    // [npairs], in group order
  const int32_t* pair_j;
  int ngroups, s;
  int64_t M;        // rows of A (the slab's rows)
  int64_t pitch;    // row pitch of the slab, a multiple of 4
  int n0, k0, nk;   // first B row, first K column, 64-wide K slices of the chunk
  int nmt, nnt;     // 256-row tiles along M and along the panel
  int lower;        // A is lower triangular: a row tile stops at the chunk's last K slice it reaches
  int diag;         // > 0: the B rows of row tile mt start at 256 mt (nnt = 1, slabs of 256 columns);
                    // 2: the units of one tile back to back, not those of one group
  const int2* tiles;  // null: every (row tile, column tile); else the ntl tiles to compute
  int ntl;
  const uint32_t* norm_a;  // [s] largest sum of squares of digit i over 512 terms of a row of A, of B
  const uint32_t* norm_b;
  int32_t* Pw;      // slab of group g at Pw + g * M * pitch, row-major M x pitch
  int* err;
  // Block-sparse form (BLOCKS): the A rows of a tile are the H rows of 2 G2
  // stacked elements, acc rows each (G2 = 128 / acc per CTA), its K slices the
  // entries of their group's schedule (the padded state column and each
  // element's first operand row, a zero tile where it does not couple), its B
  // rows states; the slabs are (states x padded H rows).
  const int32_t* sched;      // entries of 1 + 2 G2 numbers
  const int32_t* sched_ptr;  // [nmt + 1]
  const int32_t* grp_elem;   // [nmt * 2 G2], -1 past the end
  const int32_t* pnb;        // padded size and offset of each element
  const int32_t* poff;
  int G2, acc;
  int sched_in_smem;  // a unit's schedule is copied to shared memory; else read where it is
};

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}

__device__ __forceinline__ uint32_t map_to_rank(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}

__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__device__ __forceinline__ void arrive_remote(uint32_t cluster_addr) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}

// Adds one to a shared-memory counter; returns its old value. Orders what the
// warps before it did before what the last one does next.
__device__ __forceinline__ uint32_t count_acq_rel(uint32_t* p) {
  uint32_t old;
  asm volatile("atom.acq_rel.cta.shared::cta.add.u32 %0, [%1], 1;" : "=r"(old) : "r"(smem_u32(p)) : "memory");
  return old;
}

// TMA load into this CTA's shared memory, completing on a barrier that may sit
// in the peer CTA of the pair.
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap* map, int x, int y, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], "
      "[%4];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar)
      : "memory");
}

__device__ __forceinline__ void mma_bf16_pair(uint32_t d, uint64_t a, uint64_t b, uint32_t id, uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
      "l"(a), "l"(b), "r"(id), "r"(acc)
      : "memory");
}

// Arrive on the barrier at this offset in both CTAs of the pair once the MMAs
// issued so far have completed.
__device__ __forceinline__ void commit_pair(uint32_t bar) {
  const uint16_t mask = 3;
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar),
      "h"(mask)
      : "memory");
}

// Group and tile of work unit u: groups outermost, the tiles of one group back
// to back (row tiles fastest), so the units in flight walk the same pairs and
// share their slices in L2.
__device__ __forceinline__ void unit_of(const PairJob& J, int64_t u, int& g, int& mt, int& nt) {
  if (J.tiles) {
    g = (int)(u / J.ntl);
    const int2 t = J.tiles[u - (int64_t)g * J.ntl];
    mt = t.x;
    nt = t.y;
    return;
  }
  const int64_t ntiles = (int64_t)J.nmt * J.nnt;
  if (J.diag == 2) {
    mt = (int)(u / J.ngroups);
    g = (int)(u - (int64_t)mt * J.ngroups);
    nt = 0;
    return;
  }
  g = (int)(u / ntiles);
  const int64_t tile = u - (int64_t)g * ntiles;
  mt = (int)(tile % J.nmt);
  nt = (int)(tile / J.nmt);
}

// The k-th unit of cluster cid: forwards and backwards in turn, so that every
// cluster gets long and short units alike (units come longest first).
__device__ __forceinline__ int64_t nth_unit(int64_t k, int cid, int ncl) {
  return k * ncl + ((k & 1) ? ncl - 1 - cid : cid);
}

// K slices that row tile mt needs: all of the chunk's, or for a lower
// triangular A those up to its last row (at least one, so that the tile's
// accumulator is written); the entries of its schedule in the block form.
template <bool BLOCKS>
__device__ __forceinline__ int slices_of_tile(const PairJob& J, int mt) {
  if (BLOCKS) return J.sched_ptr[mt + 1] - J.sched_ptr[mt];
  if (!J.lower) return J.nk;
  const int need = (mt * 256 + 256 - J.k0 + 63) / 64;
  return max(1, min(J.nk, need));
}

template <bool BLOCKS>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(PG_THREADS, 1) k_slice_pairs_2sm(const PairJob J) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + PG_STAGES * PG_STAGE);
  int32_t* sched_sh = reinterpret_cast<int32_t*>(bars + 2 * PG_STAGES + 4);  // BLOCKS: the unit's schedule (producer)
  __shared__ uint32_t tmem_base_sh;
  __shared__ int abort_sh;
  __shared__ uint32_t drained_sh[2];       // epilogue warps done with their part, over all uses of a buffer
  __shared__ int drain_sh[kMaxPairs];    // K slices per accumulator of each pair

  const uint32_t rank = cluster_rank();
  const bool leader = rank == 0;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int cid = blockIdx.x >> 1, ncl = gridDim.x >> 1;
  const int64_t nunits = (J.tiles ? (int64_t)J.ntl : (int64_t)J.nmt * J.nnt) * J.ngroups;
  const uint32_t full0 = smem_u32(bars), empty0 = full0 + 8 * PG_STAGES;
  const uint32_t accf0 = empty0 + 8 * PG_STAGES, acce0 = accf0 + 16;

  if (threadIdx.x == 0) {
    for (int s = 0; s < PG_STAGES; ++s) {
      mbar_init(full0 + 8 * s, 1);
      mbar_init(empty0 + 8 * s, 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(accf0 + 8 * b, 1);
      mbar_init(acce0 + 8 * b, 2);  // the last epilogue warp of each CTA
    }
    abort_sh = 0;
    drained_sh[0] = drained_sh[1] = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {  // both CTAs allocate the same columns together
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_sh)),
                 "r"(512)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  for (int p = threadIdx.x; p < J.group[J.ngroups]; p += PG_THREADS)
    drain_sh[p] = drain_slices((uint64_t)J.norm_a[J.pair_i[p]] * J.norm_b[J.pair_j[p]], BLOCKS);
  tc_fence_before();
  __syncthreads();
  cluster_sync();  // barriers of both CTAs initialised before any remote use
  tc_fence_after();
  const uint32_t tmem = tmem_base_sh;

  if (warp == 0) {
    // ---------------- producer: this CTA's halves, completing on the first CTA's barrier
    const uint32_t full_l = map_to_rank(full0, 0);
    const int ent = 1 + 2 * J.G2;
    int c = 0;
    bool ok = true;
    for (int64_t k = 0, u; (u = nth_unit(k, cid, ncl)) < nunits && ok; ++k) {
      int g, mt, nt;
      unit_of(J, u, g, mt, nt);
      const int ya = mt * 256 + (int)rank * 128;
      const int yb = J.n0 + (J.diag ? mt : nt) * 256 + (int)rank * 128;
      const int nk = slices_of_tile<BLOCKS>(J, mt);
      const int32_t* sched = nullptr;
      if (BLOCKS) {
        sched = J.sched + (int64_t)J.sched_ptr[mt] * ent;
        if (J.sched_in_smem) {
          __syncwarp();
          for (int t = lane; t < nk * ent; t += 32) sched_sh[t] = sched[t];
          __syncwarp();
          sched = sched_sh;
        }
      }
      if (lane == 0) {
        for (int p = J.group[g]; p < J.group[g + 1] && ok; ++p) {
          const CUtensorMap* am = J.maps + J.pair_i[p];
          const CUtensorMap* bm = J.maps + J.s + J.pair_j[p];
          for (int ks = 0; ks < nk; ++ks) {
            const int st = c % PG_STAGES;
            const uint32_t ph = (uint32_t)(c / PG_STAGES) & 1u;
            if (!mbar_wait(empty0 + 8 * st, ph ^ 1u)) {
              ok = false;
              break;
            }
            if (leader) mbar_expect_tx(full0 + 8 * st, (uint32_t)(2 * PG_STAGE));
            const uint32_t dst = smem_u32(smem + st * PG_STAGE);
            if (BLOCKS) {
              const int32_t* e = sched + ks * ent;
              for (int q = 0; q < J.G2; ++q)
                tma_load_2d_pair(dst + q * J.acc * SLICE_BYTES, am, 0, e[1 + rank * J.G2 + q], full_l + 8 * st);
              tma_load_2d_pair(dst + PG_HALF, bm, e[0], yb, full_l + 8 * st);
            } else {
              const int x = J.k0 + ks * (SLICE_BYTES / 2);
              tma_load_2d_pair(dst, am, x, ya, full_l + 8 * st);
              tma_load_2d_pair(dst + PG_HALF, bm, x, yb, full_l + 8 * st);
            }
            ++c;
          }
        }
      }
      if (BLOCKS) ok = __shfl_sync(0xffffffffu, (int)ok, 0) != 0;
    }
    if (!ok && lane == 0) {
      atomicOr(J.err, 1);
      atomicExch(&abort_sh, 1);
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer: the first CTA of the pair only
    if (leader && lane == 0) {
      constexpr uint32_t ID = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(256 >> 3) << 17) |
                              ((uint32_t)(256 >> 4) << 24);
      const uint64_t desc0 = sdesc(smem_u32(smem));
      int c = 0, i = 0;  // ring slots and accumulators used so far
      bool ok = true;
      for (int64_t k = 0, u; (u = nth_unit(k, cid, ncl)) < nunits && ok; ++k) {
        int g, mt, nt_;
        unit_of(J, u, g, mt, nt_);
        const int nk = slices_of_tile<BLOCKS>(J, mt);
        for (int p = J.group[g], k0 = 0, len = drain_sh[p]; p < J.group[g + 1] && ok; ++i) {
          const int buf = i & 1;
          const uint32_t use = (uint32_t)(i >> 1);
          if (!mbar_wait(acce0 + 8 * buf, (use & 1u) ^ 1u)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t d = tmem + (uint32_t)(buf * 256);
          const int k1 = min(k0 + len, nk);
          for (int ks = k0; ks < k1; ++ks) {
            const int st = c % PG_STAGES;
            const uint32_t ph = (uint32_t)(c / PG_STAGES) & 1u;
            if (!mbar_wait(full0 + 8 * st, ph)) {
              ok = false;
              break;
            }
            tc_fence_after();
            const uint64_t da = desc0 + (uint64_t)((st * PG_STAGE) >> 4);
            const uint64_t db = da + (uint64_t)(PG_HALF >> 4);
#pragma unroll
            for (int kk = 0; kk < SLICE_BYTES / 32; ++kk)
              mma_bf16_pair(d, da + (uint64_t)((32 * kk) >> 4), db + (uint64_t)((32 * kk) >> 4), ID,
                            (ks > k0 || kk > 0) ? 1u : 0u);
            commit_pair(empty0 + 8 * st);
            ++c;
          }
          if (ok) commit_pair(accf0 + 8 * buf);
          k0 = k1;
          if (k0 == nk) {  // an accumulator holds terms of one pair only
            k0 = 0;
            if (++p < J.group[g + 1]) len = drain_sh[p];
          }
        }
      }
      if (!ok) {
        atomicOr(J.err, 1);
        atomicExch(&abort_sh, 1);
      }
    }
  } else {
    // ---------------- epilogue: warps 2..17, lane quarter q = tile rows 32q..32q+31 of this
    // CTA's half, columns 64h..64h+63; the running sums stay in registers for the whole unit
    const int q = warp & 3;
    const int h = (warp - 2) >> 2;
    const uint32_t acce_l = map_to_rank(acce0, 0);
    int i = 0;
    bool ready = true;
    for (int64_t n = 0, u; (u = nth_unit(n, cid, ncl)) < nunits && ready; ++n) {
      int g, mt, nt;
      unit_of(J, u, g, mt, nt);
      const int nk = slices_of_tile<BLOCKS>(J, mt);
      int ndrain = 0;
      for (int p = J.group[g]; p < J.group[g + 1]; ++p) ndrain += (nk + drain_sh[p] - 1) / drain_sh[p];
      int sum[64];
#pragma unroll
      for (int z = 0; z < 64; ++z) sum[z] = 0;
      for (int k = 0; k < ndrain; ++k, ++i) {
        const int buf = i & 1;
        const uint32_t use = (uint32_t)(i >> 1);
        ready = mbar_wait(accf0 + 8 * buf, use & 1u);
        ready = __all_sync(0xffffffffu, ready);
        if (!ready) {
          if (lane == 0) atomicOr(J.err, 1);
          break;
        }
        tc_fence_after();
        const uint32_t ta = tmem + (uint32_t)(buf * 256 + 64 * h) + ((uint32_t)(32 * q) << 16);
#pragma unroll
        for (int cc = 0; cc < 4; ++cc) {
          float v[16];
          tmem_ld16(ta + (uint32_t)(16 * cc), v);
          if (cc == 3) {  // this warp's last read: the CTA's last warp to get here frees the accumulator
            tc_fence_before();
            __syncwarp();
            if (lane == 0 && count_acq_rel(&drained_sh[buf]) == PG_EPI_WARPS * (use + 1) - 1)
              arrive_remote(acce_l + 8 * buf);
          }
#pragma unroll
          for (int z = 0; z < 16; ++z) sum[16 * cc + z] += __float2int_rn(v[z]);
        }
      }
      if (!ready || *(volatile int*)&abort_sh != 0) continue;
      int32_t* slab = J.Pw + (size_t)g * (size_t)J.M * (size_t)J.pitch;
      const int64_t c0 = (int64_t)nt * 256 + 64 * h;
      if (BLOCKS) {  // thread = H row, register = state: consecutive rows of one state are consecutive in the slab
        const int local = 32 * q + lane, n = local % J.acc;
        const int K = J.grp_elem[((int64_t)mt * 2 + rank) * J.G2 + local / J.acc];
        if (K < 0 || n >= J.pnb[K]) continue;
        int32_t* out = slab + J.poff[K] + n;
#pragma unroll
        for (int z = 0; z < 64; ++z)
          if (c0 + z < J.M) out[(c0 + z) * J.pitch] = sum[z];
      } else {
        const int64_t r = (int64_t)mt * 256 + rank * 128 + 32 * q + lane;
        if (r >= J.M) continue;
        int32_t* out = slab + (size_t)r * (size_t)J.pitch;
#pragma unroll
        for (int z = 0; z < 64; z += 4)  // pitch % 4 == 0: every vector is inside the row or past it
          if (c0 + z < J.pitch)
            *reinterpret_cast<int4*>(out + c0 + z) = make_int4(sum[z], sum[z + 1], sum[z + 2], sum[z + 3]);
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync();  // neither CTA leaves while the pair's MMAs or arrivals may still touch it
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
  }
}

PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  if (!fn) {
    void* ptr = nullptr;
    cudaDriverEntryPointQueryResult qr;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &ptr, 12000, cudaEnableDefault, &qr) ==
            cudaSuccess &&
        qr == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(ptr);
  }
  return fn;
}

// BF16 matrix rows x inner (row stride `stride` elements), boxes of 64 x box_rows, 128-byte swizzle.
dgchefsi_status slice_map(CUtensorMap* map, const __nv_bfloat16* base, uint64_t inner, uint64_t rows,
                          uint64_t stride, uint32_t box_rows = 128) {
  auto enc = tensor_map_encoder();
  if (!enc) return set_error(DGCHEFSI_ERR_CUDA, "cuTensorMapEncodeTiled unavailable");
  cuuint64_t dims[2] = {inner, rows};
  cuuint64_t strides[1] = {stride * 2};
  cuuint32_t box[2] = {64, box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<__nv_bfloat16*>(base), dims, strides, box,
                   estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return set_error(DGCHEFSI_ERR_CUDA, "cuTensorMapEncodeTiled failed (%d)", (int)r);
  return DGCHEFSI_OK;
}

}  // namespace

// Tables of a launch in one host block: 2s tensor maps (64-byte aligned), then
// the groups (slab order: weights t descending, each weight's pairs in count[t]
// groups of nearly equal size) and their pairs, then the tile list.
struct PairTables {
  std::vector<uint8_t> host;
  CUtensorMap* maps = nullptr;
  size_t maps_bytes = 0, tiles_at = 0;
  int npairs = 0;

  PairTables(int s, int nw, const PairGroups& groups, size_t ntiles) {
    for (int t = 0; t < nw; ++t) npairs += pairs_of_weight(s, t);
    const int ng = groups.total;
    maps_bytes = sizeof(CUtensorMap) * (size_t)(2 * s);
    tiles_at = (maps_bytes + sizeof(int32_t) * (size_t)(ng + 1 + 2 * npairs) + 15) / 16 * 16;
    host.resize(tiles_at + sizeof(int2) * ntiles);
    maps = reinterpret_cast<CUtensorMap*>(host.data());
    int32_t* gp = reinterpret_cast<int32_t*>(host.data() + maps_bytes);
    int32_t* pi = gp + ng + 1;
    int32_t* pj = pi + npairs;
    int n = 0, g = 0;
    for (int t = nw - 1; t >= 0; --t) {
      const int np = pairs_of_weight(s, t), i0 = std::max(0, t - s + 1);
      for (int q = 0, k = 0; q < groups.count[t]; ++q) {
        gp[g++] = n;
        for (const int end = group_end(np, q, groups.count[t]); k < end; ++k, ++n) {
          pi[n] = i0 + k;
          pj[n] = t - i0 - k;
        }
      }
    }
    gp[g] = n;
  }
};

// Copies the tables to the device, fills what every launch shares and starts the kernel.
static dgchefsi_status launch_pairs(dgchefsi_ctx* ctx, PairJob& J, const PairTables& T, int s, const PairGroups& groups,
                                    bool blocks, int64_t tiles, int sched_bytes) {
  // the context's table buffer (may be regrown here: it holds no state across launches)
  DevBuf& tables = ctx->ws_pairs;
  DG_TRY(ensure(ctx, tables, T.host.size(), "slice-pair tensor maps"));
  uint8_t* tab = static_cast<uint8_t*>(tables.p);
  // the pageable copy has been staged before it returns, so the host block may go
  DG_CUDA(cudaMemcpyAsync(tab, T.host.data(), T.host.size(), cudaMemcpyHostToDevice, ctx->stream));
  J.maps = reinterpret_cast<const CUtensorMap*>(tab);
  J.group = reinterpret_cast<const int32_t*>(tab + T.maps_bytes);
  J.pair_i = J.group + groups.total + 1;
  J.pair_j = J.pair_i + T.npairs;
  J.ngroups = groups.total;
  J.s = s;
  J.tiles = J.ntl > 0 ? reinterpret_cast<const int2*>(tab + T.tiles_at) : nullptr;
  if (!ctx->ws_pairs_err.p) return set_error(DGCHEFSI_ERR_CUDA, "slice-pair products not begun");
  J.err = static_cast<int*>(ctx->ws_pairs_err.p);
  int nsm = 0;
  DG_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, ctx->device));
  const int clusters = (int)std::min<int64_t>(tiles * groups.total, std::max(nsm / 2, 1));
  const int smem = PG_STAGES * PG_STAGE + (2 * PG_STAGES + 4) * 8 + 1024 + sched_bytes;
  auto kern = blocks ? k_slice_pairs_2sm<true> : k_slice_pairs_2sm<false>;
  DG_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
  kern<<<2 * clusters, PG_THREADS, smem, ctx->stream>>>(J);
  count_launch();
  DG_CUDA(cudaGetLastError());
  return DGCHEFSI_OK;
}

dgchefsi_status pair_products_2sm(dgchefsi_ctx* ctx, const __nv_bfloat16* Qa, int64_t lqa, int64_t sa, int64_t M,
                                  const __nv_bfloat16* Qb, int64_t lqb, int64_t sb, int64_t Nc, int64_t K, int64_t k0,
                                  int64_t kc, int64_t n0, int64_t pn, int s, int nw, const PairGroups& groups,
                                  const uint32_t* norm_a, const uint32_t* norm_b, int32_t* Pw, bool a_lower, int64_t tri) {
  if (M > 2147483647LL - 256 || Nc > 2147483647LL - 256 || K > 2147483647LL)
    return set_error(DGCHEFSI_ERR_UNSUPPORTED, "slice-pair product too large for 32-bit TMA coordinates");
  const int nmt = (int)((M + 255) / 256), nnt = (int)((pn + 255) / 256);
  // tri > 0: only entries (r, n0 + c) with n0 + c <= r mod tri are wanted (the
  // lower triangle of a symmetric product, or of each of several stacked
  // ones); tiles entirely above it are left out.
  std::vector<int2> tl;
  if (tri > 0) {
    for (int nt = 0; nt < nnt; ++nt)
      for (int mt = 0; mt < nmt; ++mt) {
        const int64_t r0 = (int64_t)mt * 256, r1 = std::min<int64_t>(r0 + 256, M) - 1;
        const int64_t c0 = n0 + (int64_t)nt * 256;
        const bool wrap = r0 / tri != r1 / tri;
        if (wrap || c0 <= r1 % tri) tl.push_back(make_int2(mt, nt));
      }
    if (tl.empty()) return DGCHEFSI_OK;
  }
  PairTables T(s, nw, groups, tl.size());
  for (int i = 0; i < s; ++i) {
    DG_TRY(slice_map(&T.maps[i], Qa + (size_t)i * sa, (uint64_t)K, (uint64_t)M, (uint64_t)lqa));
    DG_TRY(slice_map(&T.maps[s + i], Qb + (size_t)i * sb, (uint64_t)K, (uint64_t)Nc, (uint64_t)lqb));
  }
  if (!tl.empty()) std::memcpy(T.host.data() + T.tiles_at, tl.data(), sizeof(int2) * tl.size());
  PairJob J{};
  J.M = M;
  J.pitch = (pn + 3) / 4 * 4;
  J.n0 = (int)n0;
  J.k0 = (int)k0;
  J.nk = (int)((kc + 63) / 64);
  J.nmt = nmt;
  J.nnt = nnt;
  J.lower = a_lower ? 1 : 0;
  J.norm_a = norm_a;
  J.norm_b = norm_b;
  J.ntl = (int)tl.size();
  J.Pw = Pw;
  return launch_pairs(ctx, J, T, s, groups, false, tl.empty() ? (int64_t)nmt * nnt : (int64_t)tl.size(), 0);
}

dgchefsi_status pair_products_diag(dgchefsi_ctx* ctx, const __nv_bfloat16* Q, int64_t lq, int64_t sq, int64_t rows,
                                   int64_t K, int64_t k0, int64_t kc, int s, int nw, const PairGroups& groups,
                                   const uint32_t* norm, int32_t* Pw) {
  if (rows > 2147483647LL - 256 || K > 2147483647LL)
    return set_error(DGCHEFSI_ERR_UNSUPPORTED, "slice-pair product too large for 32-bit TMA coordinates");
  PairTables T(s, nw, groups, 0);
  for (int i = 0; i < s; ++i) {
    DG_TRY(slice_map(&T.maps[i], Q + (size_t)i * sq, (uint64_t)K, (uint64_t)rows, (uint64_t)lq));
    T.maps[s + i] = T.maps[i];
  }
  PairJob J{};
  J.M = rows;
  J.pitch = 256;
  J.k0 = (int)k0;
  J.nk = (int)((kc + 63) / 64);
  J.nmt = (int)((rows + 255) / 256);
  J.nnt = 1;
  // A tile's digits are read by its own units only. While the chunk's digits fit
  // L2 a few times over, the order by groups (longest first) has the shorter last
  // wave: 36 tiles of 1001 terms (129 MB) 114 us, 165 by tiles. Above that a
  // tile's units run side by side and share its reads: 128 tiles of 4096 terms
  // (3.8 GB) 2.00 -> 1.55 ms, 64 of 2000 (459 MB) 0.48 -> 0.39, 25 of 4096
  // (367 MB) 0.37 -> 0.35, 39 of 2000 (280 MB) 0.32 by groups, 0.34 by tiles.
  J.diag = 2 * (double)rows * (double)kc * s > 320e6 ? 2 : 1;
  J.norm_a = norm;
  J.norm_b = norm;
  J.Pw = Pw;
  return launch_pairs(ctx, J, T, s, groups, false, J.nmt, 0);
}

dgchefsi_status pair_products_blocks(dgchefsi_ctx* ctx, const BlockPairs& B, int64_t s0, int64_t pn, int32_t* Pw) {
  PairTables T(B.s, B.nw, B.groups, 0);
  for (int i = 0; i < B.s; ++i) {
    DG_TRY(slice_map(&T.maps[i], B.Hs + (size_t)i * B.hcopy, 64, (uint64_t)B.h_rows, 64, (uint32_t)B.acc));
    DG_TRY(slice_map(&T.maps[B.s + i], B.Xs + (size_t)i * B.xcopy, (uint64_t)B.ldp, (uint64_t)B.Ns, (uint64_t)B.ldp));
  }
  PairJob J{};
  J.M = pn;
  J.pitch = B.ldp;
  J.n0 = (int)s0;
  J.nmt = B.ngroups;
  J.nnt = (int)((pn + 255) / 256);
  J.norm_a = B.norm_h;
  J.norm_b = B.norm_x;
  J.Pw = Pw;
  J.sched = B.sched;
  J.sched_ptr = B.sched_ptr;
  J.grp_elem = B.grp_elem;
  J.pnb = B.pnb;
  J.poff = B.poff;
  J.G2 = 128 / B.acc;
  J.acc = B.acc;
  // a schedule longer than what the ring leaves (930 entries of groups of 8 elements) stays in global memory
  int64_t sched_bytes = (int64_t)B.maxent * (1 + 2 * J.G2) * (int64_t)sizeof(int32_t);
  J.sched_in_smem = PG_STAGES * PG_STAGE + (2 * PG_STAGES + 4) * 8 + 1024 + sched_bytes <= 226 * 1024 ? 1 : 0;
  if (!J.sched_in_smem) sched_bytes = 0;
  return launch_pairs(ctx, J, T, B.s, B.groups, true, (int64_t)J.nmt * J.nnt, (int)sched_bytes);
}

dgchefsi_status pair_products_begin(dgchefsi_ctx* ctx) {
  DG_TRY(ensure(ctx, ctx->ws_pairs_err, 256, "slice-pair error word"));
  DG_CUDA(cudaMemsetAsync(ctx->ws_pairs_err.p, 0, sizeof(int), ctx->stream));
  return DGCHEFSI_OK;
}

dgchefsi_status pair_products_status(dgchefsi_ctx* ctx) {
  if (!ctx->ws_pairs_err.p) return DGCHEFSI_OK;
  int err = 0;
  DG_CUDA(cudaMemcpyAsync(&err, ctx->ws_pairs_err.p, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream));
  DG_CUDA(cudaStreamSynchronize(ctx->stream));
  if (err) return set_error(DGCHEFSI_ERR_TIMEOUT, "a slice-pair CTA gave up waiting on a pipeline barrier");
  return DGCHEFSI_OK;
}

}  // namespace dg
