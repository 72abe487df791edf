// FP64 products of the Rayleigh-Ritz step (Alg. 1 steps 3-5: Gram matrix,
// Y U^{-1}, projected H, rotation) emulated on the BF16 tensor cores by exact
// splitting (the Ozaki scheme: Ozaki, Ogita, Oishi, Rump, Numer. Algorithms 59,
// 2012; BF16/FP16 tensor-core form after Mukunoki, Ozaki, Ogita, Imamura,
// ISC 2020).
//
// Over one K chunk of length L <= 4096, row r of A is written as
//   a[r,k] = 2^{e_r} sum_{i<d} q_i[r,k] 2^{-8-9i},  q_i integer, |q_i| <= 256,
// with 2^{e_r} > max_k |a[r,k]| (and likewise each column of the product's
// right operand with exponent f_c). Every q is exact in BF16 (8 significant
// bits hold the integers up to 256), every product q_i q_j is at most 2^16, so
// a slice-pair product summed over 256 terms is an integer of magnitude at
// most 2^24: the tensor core's FP32 accumulation returns it exactly, whatever
// its summation order. The pair kernel (pair_gemm.cu: tcgen05 on pairs of SMs)
// drains its accumulators every 256 terms (more where the digits' norms bound
// the longer sums too) into INT32 sums over the chunk and
// over the pairs of one weight t = i + j. The pairs with t < w are kept (w = d
// or d + 1, weights_for); their INT32 slabs are combined four weights at a time in INT64, the blocks
// meet in FP64, scaled by 2^{e_r + f_c - 16}, and the chunks are added;
// splitting and that reduction are the kernels below.
//
// `slices` s of the callers counts 6-bit digits (60 bits at 10, the splitting
// of one digit per whole 4096-term FP32 sum); digits_for(s) is the number d of
// 9-bit digits that keeps at least as much (10: d = w = 7, 28 pairs).
//
// Error per chunk (row and column maxima m_r, n_c over the chunk): the
// remainders after d digits and the dropped pairs contribute at most
// L 2^{e_r + f_c} 2^{-9d} (d + 2) <= 4 L m_r n_c 2^{-9d} (d + 2), which
// digits_for (digit_rules.h) keeps below L m_r n_c 2^{-6s} (s + 4); the FP64 steps and the sum
// over chunks add at most (5 + chunks) u L m_r n_c, u = 2^{-53}. For s = 10
// (d = 7) the splitting term is below u L m_r n_c, the size of FP64's own
// worst-case bound. The bound is normwise per row and column: entries far
// below their row's maximum keep fewer significant bits than FP64.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <climits>
#include <new>

#include "ctx.h"

namespace dg {

static constexpr int64_t kL = 4096;     // K chunk: one exponent per row and chunk; INT32 holds 7 pairs of it
static constexpr int kNormPitch = 16;  // digit norms of a chunk (at most kMaxDigits)

__device__ __forceinline__ void atomic_flag(int* flag) {
  if (flag) atomicOr(flag, 1);
}

// |x| = M 2^{E - 1075} with M normalised to [2^52, 2^53) (subnormals too).
// Returns 0 for zero, 1 for a finite nonzero x, 2 for NaN/Inf. The frexp
// exponent of x (|x| = f 2^e, f in [0.5, 1)) is E - 1022.
__device__ __forceinline__ int decompose(double x, int64_t& M, int& E) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(x);
  const int Eb = (int)((u >> 52) & 0x7ff);
  const long long m = (long long)(u & 0xfffffffffffffULL);
  if (Eb == 0x7ff) return 2;
  if (Eb == 0) {
    if (m == 0) return 0;
    const int sh = __clzll(m) - 11;  // bring the leading bit to position 52
    M = m << sh;
    E = 1 - sh;
    return 1;
  }
  M = m | (1LL << 52);
  E = Eb;
  return 1;
}

__device__ __forceinline__ int warp_max(int v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// Largest bit pattern of |x[0]| .. |x[n - 1]| (the order of the magnitudes, NaN
// and infinity above the rest), to all 256 threads of the CTA. Four loads of 16
// bytes before their use: a pass over a row waits on memory, not on instructions.
__device__ __forceinline__ unsigned long long cta_max_bits(const double* __restrict__ x, int64_t n) {
  unsigned long long m = 0;
  const auto take = [&](double v) { m = max(m, (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffULL); };
  int64_t c0 = 0;
  if ((reinterpret_cast<uintptr_t>(x) & 15) == 0) {
    const double2* x2 = reinterpret_cast<const double2*>(x);
    for (; c0 + 2048 <= n; c0 += 2048) {
      double2 v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) v[u] = x2[c0 / 2 + threadIdx.x + 256 * u];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        take(v[u].x);
        take(v[u].y);
      }
    }
  }
  for (int64_t c = c0 + threadIdx.x; c < n; c += 256) take(x[c]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  __shared__ unsigned long long red[8];
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < 8; ++w) m = max(m, red[w]);
  return m;
}

// C = 2 or 4 consecutive digits (integers, |f| <= 256) to q as BF16, their squares to *norm
// (HALF: each half of the warp has its own norm).
template <int C, bool HALF>
__device__ __forceinline__ void put_digits(const float (&f)[C], __nv_bfloat16* __restrict__ q, bool store,
                                           uint32_t* norm) {
  uint32_t w[C / 2];
  float sq = 8388608.f;  // 2^23: the low bits of the sum's pattern are the integer sum (below 2^19)
#pragma unroll
  for (int c = 0; c < C; c += 2) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(f[c], f[c + 1]);
    w[c / 2] = *reinterpret_cast<const uint32_t*>(&h);
    sq = fmaf(f[c], f[c], fmaf(f[c + 1], f[c + 1], sq));
  }
  if (store) {
    if (C == 4)
      *reinterpret_cast<uint2*>(q) = make_uint2(w[0], w[C / 2 - 1]);
    else
      *reinterpret_cast<uint32_t*>(q) = w[0];
  }
  const uint32_t mask = HALF ? 0xffffu << (threadIdx.x & 16) : 0xffffffffu;
  const uint32_t sum = __reduce_add_sync(mask, __float_as_uint(sq) & 0x7fffffu);
  if ((threadIdx.x & (HALF ? 15 : 31)) == 0) atomicAdd(norm, sum);
}

// Digits i = 0 .. d - 1 of C consecutive entries v 2^{b} scaled by 2^{-e}
// (|v 2^{b-e}| < 1; zero entries, `zero` and, beside an entry that is not finite,
// entries above that give zero digits), stored at
// q + i * stride where `store`; norm[i] (shared) collects the squares of digit
// i; every lane of the warp takes part. One store per digit.
// d <= 7: F = round(v 2^{9d - 1}) as a 64-bit integer (|F| <= 2^62;
// |v 2^{9d-1} - F| <= 1/2), then its balanced base-512 digits: with 256 added at
// the weight of every digit but the first, digit i + 256 is a 9-bit field of the
// sum and the first digit its rest (|q_0| <= 256). Each field becomes a float by
// its bit pattern (2^23 + field) and one subtraction: a conversion from integer
// would run at a quarter of that rate.
// d > 7 (F would not fit 64 bits): v is scaled in FP64, each digit rounded to
// nearest and subtracted (every step exact).
template <int C, bool HALF = false>
__device__ __forceinline__ void put_all_digits(const double (&v)[C], const int (&b)[C], int e, bool zero, int d,
                                               __nv_bfloat16* __restrict__ q, int64_t stride, bool store,
                                               uint32_t* norm) {
  float f[C];
  if (d <= 7) {
    // 256 (1 + 512 + ... + 512^{d-2})
    const int64_t bias = (int64_t)((0x0040201008040201ULL & ((1ULL << (9 * (d - 1))) - 1)) << 8);
    int64_t F[C];
#pragma unroll
    for (int c = 0; c < C; ++c) {
      int64_t M;
      int E;
      F[c] = bias;
      if (!zero && decompose(v[c], M, E) == 1) {  // |v| = M 2^{E - 1075}, M < 2^53
        // right shift of M 2^10 by r leaves one bit for the rounding; r >= 0 where |v 2^{b-e}| < 1
        const int r = 1075 + e + 10 - E - b[c] - 9 * d;
        const int64_t a = (unsigned)r < 64u ? (int64_t)((((unsigned long long)M << 10) >> r) + 1) >> 1 : 0;
        F[c] += v[c] < 0.0 ? -a : a;
      }
    }
    for (int i = d - 1; i >= 0; --i) {
#pragma unroll
      for (int c = 0; c < C; ++c) {
        const uint32_t lo = (uint32_t)F[c];
        f[c] = i > 0 ? __uint_as_float((lo & 511u) | 0x4B000000u) - 8388864.f  // 2^23 + 256
                     : __uint_as_float((lo + 512u) + 0x4B000000u) - 8389120.f; // the rest, -256 .. 256
        F[c] >>= 9;
      }
      put_digits<C, HALF>(f, q + i * stride, store, norm + i);
    }
  } else {
    double r[C];
#pragma unroll
    for (int c = 0; c < C; ++c) {
      const double y = zero || v[c] == 0.0 ? 0.0 : ldexp(v[c], b[c] - e);
      r[c] = fabs(y) < 1.0 ? y * 256.0 : 0.0;
    }
    for (int i = 0; i < d; ++i) {
#pragma unroll
      for (int c = 0; c < C; ++c) {
        const double g = rint(r[c]);
        r[c] = (r[c] - g) * 512.0;
        f[c] = (float)g;
      }
      put_digits<C, HALF>(f, q + i * stride, store, norm + i);
    }
  }
}

// One CTA per (row, chunk), 256 threads, four groups of four consecutive
// entries each. Q: d digit slices of rows x ldq BF16 (slice i at Q + i *
// sstride; ldq a multiple of 8 and at least K, the entries past K written as
// zero); E[row * nch + chunk] = e_r, the frexp exponent of the row's largest
// |entry| in the chunk (0 if all are zero). lower: entries k > row are zero (a
// lower-triangular operand). bal (may be null): entry k is split as
// X[row, k] 2^{bal[k]}. wide: rows of X start on 16 bytes. A row chunk holding
// NaN/Inf gets zero slices and raises flag. norm2[chunk * kNormPitch + i] is
// raised to the largest sum of squares of digit i over a 512-entry block of
// any row of the chunk (zero before the launch): what lets the pair kernel
// keep its FP32 sums over 512 terms or more instead of 256.
// Bound by HBM: 8 bytes read and 2 d written per entry, in 32- and 8-byte
// pieces per thread (2-byte stores of single entries took twice the time).
constexpr int kSplitThreads = 256;

__global__ void __launch_bounds__(kSplitThreads) k_split_rows(const double* __restrict__ X, int64_t ldx, int64_t K, int d,
                                                    int lower, int wide, const int32_t* __restrict__ bal,
                                                    __nv_bfloat16* __restrict__ Q, int64_t ldq, int64_t sstride,
                                                    int32_t* __restrict__ E, int nch, uint32_t* __restrict__ norm2,
                                                    int* __restrict__ flag) {
  const int64_t row = blockIdx.x;
  const int chunk = blockIdx.y;
  const int64_t k0 = (int64_t)chunk * kL;
  const int64_t kend = lower && row + 1 < K ? row + 1 : K;  // entries from here on are zero
  constexpr int NT = kSplitThreads, NU = 1024 / NT;  // groups of four entries per thread
  double v[NU][4];
  int emax = INT_MIN;
  bool bad = false;
#pragma unroll
  for (int u = 0; u < NU; ++u) {
    const int64_t k = k0 + 4 * (threadIdx.x + NT * u);
    const double* x = X + row * ldx + k;
    if (wide && k + 4 <= kend) {
      const double2 a = *reinterpret_cast<const double2*>(x), b = *reinterpret_cast<const double2*>(x + 2);
      v[u][0] = a.x;
      v[u][1] = a.y;
      v[u][2] = b.x;
      v[u][3] = b.y;
    } else {
#pragma unroll
      for (int c = 0; c < 4; ++c) v[u][c] = k + c < kend ? x[c] : 0.0;
    }
  }
#pragma unroll
  for (int u = 0; u < NU; ++u) {
    const int64_t k = k0 + 4 * (threadIdx.x + NT * u);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      int64_t M;
      int Ex;
      const int z = decompose(v[u][c], M, Ex);
      if (z == 2) bad = true;
      if (z == 1) emax = max(emax, Ex + (bal ? bal[k + c] : 0));
    }
  }
  __shared__ int red[NT / 32];
  __shared__ int sbad;
  __shared__ uint32_t norm[8][kNormPitch];  // by 512-entry block and digit
  if (threadIdx.x == 0) sbad = 0;
  if (threadIdx.x < 8 * kNormPitch) norm[threadIdx.x / kNormPitch][threadIdx.x % kNormPitch] = 0;
  emax = warp_max(emax);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = emax;
  if (bad) sbad = 1;
  __syncthreads();
  emax = red[0];
#pragma unroll
  for (int w = 1; w < NT / 32; ++w) emax = max(emax, red[w]);
  const bool zero = sbad != 0;
  const int e = (emax == INT_MIN || zero) ? 0 : emax - 1022;
  if (threadIdx.x == 0) {
    E[row * nch + chunk] = e;
    if (zero) atomic_flag(flag);
  }
#pragma unroll
  for (int u = 0; u < NU; ++u) {
    const int64_t k = k0 + 4 * (threadIdx.x + NT * u);
    if (k0 + 4 * NT * u >= K) break;  // the same for the whole CTA
    uint32_t* nrm = norm[(threadIdx.x + NT * u) >> 7];
    int b[4] = {0, 0, 0, 0};
    if (bal) {
#pragma unroll
      for (int c = 0; c < 4; ++c)
        if (k + c < K) b[c] = bal[k + c];
    }
    put_all_digits<4>(v[u], b, e, zero, d, Q + row * ldq + k, sstride, k < K, nrm);
  }
  __syncthreads();
  if (threadIdx.x < d) {
    uint32_t m = 0;
#pragma unroll
    for (int b = 0; b < 8; ++b) m = max(m, norm[b][threadIdx.x]);
    atomicMax(norm2 + chunk * kNormPitch + threadIdx.x, m);
  }
}

// bal[k] = frexp exponent of max_c |X[k, c]| (X row-major K x C), 0 for a row
// of zeros or with an entry that is not finite, and nbal[k] = -bal[k]. One CTA per
// row. Bound by HBM: 4096 x 32768 0.16 ms, 6.5 TB/s (0.26 with one 8-byte load at a time).
__global__ void __launch_bounds__(256) k_row_exponents(const double* __restrict__ X, int64_t ldx, int64_t C,
                                                       int32_t* __restrict__ bal, int32_t* __restrict__ nbal) {
  const int64_t k = blockIdx.x;
  const double top = __longlong_as_double((long long)cta_max_bits(X + k * ldx, C));
  if (threadIdx.x == 0) {
    int64_t M;
    int Ex;
    bal[k] = decompose(top, M, Ex) == 1 ? Ex - 1022 : 0;
    nbal[k] = -bal[k];
  }
}

// h 2^e (one rounding, as ldexp; the power of two is built from its bits when
// it is a normal number).
__device__ __forceinline__ double scale_pow2(double h, int e) {
  if (e > -1000 && e < 1000) return h * __longlong_as_double((long long)(e + 1023) << 52);
  return ldexp(h, e);
}

// (hi 2^36 + lo) 2^e, rounded once to nearest even, in integer instructions:
// |hi| 2^36 + |lo| < 2^126. A result below the normal range goes through ldexp.
__device__ __forceinline__ double round_pow2(int64_t hi, int64_t lo, int e) {
  const __int128 v = ((__int128)hi << 36) + lo;
  const bool neg = v < 0;
  const unsigned __int128 u = neg ? -(unsigned __int128)v : (unsigned __int128)v;
  uint64_t uh = (uint64_t)(u >> 64), ul = (uint64_t)u;
  int E = 127 + e;  // exponent of the leading bit
  if (uh == 0) {
    uh = ul;
    ul = 0;
    E -= 64;
  }
  if (uh == 0) return 0.0;
  const int n = __clzll((long long)uh);
  const uint64_t top = n == 0 ? uh : (uh << n) | (ul >> (64 - n));  // leading bit at 63
  E -= n;
  const uint32_t rest = ((uint32_t)top & 0x7ffu) << 1 | ((ul << n) != 0);  // below the last of 53 bits
  const uint64_t m = top >> 11;
  const uint64_t up = rest + ((uint32_t)m & 1u) > 0x800u;
  double y;
  if (E > -1023 && E < 1023)
    y = __longlong_as_double((long long)(((uint64_t)(E + 1022) << 52) + m + up));  // m's leading bit adds the 1
  else
    y = ldexp((double)(m + up), E - 52);
  return neg ? -y : y;
}

// 2^{e + 27} sum_{t < W} 2^{-9t} sum_of(t), |sum_of(t)| < 2^32. Four consecutive t
// are combined in INT64 (the block is below 2^60). Up to W = 8 the two blocks
// meet in 128 bits and the sum is rounded once, all in integer instructions;
// above that the blocks are converted and meet by Horner in 2^{-36}, one
// rounding of each and one per step.
template <int W, class Sums>
__device__ __forceinline__ double digits_to_double(const Sums& sum_of, int e) {
  constexpr int NB = (W + 3) / 4;
  // B_b = sum_{t = 4b}^{4b+3} g_t 2^{9(4b + 3 - t)}; sum_t g_t 2^{-9t} = 2^{-27} sum_b B_b 2^{-36b}
  int64_t B[NB];
#pragma unroll
  for (int b = 0; b < NB; ++b) {
    B[b] = 0;
#pragma unroll
    for (int t = 4 * b; t < 4 * b + 4; ++t) B[b] = B[b] * 512 + (t < W ? sum_of(t) : 0);
  }
  if constexpr (NB <= 2) return round_pow2(B[0], NB == 2 ? B[NB - 1] : 0, e - 36);
  double h = (double)B[NB - 1];
#pragma unroll
  for (int b = NB - 2; b >= 0; --b) h = h * 0x1p-36 + (double)B[b];
  return scale_pow2(h, e);
}

// C[r, n0 + c] (+)= (+-) 2^{e_r + f_{n0+c} - 16} sum_t 2^{-9t} g_t for r < M, c < P,
// g_t the sum of weight t's count[t] INT32 slabs (M rows of `pitch` entries, t
// descending).
// ONE: one slab per weight, all W loads before any use.
// Two consecutive outputs per thread, so a warp's stores are contiguous; wide:
// the rows of C at n0 start on 16 bytes. tri > 0: only the entries with
// n0 + c <= r mod tri are formed (the slice-pair kernel left the tiles above
// that line out); the others are not read or written.
// cmap (may be null): column c goes to column cmap[c] of C and is skipped when
// that is negative (the padding columns of the element-padded layout).
// Bound by HBM: 4 bytes read per slab and entry (28 at w = 7) and 8 written, 16
// when a chunk is added; on products of several chunks it runs on its own stream
// beside the next chunk's pairs. 4096 x 32768, w = 7: 0.84 ms, 5.7 TB/s. With the
// conversions, the Horner step and the scaling on the FP64 pipe (2 a clock and SM,
// about five an entry) 1.26 ms; integers but four outputs a thread (16-byte loads,
// 100 registers) 1.09 ms; two outputs with a division for the row 0.93 ms.
template <int W, bool ONE>
__global__ void __launch_bounds__(256, 4)
    k_digit_reduce(const int32_t* __restrict__ Pw, int64_t M, int64_t P, int64_t pitch, const PairGroups groups,
                   const int32_t* __restrict__ Ea, const int32_t* __restrict__ Eb, int nch, int chunk, int64_t n0,
                   double* __restrict__ C, int64_t ldc, int wide, int accumulate, int negate, int64_t tri,
                   const int32_t* __restrict__ cmap) {
  const int64_t half = M * pitch / 2;
  const uint32_t pairs = (uint32_t)(pitch / 2), stride = gridDim.x * blockDim.x;
  const uint32_t q0 = blockIdx.x * blockDim.x + threadIdx.x;
  // row and column pair of q, carried along: no division per output
  const uint32_t dr = stride / pairs, dc = stride - dr * pairs;
  uint32_t r = q0 / pairs, c = q0 - r * pairs;
  for (int64_t q = q0; q < half; q += stride, r += dr, c += dc) {
    if (c >= pairs) {
      c -= pairs;
      ++r;
    }
    const int64_t c0 = 2 * (int64_t)c;
    // the two entries share a row and a 256-column tile: when the first is
    // above the line both are, and otherwise the tile was computed
    const int64_t rdiag = tri > 0 ? r % (uint32_t)tri : 0;
    if (tri > 0 && n0 + c0 > rdiag) continue;
    const int2* p = reinterpret_cast<const int2*>(Pw) + q;
    const bool second = c0 + 1 < P;
    if (c0 >= P) continue;  // the pitch's padding
    const int er = Ea[(int64_t)r * nch + chunk] - 16 - 27;
    const int ec[2] = {er + Eb[(n0 + c0) * nch + chunk], second ? er + Eb[(n0 + c0 + 1) * nch + chunk] : 0};
    int2 v[ONE ? W : 1];  // one slab per weight: all loads before any use
    int64_t g[2][ONE ? 1 : W];
    if constexpr (ONE) {
#pragma unroll
      for (int t = W - 1; t >= 0; --t, p += half) v[t] = __ldcs(p);
    } else {
#pragma unroll
      for (int t = W - 1; t >= 0; --t) {
        g[0][t] = g[1][t] = 0;
        for (int k = 0; k < groups.count[t]; ++k, p += half) {
          const int2 x = __ldcs(p);
          g[0][t] += x.x;
          g[1][t] += x.y;
        }
      }
    }
    double y[2];
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      y[e] = digits_to_double<W>(
          [&](int t) -> int64_t {
            if constexpr (ONE) return e == 0 ? v[t].x : v[t].y;
            else return g[e][t];
          },
          ec[e]);
      if (negate) y[e] = -y[e];
    }
    if (cmap) {
      const int32_t oc = cmap[c0], od = second ? cmap[c0 + 1] : -1;
      double* o = C + r * ldc + oc;
      if (oc >= 0 && od == oc + 1 && (reinterpret_cast<uintptr_t>(o) & 15) == 0) {
        *reinterpret_cast<double2*>(o) = make_double2(y[0], y[1]);
      } else {
        if (oc >= 0) *o = y[0];
        if (od >= 0) C[r * ldc + od] = y[1];
      }
      continue;
    }
    double* o = C + r * ldc + n0 + c0;
    if (wide && second && (tri == 0 || n0 + c0 + 1 <= rdiag)) {
      if (accumulate) {
        const double2 a = *reinterpret_cast<const double2*>(o);
        y[0] += a.x;
        y[1] += a.y;
      }
      *reinterpret_cast<double2*>(o) = make_double2(y[0], y[1]);
    } else {
      o[0] = accumulate ? o[0] + y[0] : y[0];
      if (second && (tri == 0 || n0 + c0 + 1 <= rdiag)) o[1] = accumulate ? o[1] + y[1] : y[1];
    }
  }
}

typedef void (*DigitReduce)(const int32_t*, int64_t, int64_t, int64_t, const PairGroups, const int32_t*,
                            const int32_t*, int, int, int64_t, double*, int64_t, int, int, int, int64_t,
                            const int32_t*);

// the kernel of w weights; one: one slab per weight
template <bool ONE>
static DigitReduce digit_reduce(int w) {
  switch (w) {
    case 2: return k_digit_reduce<2, ONE>;
    case 3: return k_digit_reduce<3, ONE>;
    case 4: return k_digit_reduce<4, ONE>;
    case 5: return k_digit_reduce<5, ONE>;
    case 6: return k_digit_reduce<6, ONE>;
    case 7: return k_digit_reduce<7, ONE>;
    case 8: return k_digit_reduce<8, ONE>;
    case 9: return k_digit_reduce<9, ONE>;
    case 10: return k_digit_reduce<10, ONE>;
    case 11: return k_digit_reduce<11, ONE>;
    default: return nullptr;
  }
}

static int64_t round_up(int64_t x, int64_t m) { return (x + m - 1) / m * m; }

// Workspace cap of the slabs of the slice-pair products; wider outputs run in column panels.
static constexpr size_t kPairBytes = size_t(8) << 30;

// T (cols x rows, row-major, ldt) = X^T for X (rows x cols, row-major, ldx);
// 32 x 32 tiles through shared memory, 32 x 8 threads.
__global__ void __launch_bounds__(256) k_transpose_f64(const double* __restrict__ X, int64_t ldx, int64_t rows,
                                                       int64_t cols, double* __restrict__ T, int64_t ldt) {
  __shared__ double tile[32][33];
  const int64_t r0 = (int64_t)blockIdx.y * 32, c0 = (int64_t)blockIdx.x * 32;
  for (int j = threadIdx.y; j < 32; j += 8) {
    const int64_t r = r0 + j, c = c0 + threadIdx.x;
    if (r < rows && c < cols) tile[j][threadIdx.x] = X[r * ldx + c];
  }
  __syncthreads();
  for (int j = threadIdx.y; j < 32; j += 8) {
    const int64_t c = c0 + j, r = r0 + threadIdx.x;
    if (r < rows && c < cols) T[c * ldt + r] = tile[threadIdx.x][j];
  }
}

static dgchefsi_status transpose_f64(const double* X, int64_t ldx, int64_t rows, int64_t cols, double* T, int64_t ldt,
                                     cudaStream_t st) {
  if ((rows + 31) / 32 > 65535) return set_error(DGCHEFSI_ERR_UNSUPPORTED, "transpose of %lld rows", (long long)rows);
  k_transpose_f64<<<dim3((unsigned)((cols + 31) / 32), (unsigned)((rows + 31) / 32)), dim3(32, 8), 0, st>>>(
      X, ldx, rows, cols, T, ldt);
  count_launch();
  DG_CUDA(cudaGetLastError());
  return DGCHEFSI_OK;
}

dgchefsi_status sliced_gemm(dgchefsi_ctx* ctx, bool b_rows, bool a_lower, int64_t M, int64_t Nc, int64_t K,
                            const double* A, int64_t lda, const double* B, int64_t ldb, double* C, int64_t ldc,
                            int slices, int* flag, int64_t tri, bool subtract, bool negate) {
  if (M <= 0 || Nc <= 0) return DGCHEFSI_OK;
  if (slices < 2 || slices > 16) return set_error(DGCHEFSI_ERR_ARG, "slices = %d outside 2..16", slices);
  tri = std::min(tri, M);  // r mod tri = r from there on; the reduction's rows and tri are 32-bit numbers
  const int s = digits_for(slices), nw = weights_for(slices);
  cudaStream_t st = ctx->stream;
  if (K <= 0) {
    if (subtract) return DGCHEFSI_OK;
    DG_CUDA(cudaMemset2DAsync(C, sizeof(double) * ldc, 0, sizeof(double) * Nc, M, st));
    return DGCHEFSI_OK;
  }
  const int nch = (int)((K + kL - 1) / kL);
  int nsm = 0;
  DG_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, ctx->device));
  const PairGroups groups = pair_groups(s, nw, ((M + 255) / 256) * ((Nc + 255) / 256), nsm);
  const size_t slab_row = sizeof(int32_t) * (size_t)groups.total * (size_t)M;  // bytes per output column
  // Slices of A: s x M x lqa, of the right operand as rows: s x Nc x lqb (K
  // contiguous in both; the A B form transposes B first).
  const int64_t lqa = round_up(K, 8);
  const int64_t lqb = round_up(K, 8);
  const int64_t sa = M * lqa;
  const int64_t sb = Nc * lqb;
  const bool same = b_rows && A == B && lda == ldb && M == Nc && !a_lower;
  const size_t qa_bytes = sizeof(__nv_bfloat16) * (size_t)(s * sa);
  const size_t qb_bytes = same ? 0 : sizeof(__nv_bfloat16) * (size_t)(s * sb);
  const size_t ea_bytes = sizeof(int32_t) * (size_t)(M * nch);
  const size_t eb_bytes = sizeof(int32_t) * (size_t)(Nc * nch);
  const size_t bal_bytes = b_rows ? 0 : 2 * sizeof(int32_t) * (size_t)K;
  const size_t norm_bytes = 2 * sizeof(uint32_t) * (size_t)(kNormPitch * nch);
  const size_t a256 = 256;
  auto up = [&](size_t x) { return (x + a256 - 1) / a256 * a256; };
  // Column panel of the product (a multiple of the kernel's 256-column tiles)
  // so that the slabs stay under the cap; two slab buffers when the product
  // has more than one (panel, chunk) step, so that the reduction of one step
  // (on the context's reduction stream) overlaps the next step's slice pairs.
  const bool multi = nch > 1 || (int64_t)(kPairBytes / slab_row) < Nc;
  const int nbuf = multi ? 2 : 1;
  int64_t P = std::max<int64_t>(256, (int64_t)(kPairBytes / nbuf / slab_row) / 256 * 256);
  if (P >= Nc) P = Nc;
  const size_t slab_set = slab_row * (size_t)round_up(P, 4);
  const size_t pw_bytes = (size_t)nbuf * up(slab_set);
  DG_TRY(ensure(ctx, ctx->ws_sliced,
                up(qa_bytes) + up(qb_bytes) + up(ea_bytes) + up(eb_bytes) + up(bal_bytes) + up(norm_bytes) + up(pw_bytes),
                "sliced-product workspace"));
  char* base = static_cast<char*>(ctx->ws_sliced.p);
  __nv_bfloat16* Qa = reinterpret_cast<__nv_bfloat16*>(base);
  __nv_bfloat16* Qb = same ? Qa : reinterpret_cast<__nv_bfloat16*>(base + up(qa_bytes));
  int32_t* Ea = reinterpret_cast<int32_t*>(base + up(qa_bytes) + up(qb_bytes));
  int32_t* Eb = same ? Ea : reinterpret_cast<int32_t*>(base + up(qa_bytes) + up(qb_bytes) + up(ea_bytes));
  int32_t* bal = b_rows ? nullptr
                        : reinterpret_cast<int32_t*>(base + up(qa_bytes) + up(qb_bytes) + up(ea_bytes) + up(eb_bytes));
  int32_t* nbal = b_rows ? nullptr : bal + K;
  uint32_t* norm_a =
      reinterpret_cast<uint32_t*>(base + up(qa_bytes) + up(qb_bytes) + up(ea_bytes) + up(eb_bytes) + up(bal_bytes));
  uint32_t* norm_b = same ? norm_a : norm_a + kNormPitch * nch;
  int32_t* Pw = reinterpret_cast<int32_t*>(reinterpret_cast<char*>(norm_a) + up(norm_bytes));
  DG_CUDA(cudaMemsetAsync(norm_a, 0, norm_bytes, st));

  // C = A B with B (K x Nc): every K index k is balanced first, row k of B by
  // 2^{-s_k} and column k of A by 2^{s_k} (exact), s_k the exponent of B's row
  // maximum, so that rows of B with very different norms (the filtered states
  // of Y_hat^T = U^{-T} Y^T) do not share one column scale. B is then
  // transposed (Nc x K) and split by rows like the A B^T form.
  const double* Br = B;
  int64_t ldbr = ldb;
  if (!b_rows) {
    k_row_exponents<<<(unsigned)K, 256, 0, st>>>(B, ldb, Nc, bal, nbal);
    count_launch();
    DG_CUDA(cudaGetLastError());
    DG_TRY(ensure(ctx, ctx->ws_sliced_b, sizeof(double) * (size_t)Nc * (size_t)K, "transposed right operand"));
    double* Bt = static_cast<double*>(ctx->ws_sliced_b.p);
    DG_TRY(transpose_f64(B, ldb, K, Nc, Bt, K, st));
    Br = Bt;
    ldbr = K;
  }
  auto wide = [](const double* p, int64_t ld) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0 && ld % 2 == 0; };
  k_split_rows<<<dim3((unsigned)M, (unsigned)nch), kSplitThreads, 0, st>>>(A, lda, K, s, a_lower ? 1 : 0, wide(A, lda) ? 1 : 0,
                                                                  bal, Qa, lqa, sa, Ea, nch, norm_a, flag);
  count_launch();
  DG_CUDA(cudaGetLastError());
  if (!same) {
    k_split_rows<<<dim3((unsigned)Nc, (unsigned)nch), kSplitThreads, 0, st>>>(Br, ldbr, K, s, 0, wide(Br, ldbr) ? 1 : 0,
                                                                     nbal, Qb, lqb, sb, Eb, nch, norm_b, flag);
    count_launch();
    DG_CUDA(cudaGetLastError());
  }
  if (!ctx->pairs_deferred) DG_TRY(pair_products_begin(ctx));
  cudaStream_t sr = st;
  if (multi) {
    if (!ctx->s_reduce) {
      DG_CUDA(cudaStreamCreateWithFlags(&ctx->s_reduce, cudaStreamNonBlocking));
      for (int i = 0; i < 2; ++i) {
        DG_CUDA(cudaEventCreateWithFlags(&ctx->ev_pairs[i], cudaEventDisableTiming));
        DG_CUDA(cudaEventCreateWithFlags(&ctx->ev_reduce[i], cudaEventDisableTiming));
      }
    }
    sr = ctx->s_reduce;
    // nothing of an earlier call may still read a slab buffer or write C
    DG_CUDA(cudaEventRecord(ctx->ev_pairs[0], st));
    DG_CUDA(cudaStreamWaitEvent(sr, ctx->ev_pairs[0], 0));
    for (int b = 0; b < 2; ++b) DG_CUDA(cudaEventRecord(ctx->ev_reduce[b], sr));
  }
  // timing events around every slice-pair launch (read after the status check)
  const int nsteps = (int)(((Nc + P - 1) / P) * nch);
  while ((int)ctx->ev_time.size() < 2 * nsteps) {
    cudaEvent_t e = nullptr;
    DG_CUDA(cudaEventCreate(&e));
    ctx->ev_time.push_back(e);
  }
  int step = 0;
  for (int64_t n0 = 0; n0 < Nc; n0 += P) {
    const int64_t pn = std::min<int64_t>(P, Nc - n0);
    for (int chunk = 0; chunk < nch; ++chunk, ++step) {
      const int64_t k0 = (int64_t)chunk * kL;
      const int64_t kc = std::min<int64_t>(kL, K - k0);
      const int b = step & 1;
      int32_t* Pb = reinterpret_cast<int32_t*>(reinterpret_cast<char*>(Pw) + (size_t)b * up(slab_set));
      // slabs of the panel: Qa_i times the panel's rows of Qb_j over this chunk, summed per weight,
      // into buffer b once the reduction that last read it is done
      if (multi) DG_CUDA(cudaStreamWaitEvent(st, ctx->ev_reduce[b], 0));
      DG_CUDA(cudaEventRecord(ctx->ev_time[2 * step], st));
      DG_TRY(pair_products_2sm(ctx, Qa, lqa, sa, M, Qb, lqb, sb, Nc, K, k0, kc, n0, pn, s, nw, groups,
                               norm_a + kNormPitch * chunk, norm_b + kNormPitch * chunk, Pb, a_lower, tri));
      DG_CUDA(cudaEventRecord(ctx->ev_time[2 * step + 1], st));
      if (multi) {
        DG_CUDA(cudaEventRecord(ctx->ev_pairs[b], st));
        DG_CUDA(cudaStreamWaitEvent(sr, ctx->ev_pairs[b], 0));
      }
      const int64_t pitch = round_up(pn, 4), work = M * pitch / 2;
      const unsigned grid = (unsigned)std::max<int64_t>(1, std::min<int64_t>((work + 255) / 256, 152 * 16));
      const DigitReduce reduce = groups.total == nw ? digit_reduce<true>(nw) : digit_reduce<false>(nw);
      reduce<<<grid, 256, 0, sr>>>(Pb, M, pn, pitch, groups, Ea, Eb, nch, chunk, n0, C, ldc,
                                wide(C, ldc) ? 1 : 0, subtract || chunk > 0 ? 1 : 0, subtract || negate ? 1 : 0, tri,
                                nullptr);
      count_launch();
      DG_CUDA(cudaGetLastError());
      if (multi) DG_CUDA(cudaEventRecord(ctx->ev_reduce[b], sr));
    }
  }
  if (multi) {  // the caller's stream sees C complete
    DG_CUDA(cudaEventRecord(ctx->ev_reduce[0], sr));
    DG_CUDA(cudaStreamWaitEvent(st, ctx->ev_reduce[0], 0));
  }
  if (ctx->pairs_deferred) return DGCHEFSI_OK;  // the caller asks once for several products
  DG_TRY(pair_products_status(ctx));            // synchronises the stream
  double ms = 0.0;
  for (int q = 0; q < step; ++q) {
    float t = 0.f;
    DG_CUDA(cudaEventElapsedTime(&t, ctx->ev_time[2 * q], ctx->ev_time[2 * q + 1]));
    ms += t;
  }
  ctx->pairs_ms = ms;
  ctx->pairs_launches = step;
  return DGCHEFSI_OK;
}

// ---------------------------------------------------------------------------
// H X from digits (the block-sparse product of Rayleigh-Ritz, W = H Y_hat).
// Row r of H (element K, row n) contracts over the columns of K's neighbour
// blocks only, at most 4096 of them, so one K chunk covers every row: its
// exponent e_r is over the whole row. Each state's exponent f_s is over all N
// of its components (a valid bound for every row's column range). H's digits
// are written in the block layout of the tensor-core filter's operand copy of
// H (64-column slices of each block, element-padded rows), the states' digits
// in its element-padded state-major layout; the pair kernel's block form sums
// each weight's pairs into one INT32 slab and k_digit_reduce (with the
// padded-to-plain column map) combines the slabs.

// E[poff_K + n] = frexp exponent of max_j |H[(K, n), j]| over row n of element
// K's blocks (0 for an all-zero row, and for the padding rows n >= nb[K]).
// One CTA per element. A non-finite entry raises flag.
__global__ void __launch_bounds__(256) k_h_row_exponents(const int64_t* __restrict__ row_ptr,
                                                         const int32_t* __restrict__ col,
                                                         const int64_t* __restrict__ blk_off,
                                                         const double* __restrict__ vals,
                                                         const int32_t* __restrict__ nb,
                                                         const int32_t* __restrict__ pnb,
                                                         const int32_t* __restrict__ poff, int32_t* __restrict__ E,
                                                         int* __restrict__ flag) {
  __shared__ int emax[256];
  __shared__ int bad;
  const int K = blockIdx.x;
  const int nK = nb[K];
  for (int n = threadIdx.x; n < 256; n += blockDim.x) emax[n] = INT_MIN;
  if (threadIdx.x == 0) bad = 0;
  __syncthreads();
  for (int64_t e = row_ptr[K]; e < row_ptr[K + 1]; ++e) {
    const int nKp = nb[col[e]];
    const double* blk = vals + blk_off[e];
    const int64_t total = (int64_t)nK * nKp;
    for (int64_t t = threadIdx.x; t < total; t += blockDim.x) {
      int64_t Mm;
      int Ex;
      const int c = decompose(blk[t], Mm, Ex);
      if (c == 2) bad = 1;
      if (c == 1) atomicMax(&emax[(int)(t / nKp)], Ex);
    }
  }
  __syncthreads();
  for (int n = threadIdx.x; n < pnb[K]; n += blockDim.x)
    E[poff[K] + n] = (n < nK && emax[n] != INT_MIN && !bad) ? emax[n] - 1022 : 0;
  if (threadIdx.x == 0 && bad) atomic_flag(flag);
}

// d digit copies of H in the filter's operand layout: block e, 64-column
// slice sl, padded row n at row brow[e] + sl * pnb[K] + n of each copy (copy i
// starts at Q + i * cstride); entries past the block (padding) are zero. A warp
// per row of 64.
__global__ void __launch_bounds__(256) k_h_digits(const int32_t* __restrict__ blk_row, const int32_t* __restrict__ col,
                                                  const int64_t* __restrict__ blk_off, const double* __restrict__ vals,
                                                  const int32_t* __restrict__ nb, const int32_t* __restrict__ pnb,
                                                  const int32_t* __restrict__ poff, const int64_t* __restrict__ brow,
                                                  const int32_t* __restrict__ E, int d, __nv_bfloat16* __restrict__ Q,
                                                  int64_t cstride, uint32_t* __restrict__ norm2) {
  __shared__ uint32_t norm[8][kNormPitch], top[kNormPitch];
  const int64_t e = blockIdx.x;
  const int K = blk_row[e], Kp = col[e];
  const int nK = nb[K], nKp = nb[Kp], pK = pnb[K];
  const int nsl = (pnb[Kp] + 63) / 64;
  const double* blk = vals + blk_off[e];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x < kNormPitch) top[threadIdx.x] = 0;
  __syncthreads();
  for (int rr = warp; rr < nsl * pK; rr += 8) {
    const int n = rr % pK, jp = (rr / pK) * 64 + 2 * lane;
    const int b[2] = {0, 0};
    double v[2];
#pragma unroll
    for (int c = 0; c < 2; ++c) v[c] = (n < nK && jp + c < nKp) ? blk[(int64_t)n * nKp + jp + c] : 0.0;
    if (lane < kNormPitch) norm[warp][lane] = 0;
    __syncwarp();
    put_all_digits<2>(v, b, E[poff[K] + n], false, d, Q + (brow[e] + rr) * 64 + 2 * lane, cstride, true, norm[warp]);
    __syncwarp();
    if (lane < d) atomicMax(&top[lane], norm[warp][lane]);
    __syncwarp();
  }
  __syncthreads();
  if (threadIdx.x < d) atomicMax(norm2 + threadIdx.x, top[threadIdx.x]);
}

// d digit copies of the states X (Ns x ld, state-major) in the element-padded
// layout (Ns x ldp per copy, copy i at Q + i * cstride); slices[k] = {padded
// column, column, columns, padded columns} of the k-th 64-wide slice. E[s] =
// frexp exponent of the state's largest |entry|. One CTA per state, two passes;
// in the second a half warp takes a slice, four entries a lane.
// 4096 states of 32768: 0.81 ms; 1.65 with a warp per slice and two entries a
// lane, whose reductions, counters and 4-byte stores took the time.
__global__ void __launch_bounds__(256) k_state_digits(const double* __restrict__ X, int64_t ld, int64_t N,
                                                      const int4* __restrict__ slices, int nslices, int64_t ldp, int d,
                                                      __nv_bfloat16* __restrict__ Q, int64_t cstride,
                                                      int32_t* __restrict__ E, uint32_t* __restrict__ norm2,
                                                      int* __restrict__ flag) {
  const int64_t st = blockIdx.x;
  const double* x = X + st * ld;
  __shared__ uint32_t norm[16][kNormPitch], top[kNormPitch];
  if (threadIdx.x < kNormPitch) top[threadIdx.x] = 0;
  int64_t Mm;
  int Ex;
  const int kind = decompose(__longlong_as_double((long long)cta_max_bits(x, N)), Mm, Ex);  // synchronises
  const bool zero = kind == 2;
  const int e = kind == 1 ? Ex - 1022 : 0;
  if (threadIdx.x == 0) {
    E[st] = e;
    if (zero) atomic_flag(flag);
  }
  const int half = threadIdx.x >> 4, l = threadIdx.x & 15;
  for (int k0 = 0; k0 < nslices; k0 += 16) {
    // the last slices: a half warp without one repeats the last and stores nothing
    const int k = min(k0 + half, nslices - 1);
    const int4 sl = slices[k];
    const int j = 4 * l;
    const int b[4] = {0, 0, 0, 0};
    const double* xs = x + sl.y + j;
    double v[4];
    if (j + 4 <= sl.z && (reinterpret_cast<uintptr_t>(xs) & 15) == 0) {
      const double2 a = *reinterpret_cast<const double2*>(xs), c = *reinterpret_cast<const double2*>(xs + 2);
      v[0] = a.x;
      v[1] = a.y;
      v[2] = c.x;
      v[3] = c.y;
    } else {
#pragma unroll
      for (int c = 0; c < 4; ++c) v[c] = j + c < sl.z ? xs[c] : 0.0;
    }
    if (l < kNormPitch) norm[half][l] = 0;
    __syncwarp();
    put_all_digits<4, true>(v, b, e, zero, d, Q + st * ldp + sl.x + j, cstride, j < sl.w && k0 + half < nslices,
                            norm[half]);
    __syncwarp();
    if (l < d) atomicMax(&top[l], norm[half][l]);
    __syncwarp();
  }
  __syncthreads();
  if (threadIdx.x < d) atomicMax(norm2 + threadIdx.x, top[threadIdx.x]);
}

cudaError_t digits_of_h(const dgchefsi_ctx* ctx, const int32_t* blk_row, const int32_t* pnb, const int32_t* poff,
                        const int64_t* brow, int d, __nv_bfloat16* Q, int64_t cstride, int32_t* E, uint32_t* norm2,
                        int* flag, cudaStream_t st) {
  k_h_row_exponents<<<(unsigned)ctx->M, 256, 0, st>>>(ctx->row_ptr_d, ctx->col_d, ctx->blk_off_d, ctx->vals_d,
                                                      ctx->nb_d, pnb, poff, E, flag);
  count_launch();
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_h_digits<<<(unsigned)ctx->nnzb, 256, 0, st>>>(blk_row, ctx->col_d, ctx->blk_off_d, ctx->vals_d, ctx->nb_d, pnb,
                                                  poff, brow, E, d, Q, cstride, norm2);
  count_launch();
  return cudaGetLastError();
}

cudaError_t digits_of_states(const double* X, int64_t ld, int64_t Ns, int64_t N, const int4* slices, int nslices,
                             int64_t ldp, int d, __nv_bfloat16* Q, int64_t cstride, int32_t* E, uint32_t* norm2,
                             int* flag, cudaStream_t st) {
  k_state_digits<<<(unsigned)Ns, 256, 0, st>>>(X, ld, N, slices, nslices, ldp, d, Q, cstride, E, norm2, flag);
  count_launch();
  return cudaGetLastError();
}

dgchefsi_status reduce_digit_slabs(const int32_t* Pw, int64_t rows, int64_t cols, int w, const PairGroups& groups,
                                   const int32_t* Erows, const int32_t* Ecols, const int32_t* cmap, double* C,
                                   int64_t ldc, cudaStream_t st) {
  const unsigned grid = (unsigned)std::max<int64_t>(1, std::min<int64_t>((rows * cols / 2 + 255) / 256, 152 * 16));
  const DigitReduce reduce = groups.total == w ? digit_reduce<true>(w) : digit_reduce<false>(w);
  reduce<<<grid, 256, 0, st>>>(Pw, rows, cols, cols, groups, Erows, Ecols, 1, 0, 0, C, ldc, 0, 0, 0, 0, cmap);
  count_launch();
  DG_CUDA(cudaGetLastError());
  return DGCHEFSI_OK;
}

// ---------------------------------------------------------------------------
// The density blocks P_K = sum_i f_i x_i x_i^T (f >= 0) from digits: the rows of
// Z = (sqrt(f_i) x_i)^T are packed into 256-row tiles, whole elements one after
// another, and the pair kernel multiplies each tile with itself only. Bound by
// HBM: per row and state 16 bytes for Z, 8 + 14 for its digits and the pairs'
// reads of them (a tile's digits serve that tile only). FP64 tiles do n + 1
// operations there (the rule is in density_digits_fit).
// 8 x 8 x 8 elements of 64, 4096 states: 9.66 ms on the FP64 cores; here 0.44 for
// Z, 0.67 for the digits, 1.55 for the pairs, 0.04 for the blocks. Largest error
// against 64-bit mantissas, relative to sqrt(P_jj P_j'j'): 1.0e-16, FP64 1.9e-15.

// Zt[p, i] = sf[i] X[i, col[p]], 0 where col[p] < 0; 32 x 32 tiles, 32 x 8 threads.
__global__ void __launch_bounds__(256) k_density_rows(const double* __restrict__ X, int64_t ldx, int64_t Ns,
                                                      const int32_t* __restrict__ col, const double* __restrict__ sf,
                                                      double* __restrict__ Zt, int64_t ldz) {
  __shared__ double tile[32][33];
  const int64_t p0 = (int64_t)blockIdx.x * 32, i0 = (int64_t)blockIdx.y * 32;
  const int32_t c = col[p0 + threadIdx.x];
  for (int j = threadIdx.y; j < 32; j += 8) {
    const int64_t i = i0 + j;
    tile[j][threadIdx.x] = i < Ns && c >= 0 ? X[i * ldx + c] * sf[i] : 0.0;
  }
  __syncthreads();
  for (int j = threadIdx.y; j < 32; j += 8)
    if (i0 + threadIdx.x < ldz) Zt[(p0 + j) * ldz + i0 + threadIdx.x] = tile[threadIdx.x][j];
}

__global__ void k_sqrt(const double* __restrict__ f, int64_t n, double* __restrict__ out) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = sqrt(f[i]);
}

// P_K (+)= element K's block of its tile's slabs (rows x 256 each): its rows and
// columns start at row prow[K] of the packed rows. blockIdx.x: element.
template <int W>
__global__ void __launch_bounds__(256) k_density_reduce(const int32_t* __restrict__ nb, const int64_t* __restrict__ poff,
                                                        const int32_t* __restrict__ prow,
                                                        const int32_t* __restrict__ Pw, int64_t rows,
                                                        const PairGroups groups, const int32_t* __restrict__ E, int nch,
                                                        int chunk, double* __restrict__ P) {
  const int K = blockIdx.x, n = nb[K], r0 = prow[K], c0 = r0 & 255;
  double* out = P + poff[K];
  for (int q = blockIdx.y * 256 + threadIdx.x; q < n * n; q += 256 * gridDim.y) {
    const int j = q / n, jp = q - j * n;
    const int32_t* p = Pw + (int64_t)(r0 + j) * 256 + c0 + jp;
    int64_t g[W];
#pragma unroll
    for (int t = W - 1; t >= 0; --t) {
      g[t] = 0;
      for (int k = 0; k < groups.count[t]; ++k, p += rows * 256) g[t] += *p;
    }
    const int e = E[(int64_t)(r0 + j) * nch + chunk] + E[(int64_t)(r0 + jp) * nch + chunk] - 16 - 27;
    const double y = digits_to_double<W>([&](int t) -> int64_t { return g[t]; }, e);
    out[q] = chunk > 0 ? out[q] + y : y;
  }
}

typedef void (*DensityReduce)(const int32_t*, const int64_t*, const int32_t*, const int32_t*, int64_t, const PairGroups,
                              const int32_t*, int, int, double*);

static DensityReduce density_reduce(int w) {
  switch (w) {
    case 7: return k_density_reduce<7>;
    case 8: return k_density_reduce<8>;
    case 9: return k_density_reduce<9>;
    case 10: return k_density_reduce<10>;
    case 11: return k_density_reduce<11>;
    default: return nullptr;
  }
}

// Elements in order, each whole in one 256-row tile; rows of Z in all.
static int64_t pack_density_rows(const dgchefsi_ctx* ctx, std::vector<int32_t>* prow) {
  int64_t r = 0;
  for (int K = 0; K < ctx->M; ++K) {
    const int n = ctx->nb_h[K];
    if (r / 256 != (r + n - 1) / 256) r = round_up(r, 256);
    if (prow) (*prow)[K] = (int32_t)r;
    r += n;
  }
  return round_up(r, 256);
}

bool density_digits_fit(const dgchefsi_ctx* ctx, int64_t Ns) {
  int64_t sq = 0;
  for (int K = 0; K < ctx->M; ++K) {
    if (ctx->nb_h[K] > 256) return false;
    sq += (int64_t)ctx->nb_h[K] * ctx->nb_h[K];
  }
  const int64_t rows = pack_density_rows(ctx, nullptr);
  // Both forms per row of Z and state: n + 1 FP64 operations, or some 50 bytes and
  // 28 pairs of a 256-wide row whatever n is. Kernel time, FP64 and digits, us:
  // n = 8, 1.4 M row-states 77 / 75; n = 16, 8.2 M 338 / 248; n = 40, 0.8 M 67 / 90;
  // n = 64, 4.1 M 431 / 145; n = 40..120, 20 M 2040 / 590; n = 64, 134 M 9660 / 2700.
  return rows < 1 << 30 && Ns < 1 << 20 && sq >= 16 * rows && rows * Ns >= 1 << 21;
}

dgchefsi_status density_digits(dgchefsi_ctx* ctx, const double* X, int64_t Ns, int64_t ld, const double* f, double* P,
                               bool* done) {
  *done = false;
  const int slices = std::max(ctx->products_slices, 10), s = digits_for(slices), nw = weights_for(slices);
  cudaStream_t st = ctx->stream;
  const DensityReduce reduce = density_reduce(nw);
  if (!reduce) return DGCHEFSI_OK;
  const int64_t max_nb = ctx->view().max_nb;
  std::vector<int32_t> prow, col;
  int64_t rows = 0;
  try {
    prow.resize(ctx->M);
    rows = pack_density_rows(ctx, &prow);
    col.assign(rows, -1);
  } catch (const std::bad_alloc&) {
    return DGCHEFSI_OK;
  }
  const int nch = (int)((Ns + kL - 1) / kL);
  const int64_t ldz = round_up(Ns, 2), lq = round_up(Ns, 8), sq = rows * lq;
  int nsm = 0;
  DG_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, ctx->device));
  const PairGroups groups = pair_groups(s, nw, rows / 256, nsm);
  auto up = [](size_t x) { return (x + 255) / 256 * 256; };
  const size_t q_bytes = up(sizeof(__nv_bfloat16) * (size_t)(s * sq)), e_bytes = up(sizeof(int32_t) * (size_t)(rows * nch));
  const size_t n_bytes = up(sizeof(uint32_t) * (size_t)(kNormPitch * nch) + sizeof(int));
  const size_t c_bytes = up(sizeof(int32_t) * (size_t)rows), k_bytes = up(sizeof(int32_t) * (size_t)ctx->M);
  const size_t s_bytes = up(sizeof(double) * (size_t)Ns);
  const size_t w_bytes = sizeof(int32_t) * (size_t)groups.total * (size_t)rows * 256;
  // the buffers of the rotation before it, larger only where the packing pads; without the memory, the FP64 form
  if (ensure(ctx, ctx->ws_sliced_b, sizeof(double) * (size_t)(rows * ldz), "density rows") != DGCHEFSI_OK ||
      ensure(ctx, ctx->ws_sliced, q_bytes + e_bytes + n_bytes + c_bytes + k_bytes + s_bytes + w_bytes,
             "density digits") != DGCHEFSI_OK) {
    clear_error();
    return DGCHEFSI_OK;
  }
  char* at = static_cast<char*>(ctx->ws_sliced.p);
  auto take = [&](size_t bytes) { char* p = at; at += bytes; return p; };
  __nv_bfloat16* Q = reinterpret_cast<__nv_bfloat16*>(take(q_bytes));
  int32_t* E = reinterpret_cast<int32_t*>(take(e_bytes));
  uint32_t* norm = reinterpret_cast<uint32_t*>(take(n_bytes));
  int* flag = reinterpret_cast<int*>(norm + kNormPitch * nch);
  int32_t* col_d = reinterpret_cast<int32_t*>(take(c_bytes));
  int32_t* prow_d = reinterpret_cast<int32_t*>(take(k_bytes));
  double* sf = reinterpret_cast<double*>(take(s_bytes));
  int32_t* Pw = reinterpret_cast<int32_t*>(at);
  double* Zt = static_cast<double*>(ctx->ws_sliced_b.p);
  for (int K = 0; K < ctx->M; ++K)
    for (int j = 0; j < ctx->nb_h[K]; ++j) col[prow[K] + j] = (int32_t)(ctx->off_h[K] + j);
  DG_CUDA(cudaMemcpyAsync(col_d, col.data(), sizeof(int32_t) * (size_t)rows, cudaMemcpyHostToDevice, st));
  DG_CUDA(cudaMemcpyAsync(prow_d, prow.data(), sizeof(int32_t) * (size_t)ctx->M, cudaMemcpyHostToDevice, st));
  DG_CUDA(cudaMemsetAsync(norm, 0, n_bytes, st));
  k_sqrt<<<(unsigned)((Ns + 255) / 256), 256, 0, st>>>(f, Ns, sf);
  k_density_rows<<<dim3((unsigned)(rows / 32), (unsigned)((Ns + 31) / 32)), dim3(32, 8), 0, st>>>(X, ld, Ns, col_d, sf,
                                                                                              Zt, ldz);
  k_split_rows<<<dim3((unsigned)rows, (unsigned)nch), kSplitThreads, 0, st>>>(Zt, ldz, Ns, s, 0, 1, nullptr, Q, lq, sq, E,
                                                                              nch, norm, flag);
  count_launch(3);
  DG_CUDA(cudaGetLastError());
  DG_TRY(pair_products_begin(ctx));
  const unsigned ctas = (unsigned)((max_nb * max_nb + 1023) / 1024);  // four entries a thread
  for (int chunk = 0; chunk < nch; ++chunk) {
    const int64_t k0 = (int64_t)chunk * kL, kc = std::min<int64_t>(kL, Ns - k0);
    DG_TRY(pair_products_diag(ctx, Q, lq, sq, rows, Ns, k0, kc, s, nw, groups, norm + kNormPitch * chunk, Pw));
    reduce<<<dim3((unsigned)ctx->M, ctas), 256, 0, st>>>(ctx->nb_d, ctx->poff_d, prow_d, Pw, rows, groups, E, nch, chunk, P);
    count_launch();
    DG_CUDA(cudaGetLastError());
  }
  int bad = 0;  // a state or an occupation that is not finite: the FP64 form spreads it as it did
  DG_CUDA(cudaMemcpyAsync(&bad, flag, sizeof(int), cudaMemcpyDeviceToHost, st));
  DG_TRY(pair_products_status(ctx));  // synchronises the stream
  *done = bad == 0;
  return DGCHEFSI_OK;
}

dgchefsi_status sliced_gemm_tn(dgchefsi_ctx* ctx, int64_t M, int64_t Nc, int64_t K, const double* A, int64_t lda,
                               const double* B, int64_t ldb, double* C, int64_t ldc, int s, int* flag) {
  if (M <= 0 || Nc <= 0) return DGCHEFSI_OK;
  if (K > 0) {
    DG_TRY(ensure(ctx, ctx->ws_sliced_t, sizeof(double) * (size_t)M * (size_t)K, "transposed operand"));
    double* At = static_cast<double*>(ctx->ws_sliced_t.p);
    DG_TRY(transpose_f64(A, lda, K, M, At, K, ctx->stream));
    return sliced_gemm(ctx, false, false, M, Nc, K, At, K, B, ldb, C, ldc, s, flag);
  }
  return sliced_gemm(ctx, false, false, M, Nc, K, A, lda, B, ldb, C, ldc, s, flag);
}

void sliced_destroy(dgchefsi_ctx* ctx) { (void)ctx; }

}  // namespace dg
