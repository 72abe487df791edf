// Rules of the digits that FP64 products are rebuilt from (sliced.cu,
// pair_gemm.cu): how many, which pairs, in which sums, drained how often. Plain
// C++; the last rule also runs in the pair kernel.
#pragma once
#include <algorithm>
#include <cstdint>

#ifdef __CUDACC__
#define DG_HOST_DEVICE __host__ __device__
#else
#define DG_HOST_DEVICE
#endif

namespace dg {

// For a request of s 6-bit slices (2 <= s <= 16): the number of 9-bit digits,
// 9 d >= 6 s + 1, so that their remainders are below those of the slices; and
// the number of weights t = i + j kept, w >= d. w is d, or d + 1 where integer
// operands that s slices multiply exactly need it to stay exact: operands of a
// and b slices, a + b <= s + 1, have at most 6 (a + b) bits between them (53
// when the result is representable) and ceil((bits + 1) / 9) digits each, and
// the pair of their last digits is kept when those counts sum to at most w + 1.
constexpr int kMaxDigits = 11;
constexpr int kMaxPairs = 66;  // 11 digits, all weights
inline int digits_for(int s) { return (6 * s + 9) / 9; }
inline int weights_for(int s) {
  const int bits = std::min(6 * (s + 1), 53);
  return std::min(std::max(digits_for(s), (bits + 18) / 9 - 1), std::max(s, digits_for(s)));
}

// Pairs (i, t - i) of weight t with both digits below d.
inline int pairs_of_weight(int d, int t) { return std::max(0, std::min(t, d - 1) - std::max(0, t - d + 1) + 1); }

// Slabs of the digit weights.
struct PairGroups {
  uint8_t count[16];  // by weight t
  int total;
};

// Most pairs of one INT32 sum: each adds at most 4096 terms of 2^16, 2^28.
constexpr int kGroupPairs = 7;

// How many slabs each weight is split into for an output of so many 256 x 256
// tiles. Pairs per unit: all of a weight, at most kGroupPairs, when there are many
// units for the clusters; fewer when a small output would leave clusters idle or
// waiting for the longest unit.
inline PairGroups pair_groups(int d, int w, int64_t tiles, int nsm) {
  const int64_t clusters = std::max(nsm / 2, 1);
  int64_t pairs = 0;
  for (int t = 0; t < w; ++t) pairs += pairs_of_weight(d, t);
  const int64_t avg = (pairs * tiles + clusters - 1) / clusters;
  const int cap = (int)std::min<int64_t>(kGroupPairs, std::max<int64_t>(1, (avg + 1) / 2));
  PairGroups g{};
  for (int t = 0; t < w; ++t) {
    g.count[t] = (uint8_t)((pairs_of_weight(d, t) + cap - 1) / cap);
    g.total += g.count[t];
  }
  return g;
}

// End of the q-th of `count` groups of np pairs, nearly equal in size.
inline int group_end(int np, int q, int count) { return np * (q + 1) / count; }

// 64-wide K slices that a pair's FP32 accumulator sums before it is drained, sq
// the product of the two digits' largest norms. Four (256 terms of at most 2^16 are
// at most 2^24) at least. More where Cauchy-Schwarz says that no sum passes 2^24:
// norms over aligned 512-term blocks give |a||b| for such a block and 2^h |a||b| for
// 2^h of them; norms over one slice (per_slice) len |a||b| for len of them.
constexpr int kDrain = 4;
DG_HOST_DEVICE inline int drain_slices(uint64_t sq, bool per_slice) {
  int len = kDrain;
  if (per_slice) {
    while (len < 64 && (uint64_t)((len + 1) * (len + 1)) * sq <= 1ull << 48) ++len;
  } else {
    for (int h = 0; h < 4 && sq <= 1ull << (48 - 2 * h); ++h) len *= 2;
  }
  return len;
}

}  // namespace dg
