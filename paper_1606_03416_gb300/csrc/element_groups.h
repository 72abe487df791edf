// Groups of elements for the block-sparse product H X from digits (tc_filter.cu).
// Plain C++ without CUDA.
#pragma once
#include <algorithm>
#include <cstdint>
#include <iterator>
#include <vector>

namespace dg {

// M elements, neighbours of K (itself among them, ascending) at col[row_ptr[K] .. row_ptr[K + 1]).
// Returns the elements of each group, G numbers, -1 for none.
// Groups of G = 2^k elements whose neighbour lists overlap most: singles are
// merged into pairs, pairs into fours and so on, each group (in order) with the
// unmerged one of the same level among its neighbours' that adds the fewest
// neighbours. On a grid of 27-neighbour elements: pairs along x (36 neighbours),
// then 2 x 2 (48, against 54 for four in a row). At most kCandidates are tried,
// more than such a grid has, and one that adds none ends the search: 1200 elements
// that couple to 276 others each, in groups of eight, 12.5 ms; 990 with neither.
inline std::vector<int32_t> group_elements(int M, const int64_t* row_ptr, const int32_t* col, int G) {
  constexpr int kCandidates = 32;
  std::vector<std::vector<int>> elems(M), nbrs(M);
  for (int K = 0; K < M; ++K) {
    elems[K] = {K};
    nbrs[K].assign(col + row_ptr[K], col + row_ptr[K + 1]);
  }
  std::vector<int> owner(M), in_g(M), tried(M);  // in_g, tried: marked with g + 1
  for (int size = 1; size < G; size *= 2) {
    const int n = (int)elems.size();
    for (int g = 0; g < n; ++g)
      for (int K : elems[g])
        if (K >= 0) owner[K] = g;
    std::vector<char> used(n, 0);
    std::fill(in_g.begin(), in_g.end(), 0);
    std::fill(tried.begin(), tried.end(), 0);
    std::vector<std::vector<int>> e2, n2;
    for (int g = 0; g < n; ++g) {
      if (used[g]) continue;
      used[g] = 1;
      for (int K : nbrs[g]) in_g[K] = g + 1;
      int best = -1, candidates = 0;
      size_t fewest = 0;
      for (int K : nbrs[g]) {
        const int h = owner[K];
        if (used[h] || tried[h] == g + 1) continue;
        tried[h] = g + 1;
        size_t added = 0;
        for (int L : nbrs[h]) added += in_g[L] != g + 1;
        if (best < 0 || added < fewest || (added == fewest && h < best)) {
          best = h;
          fewest = added;
        }
        if (fewest == 0 || ++candidates == kCandidates) break;
      }
      std::vector<int> e = elems[g], u = nbrs[g];
      if (best >= 0) {
        used[best] = 1;
        e.resize(size, -1);
        e.insert(e.end(), elems[best].begin(), elems[best].end());
        u.clear();
        std::set_union(nbrs[g].begin(), nbrs[g].end(), nbrs[best].begin(), nbrs[best].end(), std::back_inserter(u));
      }
      e2.push_back(e);
      n2.push_back(u);
    }
    elems.swap(e2);
    nbrs.swap(n2);
  }
  std::vector<int32_t> out;
  for (auto& e : elems) {
    e.resize(G, -1);
    out.insert(out.end(), e.begin(), e.end());
  }
  return out;
}

}  // namespace dg
