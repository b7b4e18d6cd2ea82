// Work lists of the FP64-class tensor-core products (gram_high_tc.cu).  Plain C++ without CUDA, so
// that the lists can be checked on a machine without a GPU.
#pragma once
#include <stdint.h>

#include <algorithm>
#include <vector>

namespace kqr {

// Row tile (128 rows), first and end 64-column tile, and the partial sums the unit writes.
struct HtUnit {
  int tile, j0, j1, part;
};

// A list carries its own number of partial sums: it sizes the buffer the units write to, and the sum
// over the partials runs to it.
struct HtList {
  std::vector<HtUnit> units;
  int parts = 0;
};

// One vector, T row tiles: (I, run of 64-column tiles from the diagonal on), about 8 per SM but no
// shorter than 16 tiles while an SM gets that many (a unit's set-up, table and tile I, costs about one
// tile), longest first.  All units add to one set of sums.
inline HtList ht_list_symmetric(int T, int num_sms) {
  HtList l;
  const int TJ = 2 * T;
  int64_t tiles = 0;
  for (int I = 0; I < T; ++I) tiles += TJ - 2 * I;
  const int64_t C = std::max<int64_t>(1, (tiles + (int64_t)8 * num_sms - 1) / ((int64_t)8 * num_sms));
  const int C1 = (int)std::max<int64_t>(C, std::min<int64_t>(16, (tiles + num_sms - 1) / num_sms));
  for (int I = 0; I < T; ++I)
    for (int j = 2 * I; j < TJ; j += C1) l.units.push_back({I, j, std::min(TJ, j + C1), 0});
  std::stable_sort(l.units.begin(), l.units.end(),
                   [](const HtUnit& a, const HtUnit& b) { return a.j1 - a.j0 > b.j1 - b.j0; });
  l.parts = 1;
  return l;
}

// Several vectors: (I, split) with about 8 units per SM; each split's row sums are a partial of their
// own, added in a fixed order.
inline HtList ht_list_rows(int T, int num_sms) {
  HtList l;
  const int TJ = 2 * T;
  const int64_t want = ((int64_t)8 * num_sms + T - 1) / T;
  const int per = (int)std::max<int64_t>(std::min<int64_t>(8, (TJ * (int64_t)T + num_sms - 1) / num_sms),
                                         (TJ + want - 1) / want);
  l.parts = (TJ + per - 1) / per;
  for (int s = 0; s < l.parts; ++s)
    for (int I = 0; I < T; ++I) l.units.push_back({I, s * per, std::min(TJ, (s + 1) * per), s});
  return l;
}

}  // namespace kqr
