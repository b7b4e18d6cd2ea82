"""Work lists of the FP64-class tensor-core products (csrc/ht_units.h) on the CPU: every tile of K exactly once,
and a list's own count of partial sums covers every partial its units write."""
import numpy as np
import pytest

import host_cpp

SOURCE = r"""
#include <cstdio>
#include "ht_units.h"
int main() {
  int T, sms;
  while (std::scanf("%d %d", &T, &sms) == 2)
    for (int sym = 1; sym >= 0; --sym) {
      const kqr::HtList l = sym ? kqr::ht_list_symmetric(T, sms) : kqr::ht_list_rows(T, sms);
      std::printf("%d %d %d %d %zu\n", T, sms, sym, l.parts, l.units.size());
      for (const kqr::HtUnit& u : l.units) std::printf("%d %d %d %d\n", u.tile, u.j0, u.j1, u.part);
    }
}
"""


@pytest.fixture(scope="module")
def lists(tmp_path_factory):
    shapes = [(T, sms) for T in (1, 2, 3, 8, 16, 79, 157, 391) for sms in (1, 132, 152)]
    out = host_cpp.run(SOURCE, tmp_path_factory.mktemp("lists"), "\n".join(f"{T} {s}" for T, s in shapes))
    tok = np.array(out.split(), dtype=np.int64)
    res, at = [], 0
    while at < tok.size:
        T, sms, sym, parts, n = tok[at:at + 5]
        res.append((int(T), int(sms), bool(sym), int(parts), tok[at + 5:at + 5 + 4 * n].reshape(n, 4)))
        at += 5 + 4 * n
    assert len(res) == 2 * len(shapes)
    return res


def test_every_tile_is_worked_once(lists):
    for T, sms, sym, parts, u in lists:
        seen = np.zeros((T, 2 * T), dtype=np.int64)
        for tile, j0, j1, _ in u:
            assert 0 <= j0 < j1 <= 2 * T
            seen[tile, j0:j1] += 1
        want = np.array([[0 if sym and j < 2 * I else 1 for j in range(2 * T)] for I in range(T)])
        np.testing.assert_array_equal(seen, want)


def test_partials_are_counted_by_their_own_list(lists):
    several = 0
    for T, sms, sym, parts, u in lists:
        assert parts == u[:, 3].max() + 1
        if sym:
            assert parts == 1
        else:
            several += parts > 1
            # a partial holds one unit per row tile: the sum over the partials is then the whole row
            for q in range(parts):
                assert sorted(u[u[:, 3] == q, 0]) == list(range(T))
    assert several >= 10   # the rows-only lists of ordinary sizes have more than one partial
