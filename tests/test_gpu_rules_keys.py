"""GPU association rules at the edges of the set table's keys vs the oracle.

A subset of k items is its own key while k times the width of the largest id
fits 127 bits; longer subsets are hashed and their items compared.  The sizes
put every long set on both sides of that line, and 10-item sets have 1,022
candidates, so they straddle the 1,024-candidate chunks and half of their
complements lie in another chunk.  Rules, confidence and lift must match bit
for bit: both sides divide the same integers once, correctly rounded.
"""
import numpy as np
import pytest

import oracle
from oracle import rules as orules

pytestmark = pytest.mark.gpu

fim = pytest.importorskip("paper_2412_19420_gb300.fim")


@pytest.mark.parametrize("m,n,k", [(12, 300, 10), (1000, 4000, 10), (1024, 2000, 11), (50_000, 1500, 9),
                                   (50_000, 70_000, 10)])
def test_rules_of_long_sets(m, n, k):
    rng = np.random.default_rng(m + n)
    # two groups of k ids, the largest id among them; a row holds most of one
    top = np.sort(rng.permutation(m - 1)[:k - 1])
    groups = [np.append(top, m - 1), np.sort(rng.permutation(m)[:k])]
    rows = []
    for _ in range(n):
        g = groups[int(rng.random() < 0.5)]
        rows.append(np.unique(np.append(g[rng.random(k) < 0.93], rng.integers(0, m, 1))))
    indptr = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int64)
    indices = np.concatenate(rows).astype(np.int32)
    minsup = n // 8
    want = orules.rules(oracle.apriori(indptr, indices, m, minsup), n, 600_000, 0)
    ctx = fim.fim_create(0)
    try:
        fim.fim_build_bitmaps(ctx, indptr, indices, m)
        fim.fim_mine(ctx, minsup)
        assert fim.fim_rules(ctx, 600_000, 0) == len(want)
        got = fim.fim_fetch_rules(ctx)
    finally:
        fim.fim_destroy(ctx)
    assert len(want) > (1 << k) - 2
    assert np.array_equal(got.set_index, want.set_index)
    assert np.array_equal(got.ante_mask, want.ante_mask)
    assert np.array_equal(got.conf.view(np.uint64), want.conf.view(np.uint64))
    assert np.array_equal(got.lift.view(np.uint64), want.lift.view(np.uint64))
