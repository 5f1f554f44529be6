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


def _merged_rules(ctx, n_trans, sets, sups):
    """Rules of at least 0 confidence of merged sets, and the divisions they
    stand for."""
    off = np.concatenate([[0], np.cumsum([len(x) for x in sets])]).astype(np.uint64)
    part = (off, np.concatenate(sets).astype(np.uint32), np.asarray(sups, np.uint32))
    fim.fim_merge_results(ctx, n_trans, 1 + int(part[1].max()), [part])
    assert fim.fim_rules(ctx, 0) == sum(2 ** len(x) - 2 for x in sets)
    got = fim.fim_fetch_rules(ctx)
    held = fim.fim_fetch_results(ctx)
    S = held.as_dict()
    conf, lift = [], []
    with np.errstate(divide="ignore", invalid="ignore"):
        for z, mask in zip(got.set_index, got.ante_mask):
            items = held.items[held.offsets[z]:held.offsets[z + 1]]
            x = tuple(int(i) for b, i in enumerate(items) if mask >> b & 1)
            y = tuple(int(i) for b, i in enumerate(items) if not mask >> b & 1)
            sz, sx, sy = (np.float64(v) for v in (S[tuple(items.tolist())], S[x], S[y]))
            conf.append(sz / sx)
            lift.append(sz * n_trans / (sx * sy))
    assert np.array_equal(got.conf, conf, equal_nan=True)
    assert np.array_equal(got.lift, lift, equal_nan=True)
    return got


SETS = [[0], [1], [2], [0, 1], [0, 2], [1, 2], [0, 1, 2]]


def test_ratios_of_zero():
    # a merge for no transactions, and merged sets that occur nowhere
    ctx = fim.fim_create(0)
    try:
        got = _merged_rules(ctx, 0, SETS, [9, 8, 7, 5, 4, 3, 2])
        assert np.all(got.lift == 0) and np.all(got.conf > 0)
        got = _merged_rules(ctx, 100, SETS, [9, 8, 7, 5, 4, 3, 0])
        assert np.count_nonzero(got.conf == 0) == 6 == np.count_nonzero(got.lift == 0)
    finally:
        fim.fim_destroy(ctx)


def test_subsets_of_support_zero_are_held():
    # a held set of support 0 is not a missing one; a missing one still is
    ctx = fim.fim_create(0)
    try:
        got = _merged_rules(ctx, 100, SETS, [9, 0, 7, 0, 4, 0, 0])
        assert np.isnan(got.conf).any()
        _merged_rules(ctx, 100, SETS, [0] * 7)
        with pytest.raises(fim.FimError, match=rf"\({fim.FIM_E_STATE}\)"):
            _merged_rules(ctx, 100, SETS[:1] + SETS[2:], [9, 7, 5, 4, 3, 2])
    finally:
        fim.fim_destroy(ctx)


def test_a_fuller_table_where_memory_is_short():
    # 634,680 sets: a table of 2^21 entries (64 MB), or of 2^20 where only that fits
    from paper_2412_19420_gb300 import datagen
    c = datagen.planted(n=20_000, m=800, n_patterns=60, seed=4)
    got, need = [], []
    for room_mb in (0, 44, 24):
        ctx = fim.fim_create(0)
        try:
            fim.fim_build_bitmaps(ctx, c.indptr, c.indices, c.m)
            fim.fim_mine(ctx, 100)
            sets = len(fim.fim_fetch_results(ctx))
            assert 2 ** 19 < sets < 2 ** 20
            held = fim.fim_get_stats(ctx)["peak_device_bytes"] >> 20
            if room_mb:
                fim.fim_set_tuning(ctx, "test_memory_mb", held + room_mb)
            if room_mb == 24:
                with pytest.raises(fim.FimError, match=rf"\({fim.FIM_E_NOMEM}\)"):
                    fim.fim_rules(ctx, 300_000, 2)
                continue
            fim.fim_rules(ctx, 300_000, 2)
            r = fim.fim_fetch_rules(ctx)
            got.append((r.set_index, r.ante_mask, r.conf.view(np.uint64), r.lift.view(np.uint64)))
            need.append((fim.fim_get_stats(ctx)["peak_device_bytes"] >> 20) - held)
        finally:
            fim.fim_destroy(ctx)
    assert need[0] > 64 and need[1] <= 44
    assert all(np.array_equal(a, b) for a, b in zip(*got))
