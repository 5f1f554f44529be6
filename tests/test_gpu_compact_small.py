"""The one-CTA compaction of small outputs: canonical at the edges of its sort
(powers of two of sets, the largest it takes and one more), with one and
several key words, and for merged parts, which keep the caller's ids."""
import numpy as np
import pytest

import oracle
from paper_2412_19420_gb300 import datagen

pytestmark = pytest.mark.gpu
fim = pytest.importorskip("paper_2412_19420_gb300.fim")


@pytest.fixture(scope="module")
def ctx():
    c = fim.fim_create(0)
    yield c
    fim.fim_destroy(c)


# single items only: exactly `sets` itemsets
@pytest.mark.parametrize("sets", [1, 2, 63, 64, 65, 127, 511, 512, 513, 1023, 1024, 1025])
def test_set_counts(ctx, sets):
    rng = np.random.default_rng(sets)
    rows = [[int(x)] for x in rng.permutation(sets)] * 2
    c = datagen.from_lists(rows, sets)
    fim.fim_build_bitmaps(ctx, c.indptr, c.indices, c.m)
    fim.fim_mine(ctx, 2)
    got = fim.fim_fetch_results(ctx)
    assert len(got) == sets
    assert got.sha256() == oracle.apriori(c.indptr, c.indices, c.m, 2).sha256()


# longest sets of 3 .. 13 items out of up to 60,000 ids: one to four key words,
# sets that fit the local copy and sets that do not (their subsets then exceed
# one CTA and take the other compaction)
@pytest.mark.parametrize("length,m", [(3, 100), (7, 200), (8, 60_000), (9, 60_000), (10, 60_000), (11, 2_000)])
def test_key_words(ctx, length, m):
    rng = np.random.default_rng(length)
    ids = rng.choice(m, size=length, replace=False)
    rows = [[int(i) for i in ids]] * 3 + [[int(i)] for i in rng.choice(m, size=40)] * 3
    c = datagen.from_lists(rows, m)
    fim.fim_build_bitmaps(ctx, c.indptr, c.indices, c.m)
    for on in (1, 0):
        fim.fim_set_tuning(ctx, "compact_cluster", on)
        try:
            fim.fim_mine(ctx, 3)
            assert fim.fim_fetch_results(ctx).sha256() == oracle.apriori(c.indptr, c.indices, c.m, 3).sha256()
        finally:
            fim.fim_set_tuning(ctx, "compact_cluster", 1)


def test_long_sets_in_a_merge(ctx):
    # sets longer than the local copy, one CTA's worth of them
    off, items = [0], []
    sets = [list(range(k, k + n)) for n, k in ((1, 3), (12, 0), (13, 5), (20, 1), (20, 2))]
    for x in sets:
        items += x
        off.append(len(items))
    part = (np.array(off, np.uint64), np.array(items, np.uint32), np.arange(9, 4, -1).astype(np.uint32))
    fim.fim_merge_results(ctx, 100, 40, [part])
    assert fim.fim_fetch_results(ctx).as_dict() == {tuple(x): 9 - i for i, x in enumerate(sets)}


def test_merged_parts(ctx):
    c = datagen.zipf_baskets(4_000, 90, 0.9, 6.0, 1)
    want = oracle.apriori(c.indptr, c.indices, c.m, 40)
    fim.fim_build_bitmaps(ctx, c.indptr, c.indices, c.m)
    parts = []
    for s in range(3):
        fim.fim_mine_shard(ctx, 40, 0, s, 3)
        parts.append(fim.fim_fetch_results(ctx))
    fim.fim_merge_results(ctx, c.n, c.m, parts)
    assert len(want) <= 1024 and fim.fim_fetch_results(ctx).sha256() == want.sha256()


def test_large_outputs_radix(ctx):
    # the digit launches: outputs around their tile sizes (2,048 and 4,096
    # records), many tiles, several key words, and records with holes
    cases = [(datagen.planted(n=20_000, m=800, n_patterns=60, seed=4), 100),     # 400,000 sets, 3 words
             (datagen.planted(n=20_000, m=800, n_patterns=60, seed=4), 240),
             (datagen.random_dense(2_000, 22, 0.6, 4), 60),                      # 1 to 2 words, ~130,000 sets
             (datagen.from_lists([list(range(17))] * 5, 17), 5)]                 # 2^17 - 1 sets, all of one support
    fim.fim_set_tuning(ctx, "compact_cluster", 0)
    try:
        for c, thr in cases:
            want = oracle.apriori(c.indptr, c.indices, c.m, thr)
            fim.fim_build_bitmaps(ctx, c.indptr, c.indices, c.m)
            for _ in range(3):  # direct launches, the capture, the replayed graph
                fim.fim_mine(ctx, thr)
                assert fim.fim_fetch_results(ctx).sha256() == want.sha256(), (c.n, len(want))
        for sets in (2047, 2048, 2049, 4095, 4096, 4097, 12_289):
            c = datagen.from_lists([[i] for i in range(sets)], sets)
            fim.fim_build_bitmaps(ctx, c.indptr, c.indices, c.m)
            fim.fim_mine(ctx, 1)
            assert fim.fim_fetch_results(ctx).sha256() == oracle.apriori(c.indptr, c.indices, c.m, 1).sha256()
    finally:
        fim.fim_set_tuning(ctx, "compact_cluster", 1)
