"""The prefix extension's three ways (CTAs on bit columns, warps on projected
columns, warps on bit columns) give the oracle's itemsets wherever one of them
is chosen or forced, and the choice follows the matrix."""
import numpy as np
import pytest

import oracle
from paper_2412_19420_gb300 import datagen

pytestmark = pytest.mark.gpu
fim = pytest.importorskip("paper_2412_19420_gb300.fim")

CTAS, PROJECTED, COLUMNS = 0, 1, 2


@pytest.fixture(scope="module")
def ctx():
    c = fim.fim_create(0)
    yield c
    fim.fim_destroy(c)


def _words(ctx, c, minsup, way=-1, flags=0):
    """The itemsets' hash and the words of the search's columns: the projected
    ways count fewer."""
    fim.fim_set_tuning(ctx, "dfs_proj", way)
    try:
        fim.fim_build_bitmaps(ctx, c.indptr, c.indices, c.m)
        fim.fim_mine(ctx, minsup, flags)
        st = fim.fim_get_stats(ctx)
        return fim.fim_fetch_results(ctx).sha256(), st["dfs_words"], st["dfs_workers"]
    finally:
        fim.fim_set_tuning(ctx, "dfs_proj", -1)


@pytest.mark.parametrize("c,minsup,way", [
    (datagen.zipf_baskets(10_000, 169, 1.0, 4.4, 1), 100, COLUMNS),        # few frequent pairs
    (datagen.zipf_baskets(30_000, 60, 1.0, 4.4, 1), 600, COLUMNS),
    (datagen.random_dense(20_000, 64, 0.05, 2), 40, PROJECTED),            # every pair frequent
    (datagen.random_dense(100_000, 64, 0.05, 2), 200, PROJECTED),
    (datagen.random_dense(12_060, 46, 0.29, 2), 700, PROJECTED),           # long rows
])
def test_small_matrices_take_the_columns_that_pay(ctx, c, minsup, way):
    want = oracle.apriori(c.indptr, c.indices, c.m, minsup).sha256()
    got = {w: _words(ctx, c, minsup, w) for w in (-1, CTAS, PROJECTED, COLUMNS)}
    assert all(g[0] == want for g in got.values())
    assert got[PROJECTED][1] < got[COLUMNS][1]
    assert got[-1][1:] == got[way][1:]


def _correlated(n, m, rho, q, seed):
    """A share rho of the rows holds each item with probability q, the others none."""
    rng = np.random.default_rng(seed)
    a = (rng.random((n, m)) < q) & (rng.random((n, 1)) < rho)
    r, i = np.nonzero(a)
    indptr = np.concatenate([[0], np.cumsum(np.bincount(r, minlength=n))]).astype(np.int64)
    return datagen.Csr(indptr, i.astype(np.int32), m)


# from 131,072 rows on the plan's totals choose (1 million rows and more in
# earnest; the oracle is why these are shorter)
@pytest.mark.parametrize("c,minsup,way", [
    (datagen.random_dense(140_000, 40, 0.7, 3), 56_000, CTAS),              # pairs alone: nothing to project for
    (datagen.random_dense(140_000, 8, 0.7, 3), 56_000, CTAS),
    (datagen.zipf_baskets(400_000, 150, 1.0, 4.4, 3), 8_000, CTAS),         # few triples, m' below m
    (datagen.random_dense(140_000, 60, 0.1, 3), 110, PROJECTED),            # many triples, sparse
    (_correlated(140_000, 14, 0.2, 0.9, 3), 12_000, PROJECTED),             # few rows hold everything: deep
    (datagen.planted(n=140_000, m=500, n_patterns=40, seed=3), 600, PROJECTED),  # more items than one launch plans
])
def test_long_columns_take_the_workers_that_pay(ctx, c, minsup, way):
    want = oracle.apriori(c.indptr, c.indices, c.m, minsup).sha256()
    got = {w: _words(ctx, c, minsup, w) for w in (-1, CTAS, PROJECTED)}
    assert all(g[0] == want for g in got.values())
    assert got[CTAS][2] < got[PROJECTED][2]
    assert got[-1][1:] == got[way][1:]
    # the CTA workers' other forms behind the one-launch plan
    for key, value in (("sparse_div", 4), ("root_reverse", 1), ("split_depth", 0)):
        old = {"sparse_div": -1, "root_reverse": 0, "split_depth": 8}[key]
        fim.fim_set_tuning(ctx, key, value)
        try:
            assert _words(ctx, c, minsup, CTAS)[0] == want
        finally:
            fim.fim_set_tuning(ctx, key, old)
    assert _words(ctx, c, minsup, -1, fim.FIM_DIFFSET_RULE)[0] == want
    assert _words(ctx, c, minsup, CTAS, fim.FIM_DIFFSET_RULE)[0] == want


@pytest.mark.parametrize("way", [-1, CTAS, PROJECTED])
def test_overflows_and_shallow_mines_behind_the_plan(ctx, way):
    # the mine is repeated with larger buffers, whoever searches; mines that end
    # before the search; matrices without a frequent pair or triple
    c = datagen.random_dense(140_000, 20, 0.3, 5)
    fim.fim_set_tuning(ctx, "test_record_cap", 100)
    try:
        want = oracle.apriori(c.indptr, c.indices, c.m, 1_000).sha256()
        assert _words(ctx, c, 1_000, way)[0] == want
    finally:
        fim.fim_set_tuning(ctx, "test_record_cap", 0)
    for minsup in (10_000, 12_700, 41_900, 42_000, 50_000):
        want = oracle.apriori(c.indptr, c.indices, c.m, minsup).sha256()
        assert _words(ctx, c, minsup, way)[0] == want
    for k in (1, 2, 3):
        want = oracle.apriori(c.indptr, c.indices, c.m, 1_000, max_len=k).sha256()
        assert _words(ctx, c, 1_000, way, fim.FIM_MAXLEN(k))[0] == want
