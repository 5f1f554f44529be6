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
