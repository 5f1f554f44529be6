"""The prefix extension on projected columns (k_proj.cu) against the oracle.

The plain search runs on warp workers: on the bit columns themselves where the
frequent matrix is small, on columns projected onto each root item's
transactions elsewhere.  Both must give the oracle's itemsets, bit for bit, at
the edges of a projected column (one word, a 128-row step, several 128-word
chunks), of a gather tile (1,024 rows) and of a row-list segment (8,192 words),
with more candidates than a sweep or a shared-memory list holds, and for
columns too long for warp workers, which the CTA workers mine.
"""
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


def _check(ctx, c, minsup, flags=0, **kw):
    fim.fim_build_bitmaps(ctx, c.indptr, c.indices, c.m)
    fim.fim_mine(ctx, minsup, flags)
    got = fim.fim_fetch_results(ctx)
    want = oracle.apriori(c.indptr, c.indices, c.m, minsup, **kw)
    assert got.sha256() == want.sha256(), (len(got), len(want))


def _blocks(n, m, sizes, extra, seed):
    """Items 0..k-1 share exactly sizes[0] rows, the next group sizes[1], ...;
    a group has 5 items, so its sets go to size 5; `extra` noise items a row."""
    rng = np.random.default_rng(seed)
    rows = [[] for _ in range(n)]
    for g, s in enumerate(sizes):
        for r in rng.choice(n, size=s, replace=False):
            rows[r] += list(range(5 * g, 5 * g + 5))
    for r in range(n):
        rows[r] += list(rng.integers(5 * len(sizes), m, size=extra))
    return datagen.from_lists(rows, m)


# supports at the edges of a word, a 128-row step, a 1,024-row gather tile
@pytest.mark.parametrize("sizes", [(31, 32, 33, 40), (127, 128, 129, 500), (1023, 1024, 1025, 4097)])
def test_projected_column_edges(ctx, sizes):
    # 270,000 rows: the columns span a second row-list segment (262,144 rows)
    c = _blocks(270_000, 60, sizes, 1, 7)
    _check(ctx, c, 30)


@pytest.mark.parametrize("n,m,density,minsup", [
    (40_000, 70, 0.25, 2_300),    # wide lists: more candidates than a sweep, projected
    (40_000, 52, 0.25, 145),      # four levels
    (3_000, 40, 0.35, 60),        # the same on whole columns (small matrix)
])
def test_wide_classes(ctx, n, m, density, minsup):
    _check(ctx, datagen.random_dense(n, m, density, 5), minsup)


def test_long_sibling_lists_spill(ctx):
    # 400 items in every pair: root candidate lists longer than a worker's
    # shared-memory list
    rng = np.random.default_rng(3)
    m, n = 400, 20_000
    rows = [sorted(rng.choice(m, size=60, replace=False)) for _ in range(n)]
    _check(ctx, datagen.from_lists(rows, m), 85)


def test_deep_searches(ctx):
    # sets of up to 14 items: fourteen levels of stored prefixes
    n, m = 70_000, 60
    rows = [list(range(min(m, 14 + r % 3))) if r < 400 else [r % m] for r in range(n)]
    c = datagen.from_lists(rows, m)
    for flags, kw in ((0, {}), (fim.FIM_MAXLEN(4), dict(max_len=4)), (fim.FIM_STRICT, dict(strict=True))):
        _check(ctx, c, 300, flags, **kw)


def test_projection_too_long_for_warp_workers(ctx):
    # items in 1.5 million rows: projected columns past the warp workers'
    # limit, mined by the CTA workers
    c = datagen.random_dense(2_500_000, 6, 0.6, 9)
    _check(ctx, c, 200_000)


def test_shards_and_repeats(ctx):
    c = datagen.planted(n=60_000, m=500, n_patterns=40, seed=11)
    want = oracle.apriori(c.indptr, c.indices, c.m, 250)
    fim.fim_build_bitmaps(ctx, c.indptr, c.indices, c.m)
    for per_sm in (4, 3, 2, 1):
        fim.fim_set_tuning(ctx, "dfs_ctas_per_sm", per_sm)
        try:
            for _ in range(2):
                fim.fim_mine(ctx, 250)
                assert fim.fim_fetch_results(ctx).sha256() == want.sha256()
        finally:
            fim.fim_set_tuning(ctx, "dfs_ctas_per_sm", 4)
    parts = []
    for s in range(3):
        fim.fim_mine_shard(ctx, 250, 0, s, 3)
        parts.append(fim.fim_fetch_results(ctx))
    fim.fim_merge_results(ctx, c.n, c.m, parts)
    assert fim.fim_fetch_results(ctx).sha256() == want.sha256()


@pytest.mark.parametrize("logit", [-5.0, 5.0, None])
def test_representation_choice_on_projected_columns(ctx, logit):
    # the network (forced to either representation, or as drawn) and the size
    # rule on warp workers: projected, direct and with queued classes
    w = datagen.mlp_init_weights(2)
    if logit is not None:
        w[-1] = logit
    fim.fim_sched_load_weights(ctx, w)
    fim.fim_set_tuning(ctx, "learned_kmin", 1)
    try:
        for c, minsup in [(datagen.planted(n=60_000, m=500, n_patterns=40, seed=11), 250),
                          (datagen.random_dense(12_000, 40, 0.3, 3), 300),
                          (datagen.zipf_baskets(3_000, 90, 0.9, 7.0, 4), 12)]:
            for flags in (fim.FIM_LEARNED, fim.FIM_DIFFSET_RULE, fim.FIM_LEARNED | fim.FIM_MAXLEN(4)):
                _check(ctx, c, minsup, flags, **(dict(max_len=4) if flags >> 24 else {}))
                st = fim.fim_get_stats(ctx)
                if logit is not None and flags == fim.FIM_LEARNED:
                    # queued classes have no parent's bitmap to differ from
                    assert (st["diffset_classes"] > 0) == (logit > 0 and st["classes"] > st["tasks_pushed"])
            fim.fim_set_tuning(ctx, "learned_order", 1)  # pair roots, in the network's order
            _check(ctx, c, minsup, fim.FIM_LEARNED)
            fim.fim_set_tuning(ctx, "learned_order", 0)
    finally:
        fim.fim_set_tuning(ctx, "learned_order", 0)
        fim.fim_set_tuning(ctx, "learned_kmin", 8)
