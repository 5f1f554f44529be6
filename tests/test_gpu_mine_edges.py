"""Mines at the edges of what the search and the record arena are sized for,
against the oracle or closed forms, on contexts whose earlier calls left other
contents in the buffers."""
import numpy as np
import pytest

import oracle
from paper_2412_19420_gb300 import datagen

pytestmark = pytest.mark.gpu
fim = pytest.importorskip("paper_2412_19420_gb300.fim")


@pytest.fixture()
def ctx():
    c = fim.fim_create(0)
    yield c
    fim.fim_destroy(c)


def _disjoint_pairs(n, m, n_pairs, per, seed):
    """m frequent items of which only the pairs {2i, 2i + 1}, i < n_pairs, are
    frequent: no item has two partners."""
    rng = np.random.default_rng(seed)
    rows = [[] for _ in range(n)]
    for i in range(n_pairs):
        for r in rng.choice(n // 2, size=per, replace=False):
            rows[r] += [2 * i, 2 * i + 1]
    free = rng.permutation(np.arange(n // 2, n))
    at = 0
    for j in range(2 * n_pairs, m):  # the others alone in their rows
        for r in free[at:at + per]:
            rows[r].append(j)
        at += per
    return datagen.from_lists([sorted(set(x)) for x in rows], m)


# an earlier call that leaves a root order behind, longer than the new roots
# and meant for other ones: a small matrix mined on its bit columns, a trace, a
# batch, a shard
@pytest.mark.parametrize("first", ["direct", "trace", "batch", "shard", "none"])
def test_pairs_without_third_items(ctx, first):
    a = datagen.zipf_baskets(3_000, 90, 0.9, 7.0, 4)
    if first != "none":
        fim.fim_build_bitmaps(ctx, a.indptr, a.indices, a.m)
        if first == "direct":
            fim.fim_mine(ctx, 12)
        elif first == "trace":
            fim.fim_mine(ctx, 12, fim.FIM_TRACE)
        elif first == "shard":
            fim.fim_mine_shard(ctx, 12, 0, 0, 2)
        else:
            fim.fim_mine_batched(ctx, fim.BatchDescriptor([a] * 3, [12] * 3))
    c = _disjoint_pairs(16_000, 300, 9, 25, 3)
    want = oracle.apriori(c.indptr, c.indices, c.m, 20)
    assert len(want) == 309
    fim.fim_build_bitmaps(ctx, c.indptr, c.indices, c.m)
    for _ in range(2):
        fim.fim_mine(ctx, 20)
        assert fim.fim_fetch_results(ctx).sha256() == want.sha256()
        assert fim.fim_get_stats(ctx)["supports_dfs"] == 0


def test_reservations_that_end_past_the_arena(ctx):
    # workers reserve up to 64 record slots ahead: capacities from exactly the
    # sets to beyond all reservations, so that the last one ends on either side
    c = datagen.from_lists([list(range(14))] * 40, 14)
    want = oracle.apriori(c.indptr, c.indices, c.m, 40)
    sets = (1 << 14) - 1
    assert len(want) == sets
    fim.fim_build_bitmaps(ctx, c.indptr, c.indices, c.m)
    grown = 0
    for cap in range(sets, sets + 8192, 5):
        fim.fim_set_tuning(ctx, "test_record_cap", cap)
        fim.fim_mine(ctx, 40)
        assert fim.fim_fetch_results(ctx).sha256() == want.sha256(), cap
        grown += fim.fim_get_stats(ctx)["launches_mine"] > 12
    assert 0 < grown < 1638  # the arena was too small at first, and large enough at last
    fim.fim_set_tuning(ctx, "test_record_cap", 0)


def test_more_triples_than_records_fit(ctx):
    # 2,300 frequent triples and a search below them; room for fewer roots than
    # there are, for exactly as many, and for all records
    c = datagen.from_lists([list(range(25)) for _ in range(4)] + [[r % 25] for r in range(40_000)], 25)
    fim.fim_set_tuning(ctx, "spin_limit_ms", 2_000)
    fim.fim_build_bitmaps(ctx, c.indptr, c.indices, c.m)
    for max_len in (3, 4):
        want = oracle.apriori(c.indptr, c.indices, c.m, 4, max_len=max_len)
        for cap in (1, 24, 326, 1_000, 2_023, 2_024, 2_299, 2_300, 2_624, 2_625, 2_626, 20_000):
            fim.fim_set_tuning(ctx, "test_record_cap", cap)
            fim.fim_mine(ctx, 4, fim.FIM_MAXLEN(max_len))
            assert fim.fim_fetch_results(ctx).sha256() == want.sha256(), (max_len, cap)


def test_a_million_triples_on_a_fresh_context(ctx):
    # all triples of 200 items: more than the 2^20 records a context begins with
    n, m = 2_000, 200
    indptr = np.arange(n + 1, dtype=np.int64) * m
    indices = np.tile(np.arange(m, dtype=np.int32), n)
    fim.fim_set_tuning(ctx, "spin_limit_ms", 2_000)
    fim.fim_build_bitmaps(ctx, indptr, indices, m)
    fim.fim_mine(ctx, n, fim.FIM_MAXLEN(3))
    got = fim.fim_fetch_results(ctx)
    n1, n2, n3 = m, m * (m - 1) // 2, m * (m - 1) * (m - 2) // 6
    assert len(got) == n1 + n2 + n3 and np.all(got.supports == n)
    tri = got.items[n1 + 2 * n2:].reshape(-1, 3).astype(np.int64)
    assert np.all(np.diff(tri, axis=1) > 0)
    key = (tri[:, 0] * m + tri[:, 1]) * m + tri[:, 2]
    assert np.all(np.diff(key) > 0)


def test_kept_rows_give_way_to_what_a_mine_needs():
    # the rows that a build keeps for the pair pass are optional: where device
    # memory runs out (a limit of the context's own), they go first
    import torch
    rng = np.random.default_rng(2)
    n, m = 2_000_000, 300
    indptr = torch.arange(n + 1, dtype=torch.int64, device="cuda") * 4
    ids = (rng.integers(0, m, (n, 1)) + np.arange(4) * rng.integers(1, 75, (n, 1))) % m  # four distinct ids a row
    ids = torch.from_numpy(np.sort(ids, axis=1).astype(np.int32).ravel()).cuda()
    rows_mb = n * 48 >> 20

    def mine(limit_mb):
        c = fim.fim_create(0)
        try:
            fim.fim_set_tuning(c, "test_memory_mb", limit_mb)
            fim.fim_set_tuning(c, "pairs_rows", 1)
            out = []
            fim.fim_build_bitmaps(c, indptr, ids, m)
            for _ in range(2):
                fim.fim_mine(c, 200)
                out.append(fim.fim_fetch_results(c).sha256())
            st = fim.fim_get_stats(c)
            return out, st["pair_rows"], st["peak_device_bytes"] >> 20
        finally:
            fim.fim_destroy(c)

    want, rows, peak = mine(0)
    assert rows == 1 and want[0] == want[1]
    kept = []
    for less in (rows_mb // 8, rows_mb // 4, rows_mb // 2, rows_mb - 5):
        got, rows, _ = mine(peak - less)
        assert got == want
        kept.append(rows)
    assert kept[-1] == 0
    with pytest.raises(fim.FimError, match=rf"\({fim.FIM_E_NOMEM}\)"):
        mine(100)


def _built_mb(indptr, indices, m):
    c = fim.fim_create(0)
    try:
        fim.fim_build_bitmaps(c, indptr, indices, m)
        return fim.fim_get_stats(c)["peak_device_bytes"] / 2 ** 20
    finally:
        fim.fim_destroy(c)


def test_rows_are_kept_only_for_a_pass_that_reads_them():
    # up to 256 items no pair is outside the tensor cores' block: a build then
    # holds the columns (with a quarter's slack) and not 48 bytes a row more
    import torch
    n = 1_000_000
    indptr = torch.arange(n + 1, dtype=torch.int64, device="cuda") * 3
    ids = (torch.arange(3 * n, device="cuda") % 250).to(torch.int32)
    columns = 1.25 * 256 * 4 * (-(-n // 4096) * 128) / 2 ** 20
    assert columns <= _built_mb(indptr, ids, 256) <= columns + 2
    assert _built_mb(indptr, ids, 257) > columns + 40


@pytest.mark.parametrize("m", [1, 256, 257, 2_000])
def test_matrices_without_ids(ctx, m):
    # host, page-locked and device input, with and without room for kept rows
    import torch
    for limit_mb in (0, 12):
        for n in (1, 33, 5_000):
            indptr, ids = np.zeros(n + 1, np.int64), np.zeros(0, np.int32)
            for ip, ix in ((indptr, ids), (indptr.astype(np.uint32), ids.astype(np.uint16)),
                           (torch.from_numpy(indptr).pin_memory().numpy(), ids),
                           (torch.from_numpy(indptr).cuda(), torch.zeros(1, dtype=torch.int32, device="cuda"))):
                c = fim.fim_create(0)
                try:
                    fim.fim_set_tuning(c, "test_memory_mb", limit_mb)
                    fim.fim_build_bitmaps(c, ip, ix, m)
                    fim.fim_set_tuning(c, "test_memory_mb", 0)
                    fim.fim_mine(c, 1)
                    assert len(fim.fim_fetch_results(c)) == 0
                finally:
                    fim.fim_destroy(c)


def test_kept_rows_of_host_input_take_what_they_hold():
    # pageable and page-locked host arrays, wide and compact, whose number of
    # ids is known before the build
    import torch
    n, m = 1_000_000, 300
    indptr = np.arange(n + 1, dtype=np.int64) * 3
    ids = (np.arange(3 * n) % m).astype(np.int32)
    columns = 1.25 * m * 4 * (-(-n // 4096) * 128) / 2 ** 20
    rows = 1.25 * (4 * n + 2 * 3 * n) / 2 ** 20
    for ip, ix in ((indptr, ids), (indptr.astype(np.uint32), ids.astype(np.uint16))):
        staged = 1.25 * (ip.nbytes + ix.nbytes) / 2 ** 20
        assert columns + rows <= _built_mb(ip, ix, m) <= columns + rows + staged + 2
        pinned = [torch.from_numpy(a.view({4: np.int32, 8: np.int64, 2: np.int16}[a.itemsize])).pin_memory().numpy()
                  .view(a.dtype) for a in (ip, ix)]
        assert columns + rows <= _built_mb(*pinned, m) <= columns + rows + 2
    c = fim.fim_create(0)
    try:  # a matrix of longer rows, then shorter ones, then none kept
        fim.fim_set_tuning(c, "pairs_rows", 1)
        for mean, kept in ((20, 1), (4, 1), (30, 0), (4, 1)):
            d = datagen.zipf_baskets(20_000, 400, 0.3, mean, mean)
            want = oracle.apriori(d.indptr, d.indices, d.m, 30, max_len=2)
            fim.fim_build_bitmaps(c, d.indptr, d.indices, d.m)
            fim.fim_mine(c, 30, fim.FIM_MAXLEN(2))
            assert fim.fim_fetch_results(c).sha256() == want.sha256()
            assert fim.fim_get_stats(c)["pair_rows"] == kept
    finally:
        fim.fim_destroy(c)
