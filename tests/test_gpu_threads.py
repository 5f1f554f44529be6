"""Contexts of their own on threads of their own: matrices of different widths
built and mined at the same time, whose kernels take different amounts of
shared memory."""
import threading

import numpy as np
import pytest

import oracle
from paper_2412_19420_gb300 import datagen

pytestmark = pytest.mark.gpu
fim = pytest.importorskip("paper_2412_19420_gb300.fim")


def _together(jobs):
    errors = []

    def run(job):
        try:
            job()
        except Exception as e:  # noqa: BLE001  (handed to the test's thread)
            errors.append(e)

    ts = [threading.Thread(target=run, args=(j,)) for j in jobs]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not errors, errors[:2]


def _rows(n, m, seed):
    """n rows of five distinct items of m, every item among them."""
    rng = np.random.default_rng(seed)
    start, step = rng.integers(0, m, (n, 1)), rng.integers(1, m // 5, (n, 1))
    start[:m, 0] = np.arange(min(m, n))
    ids = np.sort((start + step * np.arange(5)) % m, axis=1).astype(np.int32)
    return datagen.Csr(np.arange(n + 1, dtype=np.int64) * 5, ids.ravel(), m)


@pytest.mark.parametrize("widths,reps", [((80, 900), 400), ((1_100, 7_000), 200), ((300, 20_000), 100)])
def test_builds_and_mines_of_different_widths(widths, reps):
    def job(m):
        c = _rows(max(3_000, m), m, m)
        want = oracle.apriori(c.indptr, c.indices, m, 3, max_len=2).sha256()

        def go():
            ctx = fim.fim_create(0)
            try:
                fim.fim_set_tuning(ctx, "pairs_rows", 1)
                for i in range(reps):
                    fim.fim_build_bitmaps(ctx, c.indptr, c.indices, m)
                    if i % 4 == 0:
                        fim.fim_mine(ctx, 3, fim.FIM_MAXLEN(2))
                        assert fim.fim_fetch_results(ctx).sha256() == want
            finally:
                fim.fim_destroy(ctx)
        return go

    _together([job(m) for m in widths] * 2)


def test_batches_of_different_widths():
    def job(m):
        dbs = [_rows(2_000, m, m + d) for d in range(4)]
        want = [oracle.apriori(c.indptr, c.indices, m, 20).sha256() for c in dbs]

        def go():
            ctx = fim.fim_create(0)
            try:
                for i in range(60):
                    desc = fim.BatchDescriptor(dbs[: 1 + i % 4], [20] * (1 + i % 4))  # another graph each time
                    fim.fim_mine_batched(ctx, desc)
                    for d in range(1 + i % 4):
                        assert fim.fim_fetch_batched(ctx, d).sha256() == want[d]
            finally:
                fim.fim_destroy(ctx)
        return go

    _together([job(m) for m in (40, 1_000)] * 2)
