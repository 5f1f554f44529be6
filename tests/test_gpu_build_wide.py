"""Building the bit columns around the widths where the build's tile changes.

Up to 1,024 items a CTA owns 16-word runs; beyond that 8-word runs with four
warps to a row group, up to 7,200 items to a block.  Rows are short, long
(several chunks of 32 ids per warp), empty, or repeat an id, and the last row
group is ragged.  The mine must match the oracle exactly on every input path.
"""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

fim = pytest.importorskip("paper_2412_19420_gb300.fim")


def _db(n, m, rows, seed):
    rng = np.random.default_rng(seed)
    out = []
    for i in range(n):
        k = {"short": 1 + int(rng.integers(12)), "long": 150 + int(rng.integers(100)),
             "gaps": int(rng.integers(12)) * (i % 3 != 0)}[rows]
        r = rng.integers(0, m, k)
        if k:  # the edges of the tile and a few items that every size finds frequent
            r = np.append(r, rng.choice([0, 1, m // 2, m - 2, m - 1, min(m - 1, 1023)], 3))
        out.append(r)  # (ids may repeat)
    indptr = np.concatenate([[0], np.cumsum([len(r) for r in out])]).astype(np.int64)
    return indptr, np.concatenate(out).astype(np.int32)


@pytest.mark.parametrize("path", ["host", "device", "compact"])
@pytest.mark.parametrize("rows", ["short", "long", "gaps"])
@pytest.mark.parametrize("m", [1024, 1025, 2000, 7200, 7201])
def test_build(m, rows, path):
    n = 1_000 + m % 7
    indptr, indices = _db(n, m, rows, m)
    minsup = n // 8
    want = oracle.apriori(indptr, indices, m, minsup)
    ctx = fim.fim_create(0)
    try:
        if path == "device":
            fim.fim_build_bitmaps(ctx, torch.from_numpy(indptr).cuda(), torch.from_numpy(indices).cuda(), m)
        elif path == "compact":
            fim.fim_build_bitmaps(ctx, indptr.astype(np.uint32), indices.astype(np.uint16), m)
        else:
            fim.fim_build_bitmaps(ctx, indptr, indices, m)
        fim.fim_mine(ctx, minsup)
        got = fim.fim_fetch_results(ctx)
    finally:
        fim.fim_destroy(ctx)
    assert got.sha256() == want.sha256(), (len(got), len(want))
