"""The network's kernels at the edges of their tiles (32 samples a CTA, 64 to a
gradient step, 256 to a gradient chunk) and with buffers that start on any
4-byte boundary: fp32 mode within 1e-5 of the float64 oracle, as the tolerance
of the existing tests derives it."""
import numpy as np
import pytest

from oracle import mlp as ref
from paper_2412_19420_gb300 import datagen

pytestmark = pytest.mark.gpu
fim = pytest.importorskip("paper_2412_19420_gb300.fim")
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ctx():
    c = fim.fim_create(0)
    yield c
    fim.fim_destroy(c)


def _at(a, off):
    """A device copy that starts `off` floats into its allocation."""
    buf = torch.zeros(a.size + 8, dtype=torch.float32, device="cuda")
    v = buf[off:off + a.size]
    v.copy_(torch.from_numpy(np.ascontiguousarray(a).ravel()))
    return v


@pytest.mark.parametrize("B,off", [(1, 0), (31, 1), (32, 2), (33, 3), (64, 0), (65, 1), (255, 2), (257, 3), (513, 0)])
def test_tile_edges_and_unaligned_buffers(ctx, B, off):
    rng = np.random.default_rng(B)
    x = rng.normal(size=(B, 8)).astype(np.float32)
    t = np.stack([rng.normal(4, 2, B), (rng.random(B) < 0.3)], 1).astype(np.float32)
    p = datagen.mlp_init_weights(B) + rng.normal(0, 0.05, fim.FIM_MLP_PARAMS).astype(np.float32)
    dp, dx, dt = _at(p, off), _at(x, off).view(B, 8), _at(t, off).view(B, 2)
    dy, dc = _at(np.zeros((B, 2), np.float32), off).view(B, 2), _at(np.zeros((B, 256), np.float32), off).view(B, 256)
    dg = _at(np.zeros(fim.FIM_MLP_PARAMS, np.float32), off)
    torch.cuda.synchronize()
    fim.fim_mlp_forward(ctx, dp, dx, dy, dc)
    loss = fim.fim_mlp_backward(ctx, dp, dx, dy, dt, dc, dg)
    torch.cuda.synchronize()
    ry, cache = ref.forward(p.astype(np.float64), x.astype(np.float64))
    rg = ref.backward(p.astype(np.float64), cache, ry, t.astype(np.float64))
    y, g = dy.cpu().numpy(), dg.cpu().numpy()
    assert np.max(np.abs(y - ry)) <= 1e-5 * np.max(np.abs(ry))
    assert loss == pytest.approx(ref.loss(ry, t), rel=1e-5)
    o = 0
    for s in ref.SHAPES:
        k = int(np.prod(s))
        assert np.max(np.abs(g[o:o + k] - rg[o:o + k])) <= 1e-5 * max(1e-30, np.max(np.abs(rg[o:o + k]))), s
        o += k
