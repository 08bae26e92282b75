"""The network's products at the edges of their tiles (128 rows and columns, 32
values of k, split k ranges): outputs, loss and gradients against the oracle's
definition (TF32-rounded operands).  Bounds: two units of the TF32 rounding (2^-11)."""
import numpy as np
import pytest

from oracle import mlp as OMLP

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nat():
    from paper_2604_16118_gb300 import build, native
    build.build()
    return native


@pytest.fixture(scope="module")
def ctx(nat):
    return nat.Context(0)


@pytest.mark.parametrize("widths,batch", [([1, 1], 1), ([3, 5, 2], 7), ([31, 33, 1], 32), ([32, 128, 128, 4], 128),
                                          ([130, 127, 129, 3], 33), ([64, 256, 2], 1025), ([5, 300, 7], 4100)])
def test_products_at_tile_edges(nat, ctx, widths, batch):
    rng = np.random.default_rng(batch)
    n = sum(i * o + o for i, o in zip(widths, widths[1:]))
    p = (rng.standard_normal(n) / np.sqrt(max(widths))).astype(np.float32)
    x = rng.standard_normal((batch, widths[0])).astype(np.float32)
    t = rng.standard_normal((batch, widths[-1])).astype(np.float32)
    net = nat.MLP(ctx, widths, p)
    x64, t64 = x.astype(np.float64), t.astype(np.float64)
    # both sides round the same operands to TF32; an FP32 activation next to a rounding
    # boundary may fall on the other side, which moves one term by 2^-11 of itself
    y = net.forward(x)
    yo = OMLP.forward(p, widths, x64, tf32=True)[-1]
    assert np.abs(y - yo).max() <= 2e-3 * np.abs(yo).max()
    loss, g = net.loss_grad(x, t)
    lo, go = OMLP.loss_grad(p, widths, x64, t64, tf32=True)
    assert abs(loss - lo) <= 1e-3 * lo
    assert np.abs(g - go).max() <= 2.0 ** -10 * np.abs(go).max()
