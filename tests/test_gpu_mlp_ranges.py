"""The ranges of k in which the network's products are summed.

Sums of positive terms show what FP32 accumulation loses.  A range holds c chunks of 32 values of
k, 4 c additions to an accumulator that keeps 24 bits and may truncate: after i of them the sum is i / (4 c) of
the total, so they lose at most (4 c / 2 + 1) 2^-23 of it; adding R ranges, rounded to nearest, at most
(R / 2 + 1) 2^-24.  The ranges are cut in two while there are fewer than 296 tiles of 128 x 64 and each keeps
four chunks."""
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


def range_chunks(M, N, K):
    chunks, ranges = -(-K // 32), 1
    tiles = -(-M // 128) * -(-N // 64)
    while tiles * ranges < 296 and chunks // (2 * ranges) >= 4:
        ranges *= 2
    return chunks, -(-chunks // ranges)


def loss_of_sums(M, N, K):
    chunks, length = range_chunks(M, N, K)
    return (2 * length + 1) * 2.0 ** -23 + (-(-chunks // length) / 2 + 1) * 2.0 ** -24


def tf32(v):
    return ((np.ascontiguousarray(v, dtype=np.float32).view(np.uint32) + 0x1000) & 0xFFFFE000).astype(np.uint32).view(
        np.float32)


def positive(K, N, B):
    rng = np.random.default_rng(K + N + B)
    w = (rng.integers(128, 256, (N, K)) / 128.0).astype(np.float32)   # exact in BF16
    return w, tf32(rng.uniform(0.5, 1.5, (B, K)))


@pytest.mark.parametrize("K,N,B", [(4096, 64, 16), (4096, 64, 300), (2048, 64, 16), (2050, 130, 129), (4096, 4096, 1),
                                   (1024, 300, 40), (300, 300, 300)])
def test_forward_sums(nat, ctx, K, N, B):
    w, x = positive(K, N, B)
    y = nat.MLP(ctx, [K, N], np.concatenate([w.ravel(), np.zeros(N, np.float32)])).forward(x)
    exact = x.astype(np.float64) @ w.astype(np.float64).T
    assert np.abs(y / exact - 1.0).max() <= loss_of_sums(B, N, K)


@pytest.mark.parametrize("K,N,B", [(256, 256, 8192), (128, 256, 8192), (300, 70, 5000), (40, 3, 8192),
                                   (1024, 512, 2048)])
def test_weight_gradient_sums(nat, ctx, K, N, B):
    """The mean error shows how long the sums are (roundings to nearest average out): after i of 4 c
    additions the sum is i / (4 c) of the total, an addition of eight products to an accumulator truncates twice at most, by 2^-24
    of the sum on average: (4 c + 1) 2^-24."""
    w, x = positive(K, N, B)
    net = nat.MLP(ctx, [K, N], np.concatenate([w.ravel(), np.zeros(N, np.float32)]))
    _, g = net.loss_grad(x, np.zeros((B, N), np.float32))
    y = net.forward(x)
    dy = tf32(np.float32(2.0) * (np.float32(1.0) / np.float32(B * N)) * y)
    exact = dy.astype(np.float64).T @ x.astype(np.float64)
    err = g[:N * K].reshape(N, K) / exact - 1.0
    assert abs(err.mean()) <= (4 * range_chunks(N, K, B)[1] + 1) * 2.0 ** -24
    assert np.abs(err).max() <= loss_of_sums(N, K, B) + 2.0 ** -22


@pytest.mark.parametrize("widths,batch", [([1030, 1100, 1025, 3], 33), ([2048, 992, 1056], 5), ([37, 4096, 1], 130)])
def test_wide_layers_at_small_batches(nat, ctx, widths, batch):
    """Ranges summed by different CTAs: bias, ReLU, mask and both images of the result.  Bounds: two units
    of the TF32 rounding, as at the edges of the tiles."""
    rng = np.random.default_rng(batch)
    n = sum(i * o + o for i, o in zip(widths, widths[1:]))
    p = (rng.standard_normal(n) / np.sqrt(max(widths))).astype(np.float32)
    x = rng.standard_normal((batch, widths[0])).astype(np.float32)
    t = rng.standard_normal((batch, widths[-1])).astype(np.float32)
    net = nat.MLP(ctx, widths, p)
    x64, t64 = x.astype(np.float64), t.astype(np.float64)
    yo = OMLP.forward(p, widths, x64, tf32=True)[-1]
    assert np.abs(net.forward(x) - yo).max() <= 2e-3 * np.abs(yo).max()
    loss, g = net.loss_grad(x, t)
    lo, go = OMLP.loss_grad(p, widths, x64, t64, tf32=True)
    assert abs(loss - lo) <= 1e-3 * lo
    assert np.abs(g - go).max() <= 2.0 ** -10 * np.abs(go).max()
