"""The split-precision product of one large pair of factors (operands split once,
128 x 128 tiles, three stages of 32 values of k) at the edges of its tiles and on
both sides of the size from which it is used, and the tensor-core FP64 product at
the edges of its 128 x 64 tiles, its chunks of 32 and its groups of 128 values of k.

Bounds: 2^-21 (4 + sqrt(K)) sum_k |a_ik| |b_kj| for the split product (operand
rounding 2^-22 each, the dropped low x low term, FP32 accumulation), the scheme's
own bound for the FP64 product."""
import numpy as np
import pytest

from oracle import ozaki as OZ

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nat():
    from paper_2604_16118_gb300 import build, native
    build.build()
    return native


@pytest.fixture(scope="module")
def ctx(nat):
    return nat.Context(0)


def factors(M, N, K):
    rng = np.random.default_rng(M * 7919 + N * 31 + K)
    A = rng.standard_normal((M, K)) * np.exp(rng.uniform(-3, 3, (M, 1)))
    B = rng.standard_normal((K, N)) * np.exp(rng.uniform(-3, 3, (1, N)))
    A[M // 2, : K // 2] = 0.0
    B[:, N // 2] = 0.0
    return A, B


@pytest.mark.parametrize("M,N,K", [(64, 64, 31), (64, 64, 32), (127, 129, 65), (128, 128, 96), (257, 130, 97),
                                   (1, 4000, 64), (4000, 1, 64), (900, 700, 513)])
@pytest.mark.parametrize("pad", [0, 3])
def test_split_product(nat, ctx, M, N, K, pad):
    import torch
    A, B = factors(M, N, K)
    dA = torch.from_numpy(np.hstack([A, np.full((M, pad), 1e300)])).cuda()[:, :K]
    dB = torch.from_numpy(np.hstack([B, np.full((K, pad), 1e300)])).cuda()[:, :N]
    dC = torch.full((M, N + pad), 7.0, dtype=torch.float64, device="cuda")
    nat.gemm_tf32x3(ctx, dA, dB, dC[:, :N])
    ctx.sync()
    C = dC.cpu().numpy()
    assert np.all(C[:, N:] == 7.0)
    scale = np.abs(A) @ np.abs(B)
    assert np.all(np.abs(C[:, :N] - A @ B) <= 2.0 ** -21 * (4.0 + np.sqrt(K)) * scale)


@pytest.mark.parametrize("M,N,K,S", [(1, 65, 32, 8), (129, 1, 31, 8), (128, 64, 128, 8), (128, 64, 129, 8),
                                     (257, 191, 385, 8), (300, 200, 513, 7), (64, 300, 160, 5), (200, 70, 300, 1),
                                     (1500, 1300, 96, 8)])
def test_emulated_fp64_product(nat, ctx, M, N, K, S):
    import torch
    A, B = factors(M, N, K)
    dA = torch.from_numpy(A).cuda()
    dB = torch.from_numpy(B).cuda()
    dC = torch.full((M, N + 1), 7.0, dtype=torch.float64, device="cuda")
    nat.gemm_ozaki(ctx, dA, dB, dC[:, :N], S)
    ctx.sync()
    C = dC.cpu().numpy()
    assert np.all(C[:, N] == 7.0)
    assert np.all(np.abs(C[:, :N] - A @ B) <= OZ.error_bound(A, B, S) + K * 2.0 ** -52 * (np.abs(A) @ np.abs(B)))
