"""The split-precision product of one pair of factors at the far ends of its sizes: sums so long that one
product takes more than the limit of a wait (1 s), and more columns than a grid has tiles in its second
dimension (65535 of 128)."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nat():
    from paper_2604_16118_gb300 import build, native
    build.build()
    return native


@pytest.fixture(scope="module")
def ctx(nat):
    return nat.Context(0)


def test_sum_over_2_to_27_values(nat, ctx):
    import torch
    K = 1 << 27
    A = torch.zeros(1, K, dtype=torch.float64, device="cuda")
    A[0, [0, 12345, K // 2, K - 1]] = torch.tensor([1.0, 2.0, 3.0, 4.0], dtype=torch.float64, device="cuda")
    B = torch.ones(K, 1, dtype=torch.float64, device="cuda")
    C = torch.empty(1, 1, dtype=torch.float64, device="cuda")
    nat.gemm_tf32x3(ctx, A, B, C)
    ctx.sync()
    assert C.item() == 10.0


def test_more_columns_than_65535_tiles(nat, ctx):
    import torch
    M, N = 65, 65536 * 128 + 1
    g = torch.Generator(device="cuda").manual_seed(1)
    A = torch.randn(M, 1, dtype=torch.float64, device="cuda", generator=g)
    B = torch.randn(1, N, dtype=torch.float64, device="cuda", generator=g)
    C = torch.full((M, N), 7.0, dtype=torch.float64, device="cuda")
    nat.gemm_tf32x3(ctx, A, B, C)
    ctx.sync()
    C -= A @ B
    # operands rounded by 2^-22 each, the low x low term and one FP32 rounding: 2^-21 (4 + 1) at one value of k
    assert (C.abs() <= 5 * 2.0 ** -21 * A.abs() * B.abs()).all()
