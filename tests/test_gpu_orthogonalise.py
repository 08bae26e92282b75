"""The orthogonalisation of the FP32 rotations inside the one-CTA sector SVD: P with P^T P = I + E for
E of random signs, of one sign (||E||_2 as large as its entries allow) and of one column, from far
below the size at which one pass is enough to far above it.

Bound: ||Q^T Q - I||_2 at most (k + 16) eps: k eps is the limit to which the Jacobi that follows takes
cosines, 16 eps covers the FP64 roundings of the products here and there.  Q stays next to P:
||Q - P||_2 <= ||E||_2."""
import numpy as np
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


def errors(k, kind, size):
    rng = np.random.default_rng(k)
    if kind == "random":
        E = rng.uniform(-size, size, (k, k))
    elif kind == "one sign":
        E = np.full((k, k), size)
    else:
        E = np.zeros((k, k))
        E[k // 2] = E[:, k // 2] = size
    return 0.5 * (E + E.T)


@pytest.mark.parametrize("k", [1, 2, 7, 8, 9, 16, 17, 33, 64])
@pytest.mark.parametrize("kind", ["random", "one sign", "column"])
@pytest.mark.parametrize("size", [1e-9, 1e-6, 7.5e-6, 1e-4, 2e-3])
def test_orthogonal_to_the_limit_of_the_jacobi(nat, ctx, k, kind, size):
    w, v = np.linalg.eigh(np.eye(k) + errors(k, kind, size))
    u = np.linalg.qr(np.random.default_rng(1).standard_normal((k, k)))[0]
    P = u @ ((v * np.sqrt(w)) @ v.T)    # P^T P = I + E
    Q = nat.check_orthogonalise(ctx, P)
    bound = (k + 16) * 2.0 ** -52
    assert np.linalg.norm(Q.T @ Q - np.eye(k), 2) <= bound
    assert np.linalg.norm(Q - P, 2) <= np.abs(w - 1.0).max() + bound


@pytest.mark.parametrize("k", [2, 64])
@pytest.mark.parametrize("bad", [np.nan, np.inf, 3.0])
def test_refuses_what_is_far_from_orthogonal(nat, ctx, k, bad):
    P = np.eye(k)
    P[0, k - 1] = bad
    assert nat.check_orthogonalise(ctx, P) is None
