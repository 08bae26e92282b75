"""Inner products whose environment blocks lie on both sides of the sizes up to which an entry is summed by one
thread without staging (32 rows and columns, 128 entries, 32 terms), with and without an operator, against
the oracle.  Bound: FP64 rounding of the sums, 1e-12 of the product of the norms (and of the operator's scale)."""
import numpy as np
import pytest

from oracle import bsmps as OB
from synth import spinless_random_chain
from tests._common import oracle_mpo

pytestmark = pytest.mark.gpu

K, N = 6, 3


@pytest.fixture(scope="module")
def nat():
    from paper_2604_16118_gb300 import build, native
    build.build()
    return native


@pytest.fixture(scope="module")
def ctx(nat):
    return nat.Context(0)


def iterate(d, seed):
    bonds = [{(q, 0): 1 if b in (0, K) else d for q in range(max(0, N - (K - b)), min(b, N) + 1)} for b in range(K + 1)]
    x = OB.BSMPS([0] * K, (N, 0), bonds, [dict() for _ in range(K)])
    v = np.random.default_rng(seed).standard_normal(x.layout()[1]) / np.sqrt(d)
    return OB.BSMPS.from_flat([0] * K, (N, 0), bonds, v)


@pytest.mark.parametrize("da,db", [(1, 1), (1, 33), (2, 32), (4, 8), (8, 16), (8, 17), (11, 12), (12, 11), (15, 16),
                                   (16, 8), (17, 2), (32, 4), (33, 3), (40, 40)])
def test_inner_products(nat, ctx, da, db):
    wl = spinless_random_chain(K=K, N=N, seed=1)
    a, b = iterate(da, 1), iterate(db, 2)
    ga, gb = [nat.mps_import(ctx, K, 0, N, 0, o.bonds, o.to_flat()) for o in (a, b)]
    size = np.sqrt(OB.dot(a, a) * OB.dot(b, b))
    assert abs(nat.dot(ctx, ga, gb) - OB.dot(a, b)) <= 1e-12 * size
    W = nat.mpo_from_integrals(ctx, wl.h, wl.eri, 0, N, 4.0)
    oW = oracle_mpo(wl, 4.0)
    scale = max(abs(OB.dot(x, OB.apply_exact(oW, x, shift=0.5))) / OB.dot(x, x) for x in (a, b))
    assert abs(nat.dot(ctx, ga, gb, W, 0.5) - OB.dot(a, OB.apply_exact(oW, b, shift=0.5))) <= 1e-12 * size * (1 + scale)
