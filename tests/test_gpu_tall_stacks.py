"""QR of tall stacks on a cluster (60 and 97 columns, which one CTA has no room for) around 256 rows, where four
warps instead of one share the chain of a reflector (csrc/qr_cluster.cu), and well above.

Bounds as for every truncation of this library: kept dims equal, the represented tensors within 1e-12 of the
norm."""
import math

import numpy as np
import pytest

from oracle import bsmps as OB
from tests._common import rel_distance

pytestmark = pytest.mark.gpu

K, N = 20, 10


@pytest.fixture(scope="module")
def nat():
    from paper_2604_16118_gb300 import build, native
    build.build()
    return native


@pytest.fixture(scope="module")
def ctx(nat):
    return nat.Context(0)


def tall_iterate(rows, cols):
    """A chain of 20 sites, 10 particles: sectors 4 and 5 of bond 10 have `rows` columns together, which are
    the rows of the stack that ends in sector 5 of bond 11; that sector has `cols` columns."""
    bonds = []
    for b in range(K + 1):
        d = {}
        for q in range(max(0, N - (K - b)), min(b, N) + 1):
            left, right = math.comb(b, q), math.comb(K - b, N - q)
            d[(q, 0)] = min(left, 12 if b > 10 else right)
        bonds.append(d)
    bonds[10] = {(q, 0): 8 for q in range(1, 9)}
    bonds[10][(4, 0)], bonds[10][(5, 0)] = rows // 2, rows - rows // 2
    bonds[11][(5, 0)] = cols
    bonds[12][(5, 0)] = bonds[12][(6, 0)] = cols
    x = OB.BSMPS([0] * K, (N, 0), bonds, [dict() for _ in range(K)])
    n = x.layout()[1]
    return OB.BSMPS.from_flat([0] * K, (N, 0), bonds, np.random.default_rng(rows).standard_normal(n) / 8.0)


@pytest.mark.parametrize("rows", [255, 256, 257, 300, 419])
@pytest.mark.parametrize("cols", [60, 97])
def test_truncation_with_a_tall_stack(nat, ctx, rows, cols):
    ox = tall_iterate(rows, cols)
    lo = OB.left_orthogonalize(ox)
    assert lo.bonds[10][(4, 0)] + lo.bonds[10][(5, 0)] == rows and lo.bonds[11][(5, 0)] == cols >= 48
    x = nat.mps_import(ctx, K, 0, N, 0, ox.bonds, ox.to_flat())
    nrm = float(np.sqrt(OB.dot(ox, ox)))
    for rel in (0.0, 1e-2):
        y, dt, _ = nat.truncate(ctx, x, rel * nrm)
        oy, odt, _ = OB.truncate(ox, rel * nrm)
        assert y.bonds() == oy.bonds
        assert abs(dt - odt) <= 1e-12 * nrm
        assert rel_distance(OB.BSMPS.from_flat([0] * K, (N, 0), y.bonds(), y.export()), oy) <= 1e-12


@pytest.mark.parametrize("cols", [300, 331])
def test_stack_beyond_a_cluster(nat, ctx, cols):
    """924 rows: neither one CTA nor a cluster of 16 holds the stack, which is factorised in global memory."""
    K, N = 22, 11
    bonds = [{(q, 0): min(math.comb(b, q), 6 if b > 12 else math.comb(K - b, N - q))
              for q in range(max(0, N - (K - b)), min(b, N) + 1)} for b in range(K + 1)]
    bonds[11] = {(q, 0): 462 if q in (5, 6) else 6 for q in range(12)}
    bonds[12] = {(q, 0): cols if q == 6 else 6 for q in range(1, 12)}
    bonds[13][(6, 0)] = bonds[13][(7, 0)] = cols
    ox = OB.BSMPS([0] * K, (N, 0), bonds, [dict() for _ in range(K)])
    n = ox.layout()[1]
    ox = OB.BSMPS.from_flat([0] * K, (N, 0), bonds, np.random.default_rng(cols).standard_normal(n) / 16.0)
    lo = OB.left_orthogonalize(ox)
    assert lo.bonds[11][(5, 0)] + lo.bonds[11][(6, 0)] == 924 and lo.bonds[12][(6, 0)] == cols
    x = nat.mps_import(ctx, K, 0, N, 0, ox.bonds, ox.to_flat())
    nrm = float(np.sqrt(OB.dot(ox, ox)))
    y, dt, _ = nat.truncate(ctx, x, 1e-2 * nrm)
    oy, odt, _ = OB.truncate(ox, 1e-2 * nrm)
    assert y.bonds() == oy.bonds
    assert abs(dt - odt) <= 1e-12 * nrm
    assert rel_distance(OB.BSMPS.from_flat([0] * K, (N, 0), y.bonds(), y.export()), oy) <= 1e-12
