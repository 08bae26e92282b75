"""Sector SVDs of one and two kept columns over 1 to 33 rows (rotated in FP64 from the start up to 32 rows, by the
general path beyond), with independent, dependent, vanishing and nearly orthogonal columns, against the oracle's truncation.

Bounds as for every truncation of this library: kept dims equal, the represented tensors within 1e-12 of the
norm."""
import math

import numpy as np
import pytest

from oracle import bsmps as OB
from tests._common import rel_distance

pytestmark = pytest.mark.gpu

K, N = 10, 5


@pytest.fixture(scope="module")
def nat():
    from paper_2604_16118_gb300 import build, native
    build.build()
    return native


@pytest.fixture(scope="module")
def ctx(nat):
    return nat.Context(0)


def iterate(rows, kind):
    """Sector 4 of bond 8 has `rows` rows and two ways to be completed over the last two sites."""
    bonds = OB.default_dims([0] * K, (N, 0), 400)
    for b in range(8):
        bonds[b] = {(q, 0): math.comb(b, q) for q in range(max(0, b - 5), min(b, N) + 1)}
    bonds[8] = {(3, 0): min(rows, 7), (4, 0): rows, (5, 0): min(rows, 3)}
    x = OB.BSMPS([0] * K, (N, 0), bonds, [dict() for _ in range(K)])
    rng = np.random.default_rng(rows)
    x = OB.BSMPS.from_flat([0] * K, (N, 0), bonds, rng.standard_normal(x.layout()[1]) / 4.0)
    a, b = x.cores[8][((4, 0), 0)], x.cores[8][((4, 0), 1)]
    if kind == "dependent":
        b[:, 0] = 0.5 * a[:, 0]
    elif kind == "vanishing":
        b[:] = 0.0
    elif kind == "graded":
        b *= 1e-9
    elif kind == "small":     # fourth powers of the entries leave the range
        x.cores[0] = {k: 1e-80 * v for k, v in x.cores[0].items()}
    return x


@pytest.mark.parametrize("rows", [1, 2, 3, 4, 8, 9, 16, 17, 31, 32, 33])
@pytest.mark.parametrize("kind", ["independent", "dependent", "vanishing", "graded", "small"])
def test_truncation(nat, ctx, rows, kind):
    ox = iterate(rows, kind)
    x = nat.mps_import(ctx, K, 0, N, 0, ox.bonds, ox.to_flat())
    nrm = float(np.sqrt(OB.dot(ox, ox)))
    assert OB.left_orthogonalize(ox).bonds[8][(4, 0)] == rows
    for rel in (1e-11, 1e-2, 0.3):
        y, dt, _ = nat.truncate(ctx, x, rel * nrm)
        oy, odt, _ = OB.truncate(ox, rel * nrm)
        assert y.bonds() == oy.bonds
        assert abs(dt - odt) <= 1e-12 * nrm
        assert rel_distance(OB.BSMPS.from_flat([0] * K, (N, 0), y.bonds(), y.export()), oy) <= 1e-12


@pytest.mark.parametrize("sites,r,D", [(4, 4, 3), (8, 4, 17), (12, 4, 33), (12, 6, 40), (12, 4, 70)])
def test_joint_iterates_of_few_rows_and_many_vectors(nat, ctx, sites, r, D):
    """Two rows over as many columns as vectors: sectors of two kept columns that are too long for the plain Jacobi,
    in launches that hold no wider ones."""
    wl_species, target = [0] * sites, (sites // 2, 0)
    n = nat.mps_joint_random_size(sites, 0, sites // 2, 0, r, D)
    vals = np.random.default_rng(D).standard_normal(n)
    x = nat.mps_create_joint(ctx, sites, 0, sites // 2, 0, D, r_max=r, values=vals)
    ox = OB.BSMPS.from_flat(wl_species, target, OB.default_dims(wl_species, target, r, D), vals)
    assert x.bonds() == ox.bonds
    nrm = float(np.sqrt(sum(np.sum(B * B) for B in OB.left_orthogonalize(ox).cores[-1].values())))
    for rel in (1e-11, 1e-1):
        y, dt, _ = nat.truncate(ctx, x, rel * nrm)
        oy, odt, _ = OB.truncate(ox, rel * nrm)
        assert y.bonds() == oy.bonds
        assert abs(dt - odt) <= 1e-12 * nrm
        assert rel_distance(OB.BSMPS.from_flat(wl_species, target, y.bonds(), y.export()), oy) <= 1e-12
