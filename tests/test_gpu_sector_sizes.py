"""Truncations whose charge sectors cross the sizes at which the factorisations
change their path (kept columns 16/17, 24/25, 32/33, 40/41, 56/57 and 64/65 of the
one-CTA SVD, stacks of more than 48 columns on clusters, more than 256 rows), tall
and wide, with flat and graded spectra and with linearly dependent columns,
against the oracle's truncation.

Bounds as for every truncation of this library: kept dims equal, the
represented tensors within 1e-12 of the norm."""
import numpy as np
import pytest

from oracle import bsmps as OB
from synth import hubbard_chain, random_block_values, spinless_random_chain
from tests._common import n_random, oracle_random, rel_distance, species_of, target_of, to_oracle

pytestmark = pytest.mark.gpu

SIZES = [(13, 6, 90), (14, 7, 110), (16, 7, 130), (17, 8, 300), (18, 9, 160), (18, 9, 230), (19, 9, 180),
         (19, 9, 240)]


@pytest.fixture(scope="module")
def nat():
    from paper_2604_16118_gb300 import build, native
    build.build()
    return native


@pytest.fixture(scope="module")
def ctx(nat):
    return nat.Context(0)


def truncated_widths(x):
    """Kept columns of every sector SVD of the right sweep of x (left-orthogonalised dims)."""
    lo = OB.left_orthogonalize(x)
    return sorted({d for b in lo.bonds for d in b.values()})


@pytest.mark.parametrize("K,N,r", SIZES)
@pytest.mark.parametrize("decay", [0.0, 0.25])
def test_truncation_over_sector_sizes(nat, ctx, K, N, r, decay):
    wl = spinless_random_chain(K=K, N=N, seed=K)
    vals = random_block_values(n_random(wl, r), 11 * K)
    x = nat.mps_create(ctx, wl.n_orb, wl.spin, wl.n_up, wl.n_dn, r, vals)
    # graded spectra: occupied sites damped, as a preconditioner term does
    f0, f1 = np.ones(K), np.exp(-decay * np.arange(K) * np.arange(K) / K)
    xs = nat.scale_sites(ctx, x, f0, f1)
    ox = oracle_random(wl, r, vals)
    ox = OB.BSMPS(ox.species, ox.target, ox.bonds,
                  [{k: B * (f1[t] if k[1] else f0[t]) for k, B in c.items()} for t, c in enumerate(ox.cores)])
    nrm = float(np.sqrt(OB.dot(ox, ox)))
    for rel in (1e-2, 1e-5):
        y, dt, _ = nat.truncate(ctx, xs, rel * nrm)
        oy, odt, _ = OB.truncate(ox, rel * nrm)
        assert y.bonds() == oy.bonds
        assert abs(dt - odt) <= 1e-12 * nrm
        assert rel_distance(to_oracle(wl, y), oy) <= 1e-12


def test_sizes_cross_every_path(nat):
    widths = set()
    for K, N, r in SIZES:
        wl = spinless_random_chain(K=K, N=N, seed=K)
        widths |= set(truncated_widths(oracle_random(wl, r, random_block_values(n_random(wl, r), 11 * K))))
    for lo, hi in [(1, 16), (17, 24), (25, 32), (33, 40), (41, 56), (57, 64), (65, 400)]:
        assert any(lo <= w <= hi for w in widths), (lo, hi, sorted(widths))


@pytest.mark.parametrize("K,N,r", [(12, 6, 40), (15, 7, 120)])
def test_linearly_dependent_columns(nat, ctx, K, N, r):
    """x + x: every stack has twice the columns and half of them depend on the others."""
    wl = spinless_random_chain(K=K, N=N, seed=3)
    vals = random_block_values(n_random(wl, r), 5)
    x = nat.mps_create(ctx, wl.n_orb, wl.spin, wl.n_up, wl.n_dn, r, vals)
    ox = oracle_random(wl, r, vals)
    nrm = float(np.sqrt(OB.dot(ox, ox)))
    y, _, _ = nat.truncate(ctx, nat.add(ctx, x, x, 1.0, 1.0), 1e-6 * nrm)
    o1, _, _ = OB.truncate(OB.add(ox, ox, 1.0, 1.0), 1e-6 * nrm)
    assert y.bonds() == o1.bonds
    assert rel_distance(to_oracle(wl, y), o1) <= 1e-12


@pytest.mark.parametrize("L,r", [(6, 60), (8, 120)])
def test_wide_and_tall_sectors_of_an_application(nat, ctx, L, r):
    wl = hubbard_chain(L=L)
    from oracle import mpo as OM
    vals = random_block_values(n_random(wl, r), 2)
    x = nat.mps_create(ctx, wl.n_orb, 1, wl.n_up, wl.n_dn, r, vals)
    W = nat.mpo_from_integrals(ctx, wl.h, wl.eri, 1, wl.n_particles, 4.0)
    oy = OB.apply_exact(OM.build_mpo(wl.h, wl.eri, 1, wl.n_particles, 4.0), oracle_random(wl, r, vals), shift=0.5)
    nrm = float(np.sqrt(OB.dot(oy, oy)))
    y, _ = nat.apply_H(ctx, W, x, shift=0.5, tol=1e-4 * nrm, r_max=r)
    ot, _, _ = OB.truncate(oy, 1e-4 * nrm, r)
    assert y.bonds() == ot.bonds
    assert rel_distance(to_oracle(wl, y), ot) <= 1e-12 * max(1.0, nrm / float(np.sqrt(OB.dot(ot, ot))))


def test_zero_iterate(nat, ctx):
    """Zero blocks: no division by a vanishing norm."""
    wl = spinless_random_chain(K=14, N=7, seed=1)
    z = nat.mps_create(ctx, wl.n_orb, 0, wl.n_up, 0, 110, np.zeros(n_random(wl, 110)))
    y, dt, _ = nat.truncate(ctx, z, 0.0)
    assert dt == 0.0 and np.all(np.isfinite(y.export()))


def with_spectrum(x, t, s_of):
    """x with the singular values of bond t replaced: sector q of width d takes s_of(d)."""
    rc, _, _ = OB.truncate(x, 0.0)                 # right-orthogonal
    lc = OB.left_orthogonalize(rc)
    assert lc.bonds == rc.bonds == x.bonds
    rng = np.random.default_rng(7)
    cores = [dict(c) for c in lc.cores[:t]] + [dict(c) for c in rc.cores[t:]]
    for q, d in x.bonds[t].items():
        u, _ = np.linalg.qr(rng.standard_normal((d, d)))
        v, _ = np.linalg.qr(rng.standard_normal((d, d)))
        C = (u * s_of(d)) @ v.T
        for key in cores[t]:
            if key[0] == q:
                cores[t][key] = C @ cores[t][key]
    return OB.BSMPS(x.species, x.target, x.bonds, cores)


@pytest.mark.parametrize("K,N", [(8, 4), (12, 6), (14, 7)])
@pytest.mark.parametrize("gap", [0.0, 1e-13, 1e-9, 1e-5])
def test_nearly_equal_singular_values(nat, ctx, K, N, gap):
    """Pairs of values a relative gap apart: rotations by large angles in the last sweeps, which a
    step of first order must not stand in for.  Nothing is cut: the tensor stays, and every core
    right of the first has orthonormal rows to k^2 eps (cosines up to k eps, k < 64)."""
    wl = spinless_random_chain(K=K, N=N, seed=2)
    r = 4096
    vals = random_block_values(n_random(wl, r), 9)
    ox = with_spectrum(oracle_random(wl, r, vals), K // 2,
                       lambda d: 10.0 ** (-0.3 * (np.arange(d) // 2)) * (1.0 + gap * (np.arange(d) % 2)))
    x = nat.mps_create(ctx, wl.n_orb, wl.spin, wl.n_up, wl.n_dn, r, ox.to_flat())
    y, dt, _ = nat.truncate(ctx, x, 0.0)
    oy = to_oracle(wl, y)
    assert dt == 0.0 and oy.bonds == ox.bonds
    assert rel_distance(oy, ox) <= 1e-12
    for t in range(1, K):
        for q, d in oy.bonds[t].items():
            rows = np.hstack([B for key, B in oy.cores[t].items() if key[0] == q])
            assert np.linalg.norm(rows @ rows.T - np.eye(d)) <= 1e-12
