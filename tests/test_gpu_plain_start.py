"""bsmps_ctx_set_jacobi_precond(0): truncations in FP64 throughout, on every path of the sector SVDs (one SM: persistent
and per-site sweeps; clusters).  The two starts give the same truncation, but not the same roundings."""
import numpy as np
import pytest

from oracle import bsmps as OB
from synth import random_block_values, spinless_random_chain
from tests._common import n_random, oracle_random, rel_distance, to_oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nat():
    from paper_2604_16118_gb300 import build, native
    build.build()
    return native


@pytest.mark.parametrize("K,N,r", [(8, 4, 24), (12, 6, 48), (14, 7, 110), (16, 7, 130), (18, 9, 230)])
def test_off_means_fp64_throughout(nat, K, N, r):
    wl = spinless_random_chain(K=K, N=N, seed=K)
    vals = random_block_values(n_random(wl, r), 11 * K)
    ox = oracle_random(wl, r, vals)
    nrm = float(np.sqrt(OB.dot(ox, ox)))
    oy, odt, _ = OB.truncate(ox, 1e-2 * nrm)
    got = []
    for min_k in (0, 48):
        ctx = nat.Context(0)
        ctx.set_jacobi_precond(min_k)
        x = nat.mps_create(ctx, wl.n_orb, wl.spin, wl.n_up, wl.n_dn, r, vals)
        y, dt, _ = nat.truncate(ctx, x, 1e-2 * nrm)
        assert y.bonds() == oy.bonds
        assert abs(dt - odt) <= 1e-12 * nrm
        assert rel_distance(to_oracle(wl, y), oy) <= 1e-12
        got.append(y.export())
    assert not np.array_equal(got[0], got[1])
