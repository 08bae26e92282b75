"""Flops of the terms (2 m n k each) and flops run by the zip-up contraction, against counts from the block
dims alone: contributions of an output that read the same block of x are summed before they are multiplied in
outputs of more than 32 rows or columns (smaller ones may take either kernel), 64 descriptors at a time."""
import numpy as np
import pytest

from oracle import bsmps as OB
from synth import hubbard_chain, random_block_values, spinless_random_chain
from tests._common import n_random, oracle_mpo, oracle_random

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nat():
    from paper_2604_16118_gb300 import build, native
    build.build()
    return native


def outputs(mpo, x, shift):
    """(rows, columns, [(occupation, k) of every contribution, occupation 0 first]) of every block product of the
    contraction (OB.apply_zipup's loops on dims)."""
    segs = OB._exact_segments(mpo, x)
    C = {m: v[1] for m, v in segs[0].items()}
    for t in range(x.K):
        ents, rows = mpo.entries(t, shift), {}
        for m, r in C.items():
            left = {a: n for a, n, _, _ in segs[t][m][0]}
            for so in (0, 1):
                m2 = OB.add_charge(m, OB.delta(x.species[t], so))
                if m2 not in segs[t + 1]:
                    continue
                rows[m2] = rows.get(m2, 0) + r
                for b, nb, _, cols in segs[t + 1][m2][0]:
                    ins = sorted((ei, x.bonds[t][left[a]]) for a, bb, eo, ei, _ in ents
                                 if bb == b and eo == so and a in left and (left[a], ei) in x.cores[t])
                    yield r, cols, ins
        C = {m2: min(r, segs[t + 1][m2][1]) for m2, r in rows.items()}


def run_flops(M, N, ins):
    total, c = 0.0, 0
    while c < len(ins):
        v = c + 1
        while v < len(ins) and v % 64 and ins[v] == ins[c]:
            v += 1
        k, n = ins[c][1], v - c
        total += 2.0 * M * N * k + (2.0 * M * k * n * -(-N // 32) if n > 1 else 0.0)
        c = v
    return total


@pytest.mark.parametrize("wl,r", [(spinless_random_chain(K=12, N=6, seed=1), 200), (hubbard_chain(L=8), 300)])
def test_contraction(nat, wl, r):
    ctx = nat.Context(0)
    vals = random_block_values(n_random(wl, r), 3)
    x = nat.mps_create(ctx, wl.n_orb, wl.spin, wl.n_up, wl.n_dn, r, vals)
    W = nat.mpo_from_integrals(ctx, wl.h, wl.eri, wl.spin, wl.n_particles, 4.0)
    ctx.profile(True)
    nat.apply_zipup(ctx, W, x, shift=-70.0)
    run, terms = ctx.kernel_executed(), {k: v[2] for k, v in ctx.kernel_stats(reset=True).items()}
    ctx.profile(False)
    out = list(outputs(oracle_mpo(wl, 4.0), oracle_random(wl, r, vals), -70.0))
    each = [(M, N, sum(2.0 * M * N * k for _, k in ins), run_flops(M, N, ins)) for M, N, ins in out]
    assert np.isclose(terms["apply"], sum(f for _, _, f, _ in each), rtol=1e-12)
    most = sum(f if max(M, N) <= 32 else g for M, N, f, g in each)
    least = sum(min(f, g) for _, _, f, g in each)
    assert least * (1 - 1e-12) <= run["apply"] <= most * (1 + 1e-12)
    assert most < terms["apply"]
    assert run["apply_qr"] == terms["apply_qr"]
    assert not any(ctx.kernel_executed().values())


def test_inner_product(nat):
    """Environment updates sum the blocks that a block of the iterate meets: fewer flops run than terms."""
    wl = spinless_random_chain(K=12, N=6, seed=1)
    ctx = nat.Context(0)
    x = nat.mps_create(ctx, wl.n_orb, 0, wl.n_up, 0, 100, random_block_values(n_random(wl, 100), 3))
    W = nat.mpo_from_integrals(ctx, wl.h, wl.eri, 0, wl.n_particles, 4.0)
    ctx.profile(True)
    nat.dot(ctx, x, x, W, -0.5)
    run, terms = ctx.kernel_executed()["gemm"], ctx.kernel_stats(reset=True)["gemm"][2]
    assert 0.0 < run < 0.8 * terms
