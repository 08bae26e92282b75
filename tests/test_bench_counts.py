"""What bench.py counts and on what its reference arm runs (no GPU needed)."""
import os
import re

import pytest

import bench

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_emulated_product_counts_the_products_it_issues():
    src = open(os.path.join(ROOT, "paper_2604_16118_gb300", "csrc", "ozaki.cu")).read()
    # the instance launched for 8 slices: k_oz_gemm<digits, bits>, with digit pairs p + q <= digits + 1
    digits, bits = map(int, re.search(r"default: launch_oz_gemm<(\d+), (\d+)>", src).groups())
    assert digits * bits == 56
    assert bench.ozaki_products(8) == sum(1 for p in range(1, digits + 1) for q in range(1, digits + 1)
                                          if p + q <= digits + 1)
    for s in range(1, 8):
        assert f"case {s}: launch_oz_gemm<{s}>" in src
        assert bench.ozaki_products(s) == s * (s + 1) // 2


def test_reference_arm_loads_nothing_of_the_library():
    import json
    import subprocess
    import sys
    code = ("import sys, json; sys.argv = ['bench.py', '--impl', 'reference', '--steps', '1', '--warmup', '3']\n"
            "import bench; f = bench.oracle_apply_times\n"
            "bench.oracle_apply_times = lambda cores, reps: f(cores, reps=reps, L=4, r=6)\n"
            "assert bench.main() == 0\n"
            "assert not [m for m in sys.modules if m.startswith('paper_2604_16118_gb300')]\n"
            "assert 'libbsmps' not in open('/proc/self/maps').read()\n")
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    line = json.loads(r.stdout.strip().splitlines()[-1])
    assert line["impl"] == "reference" and line["value"] > 0.0 and "note" not in line


@pytest.mark.gpu
@pytest.mark.parametrize("L,r", [(4, 6), (8, 300)])
def test_reference_arm_counts_as_the_library_does(L, r):
    from paper_2604_16118_gb300 import build, native as nat
    from synth import hubbard_chain, random_block_values
    from tests._common import n_random, oracle_mpo, oracle_random
    build.build()
    ctx = nat.Context(0)
    wl = hubbard_chain(L=L)
    vals = random_block_values(n_random(wl, r), 3)
    S = {"x": nat.mps_create(ctx, wl.n_orb, wl.spin, wl.n_up, wl.n_dn, r, vals),
         "W": nat.mpo_from_integrals(ctx, wl.h, wl.eri, wl.spin, wl.n_particles, 4.0)}
    assert bench.apply_flops_per_branch(nat, ctx, S) == bench.zipup_flops(oracle_mpo(wl, 4.0),
                                                                          oracle_random(wl, r, vals), -70.0)
