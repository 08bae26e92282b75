"""What bench.py counts and on what its reference arm runs (no GPU needed)."""
import os
import re

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
