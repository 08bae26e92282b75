"""Device memory that a call takes beside its inputs and results: what the context's pool
holds after the call, in a process of its own (the pool keeps what it once reserved)."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
MB = 1 << 20

HEAD = """
import numpy as np, torch
from paper_2604_16118_gb300 import build, native as nat
build.build()
ctx = nat.Context(0)
{setup}
ctx.sync()
free = torch.cuda.mem_get_info()[0]
{call}
ctx.sync()
print("TAKEN", free - torch.cuda.mem_get_info()[0])
"""


def taken(setup, call):
    r = subprocess.run([sys.executable, "-c", HEAD.format(setup=setup, call=call)], cwd=ROOT, capture_output=True,
                       text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    return int(r.stdout.split("TAKEN")[1])


def test_narrow_network_on_a_large_batch():
    """Two inputs, two outputs, batch 2^21: eight arrays of the batch (16 MB each, rounded up to 64 MB by
    the pool), and the operand images whose rows are the batch, padded to 32 values (256 MB each, two)."""
    call = "net.loss_grad(x, x)"
    setup = "x = np.ones((1 << 21, 2), np.float32); net = nat.MLP(ctx, [2, 2], np.ones(6, np.float32))"
    assert taken(setup, call) <= 2 * 256 * MB + 8 * 64 * MB


def test_thin_emulated_product():
    """One row times one column over 2^22 values of k: 16 bytes of slices a value (two factors), 64 MB aside."""
    setup = "A = torch.ones(1, 1 << 22, dtype=torch.float64, device='cuda'); B = A.T.contiguous(); C = A[:, :1].clone()"
    assert taken(setup, "nat.gemm_ozaki(ctx, A, B, C)") <= 2 * 16 * (4 * MB) + 64 * MB


def test_thin_split_product():
    """Two rows times two columns over 2^20 values of k: 8 bytes of parts a value, 64 MB aside."""
    setup = "A = torch.ones(2, 1 << 20, dtype=torch.float64, device='cuda'); B = A.T.contiguous(); C = A[:, :2].clone()"
    assert taken(setup, "nat.gemm_tf32x3(ctx, A, B, C)") <= 4 * 8 * MB + 64 * MB


def test_split_product_without_room_for_its_parts():
    """The device full up to half of the workspace of the product: it runs on the kernel that needs none."""
    setup = """
n, k = 2048, 65536
g = torch.Generator(device="cuda").manual_seed(1)
A = torch.randn(n, k, dtype=torch.float64, device="cuda", generator=g)
B = torch.randn(k, n, dtype=torch.float64, device="cuda", generator=g)
C = torch.empty(n, n, dtype=torch.float64, device="cuda")
nat.gemm_tf32x3(ctx, A[:64, :64], B[:64, :64], C[:64, :64])
full = torch.empty(torch.cuda.mem_get_info()[0] - 8 * n * k, dtype=torch.uint8, device="cuda")
"""
    check = """
ctx.sync()
del full
torch.cuda.empty_cache()
R, S = A[:100] @ B, A[:100].abs() @ B.abs()
assert ((C[:100] - R).abs() <= 2.0 ** -21 * (4 + k ** 0.5) * S).all()
"""
    taken(setup, "nat.gemm_tf32x3(ctx, A, B, C)" + check)


def test_few_rows_and_short_sums_take_no_parts():
    """One row times 2^20 columns, one value of k: the kernel without a workspace (a list of 2^14 tiles)
    is the faster one there."""
    setup = "A = torch.ones(1, 1, dtype=torch.float64, device='cuda'); B = torch.ones(1, MB, dtype=torch.float64, " \
            "device='cuda'); C = B.clone()".replace("MB", str(MB))
    assert taken(setup, "nat.gemm_tf32x3(ctx, A, B, C)") <= 64 * MB


def test_import_and_write_of_a_large_iterate():
    """Eight blocks of 3000 x 3000 (576 MB): the calls need 64 MB at most beside the iterate, and the values
    come back as they went in."""
    setup = """
d = 3000
bonds = [{(0, 0): 1}, {(0, 0): d, (1, 0): d}, {(0, 0): d, (1, 0): d, (2, 0): d}, {(1, 0): d, (2, 0): d}, {(2, 0): 1}]
n = 8 * d * d + 4 * d
v = np.random.default_rng(1).standard_normal(n)
base = torch.cuda.mem_get_info()[0]
x = nat.mps_import(ctx, 4, 0, 2, 0, bonds, v)
x.write(v[::-1].copy())
assert base - torch.cuda.mem_get_info()[0] <= 8 * n + 4 * 64 * 2 ** 20, base - torch.cuda.mem_get_info()[0]
assert np.array_equal(x.export(), v[::-1])
"""
    taken(setup, "")


def test_export_without_room_for_a_second_buffer():
    """The device full but for half of the iterate: its cores are read one by one."""
    setup = """
d = 3000
bonds = [{(0, 0): 1}, {(0, 0): d, (1, 0): d}, {(0, 0): d, (1, 0): d, (2, 0): d}, {(1, 0): d, (2, 0): d}, {(2, 0): 1}]
n = 8 * d * d + 4 * d
v = np.random.default_rng(1).standard_normal(n)
x = nat.mps_import(ctx, 4, 0, 2, 0, bonds, v)
y = nat.scale_sites(ctx, x, np.ones(4), np.ones(4))     # (takes what the import may have left in the pool)
ctx.sync()
full = torch.empty(torch.cuda.mem_get_info()[0] - 4 * n, dtype=torch.uint8, device="cuda")
"""
    taken(setup, "assert np.array_equal(y.export(), v) and np.array_equal(x.export(), v)")


def test_large_and_small_cores_side_by_side():
    """Cores of 16 MB and more are copied by themselves, the others staged in between: every value arrives."""
    setup = """
for d in (1023, 1024, 1025, 2300):
    bonds = [{(0, 0): 1}, {(0, 0): 3, (1, 0): d}, {(0, 0): 2, (1, 0): d, (2, 0): d}, {(1, 0): d, (2, 0): 5},
             {(2, 0): 7}, {(2, 0): 1}]
    n = (3 + d) + (6 + 3 * d + d * d + d * d) + (2 * d + d * d + 5 * d + 5 * d) + (7 * d + 35) + 7
    v = np.random.default_rng(d).standard_normal(n)
    x = nat.mps_import(ctx, 5, 0, 2, 0, bonds, v)
    assert np.array_equal(x.export(), v)
    x.write(2.0 * v)
    assert np.array_equal(x.export(), 2.0 * v)
"""
    taken(setup, "")
