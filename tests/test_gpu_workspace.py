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
