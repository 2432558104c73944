"""Workspace of a TT-SVD by parity sectors: no more than the two tensors that the factorisation of whole unfoldings takes
beside its copy of C (the transposed QR input and the projected tensor), also for an odd n with one symmetric dimension, whose
two sectors have (n + 1) / n times half of the tensor's entries. A fresh process leaves those three tensors free, and
5 % of one for granules and what does not grow with the tensor."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PROG = """
import sys
import torch
from paper_2406_06344_gb300 import pttk as P
n = int(sys.argv[1])
box = ((0.0, 1.0),) * 3, ((2.0, 3.0), (0.3, 1.3), (0.0, 1.0)), 2, ((0.5, 2.0), (0.5, 2.5))
def build(n):
    C = P.grid_coeffs(P.MATERN_NU, 3, *box, n)
    return C, lambda: P.TT.from_coeffs(P.MATERN_NU, 3, *box, n, 1e-6, C)
_, make = build(6)
make().free()           # every kernel is loaded, and the last handle's workspace given back
C, make = build(n)
torch.cuda.synchronize()
_, small = build(4)
small().free()
torch.cuda.synchronize()
fill = torch.empty(torch.cuda.mem_get_info()[0] - int(3.05 * 8 * C.numel()), dtype=torch.uint8, device="cuda")
print(make().ranks)
"""


@pytest.mark.parametrize("n", [11])
def test_three_tensors_are_room_enough(n):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    r = subprocess.run([sys.executable, "-c", PROG, str(n)], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
