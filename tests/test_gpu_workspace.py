"""The library keeps workspace between calls (up to 1 GiB) only while a handle lives, and 32 MiB otherwise. Each case runs in a
process of its own, and compares the free memory (within one granule of 32 MiB) before a call and after it and a
synchronisation."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HEAD = """
import torch
from paper_2406_06344_gb300 import pttk as P
dev = "cuda"
box3 = ((0.0, 1.0),) * 3, ((2.0, 3.0), (0.0, 1.0), (0.0, 1.0))
def free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]
GRANULE = 32 << 20
X, v = torch.rand(20000, 3, dtype=torch.float64, device=dev), torch.rand(20000, dtype=torch.float64, device=dev)
C = torch.empty(10 ** 8, dtype=torch.float64, device=dev)
def grid():
    P.grid_coeffs(P.MATERN_NU, 3, *box3, 2, ((0.5, 2.0), (0.5, 2.5)), 10, out=C)   # 200 MB of scratch
def small(tol=1e-8):
    return P.TT.build_offline(P.GAUSS, 1, ((0.0, 1.0),), ((0.0, 1.0),), 1, ((0.5, 2.0),), 8, tol)
"""


def run(body):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    r = subprocess.run([sys.executable, "-c", HEAD + body], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr


def test_calls_without_a_handle_keep_nothing():
    run("""
small().free()
grid()
P.gp_kv(P.GAUSS, X, [0.7], 0.1, v)
base = free()
grid()
P.gp_kv(P.GAUSS, X, [0.7], 0.1, v)
after = free()
assert base >= torch.cuda.mem_get_info()[1] * 0.5 and abs(base - after) <= GRANULE
keep = small()
grid()
held = base - free()
assert held >= 4 * GRANULE, held      # with a handle the scratch stays
keep.free()
torch.cuda.synchronize()
grid()
assert base - free() <= GRANULE, base - free()
""")


@pytest.mark.parametrize("kind", ["global", "fixed"])
def test_last_handle_of_any_kind(kind):
    """A Global or a Fixed that outlives its tensor train keeps the workspace, and gives it back when it goes, also
    where the work that used it is still running at that moment."""
    run("KIND = %r" % kind + """
tt = small()
Z = torch.rand(100, 1, dtype=torch.float64, device=dev)
h = P.Global(tt, Z) if KIND == "global" else P.Fixed(tt, Z, Z, 1e-6)
tt.free()
grid()
base = free()
grid()
h.free()          # the scratch is in use
assert free() - base >= 4 * GRANULE, free() - base
""")
