"""The ranks by parity sectors are those of one factorisation: the same coefficient tensor with a value of 1e-300
where a sector's zero stood takes the whole-unfolding path, and gives the same ranks at every tolerance (the
sectors' QRs keep the rows that one pivoted QR keeps, so also a tail within 1e-3 of the threshold counts alike)."""
import numpy as np
import pytest

from paper_2406_06344_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,n,kernel", [(2, 12, W.MATERN32), (2, 15, W.GAUSS), (3, 7, W.GAUSS), (3, 8, W.MATERN32)])
def test_sector_ranks(d, n, kernel):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2406_06344_gb300 import pttk as P
    P.load()
    src = ((0.0, 1.0),) * d
    tgt = ((1.75, 2.85),) + src[1:]
    args = (kernel, d, src, tgt, 1, ((0.5, 2.0),), n)
    C = P.grid_coeffs(*args, "fp64")
    whole = C.clone().reshape(-1)
    for j in range(1, d):
        assert float(whole[n ** j]) == 0.0
        whole[n ** j] = 1e-300
    for tol in np.geomspace(1e-5, 1e-9, 24):
        a, b = (P.TT.from_coeffs(*args, float(tol), c.reshape(C.shape)) for c in (C, whole))
        assert a.ranks == b.ranks, tol
        a.free()
        b.free()
