"""The pivoted QR deals the columns left to its blocks by their number among those left, found from counts per 32 columns
and a bit mask. TT-Round of a random tensor train whose QRs have N columns, N around multiples of 32 and of
1,024 (32 words of counts): the tensor moves by at most tol ||T||_F (Algorithm 1), with as much again for the rounding of the
factorisations."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cols", [1, 2, 31, 32, 33, 64, 65, 992, 1023, 1024, 1025, 1100])
def test_round(cols):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2406_06344_gb300 import pttk as P
    P.load()
    n, r2, tol = 32, 40, 1e-12
    rng = np.random.default_rng(cols)
    cores = [rng.standard_normal((1, n, cols)), rng.standard_normal((cols, n, r2)) / np.sqrt(cols * n), rng.standard_normal((r2, n, 1))]
    tt = P.TT.from_cores(P.GAUSS, 1, ((0.0, 1.0),), ((2.0, 3.0),), 1, ((0.5, 2.0),), n, cores)
    rd = tt.round(tol)
    assert all(a <= b for a, b in zip(rd.ranks, [1, min(cols, n), min(r2, n), 1]))
    T, R = (np.einsum("iaj,jbk,kcl->abc", *c, optimize=True) for c in (cores, rd.cores()))
    assert np.linalg.norm(T - R) <= 2 * tol * np.linalg.norm(T)
