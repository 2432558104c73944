"""TT-SVD by parity sectors: coefficient tensors whose source and target boxes share their centre in
none, some or all dimensions, odd and even n, tolerances from loose (sectors with no kept direction) to
tight, against the oracle's TT-SVD of the same tensor (equal ranks), the truncation bound
||C - TT|| <= tol ||C||, and left-orthonormal cores to 1e-12 (rounding of products of up to a few hundred
terms)."""
import numpy as np
import pytest

import oracle.pttk_oracle as o
from paper_2406_06344_gb300 import workloads as W

pytestmark = pytest.mark.gpu

B = (0.0, 1.0)
CASES = [
    (W.GAUSS, 1, 9, (B,), (B,)), (W.GAUSS, 1, 12, (B,), ((2.0, 3.0),)), (W.MULTIQUADRIC, 1, 16, (B,), ((-1.0, 2.0),)),
    (W.MATERN32, 2, 6, (B, B), ((2.0, 3.0), B)), (W.MATERN52, 2, 7, (B, B), ((2.0, 3.0), B)), (W.GAUSS, 2, 8, (B, B), (B, B)),
    (W.MULTIQUADRIC, 2, 5, (B, B), (B, (2.0, 3.0))), (W.LAPLACE3D, 2, 8, (B, B), ((2.0, 3.0), B)),
    (W.GAUSS, 3, 4, (B, B, B), (B, B, B)), (W.MATERN32, 3, 5, (B, B, B), ((3.0, 4.0), B, B)), (W.MATERN_NU, 2, 5, (B, B), ((2.0, 3.0), B)),
]


@pytest.mark.parametrize("tol", [1e-1, 1e-4, 1e-8])
@pytest.mark.parametrize("kernel,d,n,src,tgt", CASES)
def test_sectors(kernel, d, n, src, tgt, tol):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2406_06344_gb300 import pttk as P
    P.load()
    dth = 2 if kernel == W.MATERN_NU else 0 if kernel in (W.LAPLACE3D,) else 1
    theta = ((0.5, 2.0), (0.5, 2.5))[:dth]
    C = P.grid_coeffs(kernel, d, src, tgt, dth, theta, n, "fp64")
    tt = P.TT.from_coeffs(kernel, d, src, tgt, dth, theta, n, tol, C)
    D = 2 * d + dth
    Ch = C.cpu().numpy().reshape((n,) * D, order="F")
    _, ranks = o.tt_svd(Ch, tol)
    assert tt.ranks == list(ranks)
    cores = tt.cores()
    full = cores[0]
    for G in cores[1:]:
        full = np.tensordot(full, G, axes=([-1], [0]))
    full = full.reshape((n,) * D)
    assert np.linalg.norm(full - Ch) <= tol * np.linalg.norm(Ch) * (1 + 1e-6)
    for G in cores[:-1]:
        M = G.reshape(-1, G.shape[2])
        assert np.abs(M.T @ M - np.eye(M.shape[1])).max() <= 1e-12
