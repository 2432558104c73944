"""Grid coefficients where source and target boxes have the same centre in some dimensions (the folded
path), with odd and even n, boxes of different width, and every kernel of the path, against the
oracle. Tolerances are those of the other grid tests: 1e-13 of max|C| in FP64, 1e-5 in FP32; entries
whose parity the symmetry forbids are exactly zero."""
import numpy as np
import pytest

import oracle.pttk_oracle as o
from paper_2406_06344_gb300 import workloads as W

pytestmark = pytest.mark.gpu

B = (0.0, 1.0)
CASES = [
    # kernel, d, n, source boxes, target boxes (equal centres: none, some or all dimensions)
    (W.GAUSS, 1, 7, (B,), (B,)), (W.GAUSS, 1, 8, (B,), ((-1.0, 2.0),)), (W.MATERN32, 1, 32, (B,), (B,)), (W.MATERN32, 1, 2, (B,), (B,)),
    (W.EXPONENTIAL, 2, 5, (B, B), ((2.0, 3.0), (0.25, 0.75))), (W.MATERN52, 2, 6, (B, B), (B, (2.0, 3.0))),
    (W.MULTIQUADRIC, 2, 9, (B, B), (B, B)), (W.GAUSS, 2, 10, (B, (-1.0, 1.0)), ((2.0, 3.0), (-3.0, 3.0))),
    (W.THIN_PLATE_SPLINE, 2, 4, (B, B), ((1.5, 2.5), B)), (W.LAPLACE3D, 2, 7, (B, B), ((2.0, 3.0), B)),
    (W.MATERN_NU, 1, 9, (B,), (B,)), (W.MATERN_NU, 2, 5, (B, B), ((2.0, 3.0), B)), (W.MATERN_NU, 2, 6, (B, B), ((0.1, 1.1), B)),
    (W.GAUSS, 3, 5, (B, B, B), (B, B, B)), (W.MATERN32, 3, 4, (B, B, B), ((3.0, 4.0), B, B)), (W.GAUSS, 3, 4, (B, B, B), (B, (2.0, 3.0), B)),
]


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-13), ("fp32", 1e-5)])
@pytest.mark.parametrize("kernel,d,n,src,tgt", CASES)
def test_folded_coefficients(kernel, d, n, src, tgt, prec, tol):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2406_06344_gb300 import pttk as P
    P.load()
    dth = 2 if kernel == W.MATERN_NU else 0 if kernel in (W.LAPLACE3D,) else 1
    theta = ((0.5, 2.0), (0.5, 2.5))[:dth]
    C = P.grid_coeffs(kernel, d, src, tgt, dth, theta, n, prec).double().cpu().numpy()
    D = 2 * d + dth
    C = C.reshape((n,) * D, order="F")
    boxes = np.array(list(src) + list(theta) + list(tgt))
    with np.errstate(invalid="ignore"):
        M = o.grid_tensor(o.kernel_f(kernel), d, dth, boxes, n)
    if kernel == W.MATERN_NU:
        M = np.where(np.isnan(M), 1.0, M)   # the oracle's z^nu K_nu(z) at z = 0, whose limit gives kappa = 1
    ref = o.coefficient_tensor(M, n)
    assert np.abs(C - ref).max() <= tol * np.abs(ref).max()
    for j in range(d):
        if sum(src[j]) == sum(tgt[j]):
            i = np.arange(n)
            odd = (i[:, None] + i[None, :]) % 2 == 1
            assert not np.moveaxis(C, (j, d + dth + j), (0, 1))[odd].any()
