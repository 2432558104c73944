"""Grid coefficients where the launch changes form: one tile or several (around 4096 entries), the length scales of a point pair
over 1 to n threads, few or many indices a block in the folded modes' expansion, kernels with and without a fast form, and
length scales whose inverse overflows. Oracle and tolerances as in the other grid tests: 1e-13 of max|C| in FP64,
1e-5 in FP32."""
import numpy as np
import pytest

import oracle.pttk_oracle as o
from paper_2406_06344_gb300 import workloads as W

pytestmark = pytest.mark.gpu

B, G = (0.0, 1.0), (0.13, 1.21)
CASES = [(W.THIN_PLATE_SPLINE, 1, 32, (B,), (B,)), (W.MATERN52, 1, 24, (B,), (B,)), (W.GAUSS, 1, 16, (B,), (G,)), (W.EXPONENTIAL, 1, 15, (B,), (G,)),
         (W.GAUSS, 2, 12, (B, B), (B, B)), (W.MATERN32, 2, 13, (B, B), ((2.0, 3.0), G)), (W.MULTIQUADRIC, 2, 8, (B, B), (G, B)),
         (W.LAPLACE3D, 3, 8, (B, B, B), ((2.0, 3.0), B, B)), (W.LAPLACE3D, 3, 5, (B, B, B), ((2.0, 3.0), G, B)),
         (W.BIHARMONIC, 2, 11, (B, B), ((2.0, 3.0), B)), (W.MATERN_NU, 2, 7, (B, B), ((2.0, 3.0), G)), (W.MATERN_NU, 1, 11, (B,), ((2.0, 3.0),))]


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-13), ("fp32", 1e-5)])
@pytest.mark.parametrize("kernel,d,n,src,tgt", CASES)
def test_coefficients(kernel, d, n, src, tgt, prec, tol):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2406_06344_gb300 import pttk as P
    P.load()
    dth = 2 if kernel == W.MATERN_NU else 0 if kernel in (W.LAPLACE3D, W.BIHARMONIC) else 1
    theta = ((0.5, 2.0), (0.5, 2.5))[:dth]
    C = P.grid_coeffs(kernel, d, src, tgt, dth, theta, n, prec).double().cpu().numpy().reshape((n,) * (2 * d + dth), order="F")
    ref = o.coefficient_tensor(o.grid_tensor(o.kernel_f(kernel), d, dth, np.array(list(src) + list(theta) + list(tgt)), n), n)
    assert np.abs(C - ref).max() <= tol * np.abs(ref).max()


def test_scales_whose_inverse_overflows():
    """exp(-r / l) is 1 at r = 0 and 0 elsewhere, whatever l."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2406_06344_gb300 import pttk as P
    P.load()
    n = 4
    C = P.grid_coeffs(W.EXPONENTIAL, 1, (B,), (B,), 1, ((1e-310, 2e-310),), n).cpu().numpy().reshape((n,) * 3, order="F")
    M = np.einsum("ik,j->ijk", np.eye(n), np.ones(n))
    assert np.abs(C - o.coefficient_tensor(M, n)).max() <= 1e-13
