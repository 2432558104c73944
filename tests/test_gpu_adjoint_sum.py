"""The last sum of each point derivative, over T_j'(x) of one coordinate, is in FP64 in every form with FP32 points. With all
ranks 1, every core but the tested coordinate's the constant 1, that one's coefficients small integers, and w and z powers of two,
everything before that sum is exact: the result may differ from the FP64 value by its rounding to FP32 and by the rounding
of the FP64 recurrences alone (64 n eps of the sum of the terms' largest sizes, 2 |c_j| j^2 on the unit box)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp32", "tf32", "tf32x3", "bf16", "bf16x3", "fp16", "fp16x3"])
@pytest.mark.parametrize("d,which", [(1, 0), (2, 0), (2, 1), (3, 0), (3, 1), (3, 2)])
@pytest.mark.parametrize("n", [2, 12, 32])
def test_sum_over_derivatives(prec, d, which, n):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2406_06344_gb300 import pttk as P
    P.load()
    rng = np.random.default_rng(100 * d + 10 * which + n)
    one = np.zeros((1, n, 1))
    one[0, 0, 0] = 1.0
    c = rng.integers(-8, 9, n).astype(float)
    cores = [one] * which + [c.reshape(1, n, 1)] + [one] * (2 * d - which)
    src, tgt = ((0.0, 1.0),) * d, ((2.0, 3.0),) + ((0.0, 1.0),) * (d - 1)
    tt = P.TT.from_cores(P.GAUSS, d, src, tgt, 1, ((0.5, 2.0),), n, cores)
    ns = 1000
    X = torch.tensor(rng.random((ns, d)), device="cuda", dtype=torch.float32)
    Y = torch.tensor([[2.5] + [0.5] * (d - 1)], device="cuda", dtype=torch.float32)
    w = torch.tensor(2.0 ** rng.integers(-3, 4, ns), device="cuda", dtype=torch.float32)
    _, _, dX = P.grad(tt, [1.2], X, Y, w, torch.ones(1, device="cuda"), prec)
    x = X[:, which].double().cpu().numpy()
    ref = w.double().cpu().numpy() * np.polynomial.chebyshev.chebval(1.0 - 2.0 * x, np.polynomial.chebyshev.chebder(c)) * -2.0
    slack = w.double().cpu().numpy() * (64 * n * 2.0 ** -53 * 2.0 * float(np.abs(c) @ np.arange(n) ** 2))
    got = dX.double().cpu().numpy()
    assert (np.abs(got[:, which] - ref) <= 2.0 ** -24 * np.abs(ref) + slack).all()
    assert (np.delete(got, which, axis=1) == 0.0).all()
