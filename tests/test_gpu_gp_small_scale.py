"""K v in FP64 at length scales whose square or inverse leaves the range of a double: the kernel is 1 at r = 0 and 0 elsewhere, so
the product is exactly (1 + s2) v up to the rounding of one addition and one product."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kernel,l", [("GAUSS", 1e-154), ("GAUSS", 1e-100), ("EXPONENTIAL", 1e-310), ("EXPONENTIAL", 1e-300)])
@pytest.mark.parametrize("N", [1, 300])
def test_identity(kernel, l, N):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2406_06344_gb300 import pttk as P
    P.load()
    X = torch.linspace(0.0, 1.0, 2 * N, dtype=torch.float64, device="cuda").view(N, 2)
    v = torch.linspace(1.0, 2.0, N, dtype=torch.float64, device="cuda")
    out = P.gp_kv(getattr(P, kernel), X, [l], 0.25, v)
    assert bool(((out - 1.25 * v).abs() <= 4 * 2.0 ** -53 * v).all())
