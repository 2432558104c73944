"""V^T w keeps every serial sum of 256 rows to chains of at most 64. The entries are m = 2^(p - 6) - 3 (p the type's
significant bits): sums of up to 64 of them are exact, and so are the sums of equal powers of two of those, while a
chain that goes on past 64 terms loses low bits. U and M are identities, so the product must be exactly 256 m."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("rt,rows", [(12, 256), (63, 256), (260, 256), (516, 256), (1028, 256), (514, 65536)])
@pytest.mark.parametrize("off", [0, 1])
def test_chains_of_at_most_64(prec, rt, rows, off):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2406_06344_gb300 import pttk as P
    P.load()
    dt, bits = (torch.float64, 53) if prec == "fp64" else (torch.float32, 24)
    m = float(2 ** (bits - 6) - 3)
    V = torch.full((rows * rt + off,), m, device="cuda", dtype=dt)[off:].view(rows, rt)
    w = torch.zeros(rows, device="cuda", dtype=dt)
    w[:256] = 1.0
    eye = torch.eye(rt, device="cuda", dtype=dt)
    assert bool((P.apply(eye, eye, V, w) == 256.0 * m).all())
