"""y = U (M (V^T w)) at the edges of the reads: V in units of 1, 2 or 4 rows, more than 256 units a group,
a base off the 16-byte boundary, few and many partial rows, tails of rows. The bound is the rounding of
the longest chain of sums (fewer than 512 additions at these sizes) on the product of absolute values."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rs,rt,ns,nt", [(1, 1, 1, 1), (3, 2, 5, 7), (7, 5, 33, 257), (12, 6, 1000, 1003),
                                         (177, 180, 4099, 4101), (64, 63, 9001, 9003), (5, 255, 2, 3001),
                                         (9, 1030, 130, 517), (8, 1021, 31, 12001)])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("off", [0, 1])
def test_apply(rs, rt, ns, nt, prec, off):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2406_06344_gb300 import pttk as P
    P.load()
    dt = torch.float64 if prec == "fp64" else torch.float32
    rng = np.random.default_rng(rs + rt)
    U, M, w = (torch.tensor(rng.standard_normal(k), device="cuda", dtype=dt) for k in ((ns, rs), (rs, rt), nt))
    V = torch.tensor(rng.standard_normal(nt * rt + off), device="cuda", dtype=dt)[off:].view(nt, rt)
    y = P.apply(U, M, V, w).double()
    Ud, Md, Vd, wd = U.double(), M.double(), V.double(), w.double()
    ref = Ud @ (Md @ (Vd.T @ wd))
    bound = Ud.abs() @ (Md.abs() @ (Vd.abs().T @ wd.abs()))
    assert bool(((y - ref).abs() <= 3 * 512 * torch.finfo(dt).eps * bound).all())
