"""A Fixed may be freed while the copy that factors() has queued still waits for its stream: freeing its factors
waits for the copy. (The other stream's allocations would otherwise be handed the memory and overwrite it.)"""
import pytest

pytestmark = pytest.mark.gpu


def test_free_behind_a_queued_copy():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2406_06344_gb300 import pttk as P
    P.load()
    tt = P.TT.build_offline(P.GAUSS, 1, ((0.0, 1.0),), ((0.0, 1.0),), 1, ((0.5, 2.0),), 12, 1e-8)
    X = torch.rand(30011, 1, dtype=torch.float64, device="cuda")
    F = P.Fixed(tt, X, X, 1e-8)
    S0, T0 = F.factors()
    torch.cuda.synchronize()
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        torch.cuda._sleep(100_000_000)   # about 50 ms
        S1, T1 = F.factors()
    F.free()
    Y = 1.0 - X
    other = P.Fixed(tt, Y, Y, 1e-8)
    torch.cuda.synchronize()
    assert torch.equal(S0, S1) and torch.equal(T0, T1)
    other.free()
