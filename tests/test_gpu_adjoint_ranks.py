"""The one-kernel reverse pass of the adjoint at the edges of its forms (R_2 of 1 to 64 in its four padded
widths, 65 in the separate kernels; d = 1, 2, 3; n = 2 to 32), against torch's own differentiation of the
chain in FP64 on the same seeded cores. FP64: 1e-10 relative; FP32 (rounded bases and products of a
few hundred terms): 1e-4, as in the other adjoint tests."""
import numpy as np
import pytest

from paper_2406_06344_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2406_06344_gb300 import pttk as P
    P.load()
    return torch, P


def _cheb(torch, x, lo, hi, n):
    xh = (2 * x - lo - hi) / (lo - hi)
    T = [torch.ones_like(xh), xh]
    for _ in range(2, n):
        T.append(2 * xh * T[-1] - T[-2])
    return torch.stack(T[:n], -1)


CASES = [(1, 2, (1, 2, 2, 1)), (1, 32, (1, 30, 9, 1)), (2, 5, (1, 4, 6, 7, 3, 1)), (2, 32, (1, 31, 40, 7, 3, 1)),
         (3, 4, (1, 3, 1, 5, 4, 6, 2, 1)), (3, 6, (1, 5, 17, 21, 8, 9, 4, 1)), (3, 12, (1, 9, 48, 50, 30, 60, 9, 1)),
         (3, 10, (1, 10, 64, 33, 30, 20, 9, 1)), (3, 10, (1, 10, 65, 33, 30, 20, 9, 1))]


@pytest.mark.parametrize("d,n,ranks", CASES)
@pytest.mark.parametrize("prec,tol", [("fp64", 1e-10), ("fp32", 1e-4)])
def test_gradients(env, d, n, ranks, prec, tol):
    torch, P = env
    rng = np.random.default_rng(3)
    dth = len(ranks) - 1 - 2 * d
    assert dth == 1
    cores = [rng.standard_normal((ranks[k], n, ranks[k + 1])) / np.sqrt(ranks[k] * n) for k in range(len(ranks) - 1)]
    box = ((0.0, 1.0),) * d
    tgt = ((2.0, 3.0),) + box[1:]
    tt = P.TT.from_cores(W.GAUSS, d, box, tgt, 1, ((0.5, 2.0),), n, cores)
    ns, nt = 333, 130
    dt = torch.float64 if prec == "fp64" else torch.float32
    X = torch.tensor(rng.random((ns, d)), device="cuda", dtype=dt)
    Y = torch.tensor(rng.random((nt, d)) + np.array([2.0] + [0.0] * (d - 1)), device="cuda", dtype=dt)
    w, z = (torch.tensor(rng.standard_normal(k), device="cuda", dtype=dt) for k in (ns, nt))
    L, dtheta, dX = P.grad(tt, [1.2], X, Y, w, z, prec)
    tt.check()
    G = [torch.tensor(c, device="cuda") for c in cores]
    x = X.double().requires_grad_(True)
    th = torch.tensor(1.2, dtype=torch.float64, device="cuda", requires_grad=True)
    S = torch.ones(ns, 1, dtype=torch.float64, device="cuda")
    for i in range(d):
        S = torch.einsum("pa,pj,ajb->pb", S, _cheb(torch, x[:, i], 0.0, 1.0, n), G[i])
    T = torch.ones(nt, 1, dtype=torch.float64, device="cuda")
    for i in reversed(range(d)):
        T = torch.einsum("pb,pj,ajb->pa", T, _cheb(torch, Y[:, i].double(), *tgt[i], n), G[d + 1 + i])
    H = torch.einsum("ajb,j->ab", G[d], _cheb(torch, th, 0.5, 2.0, n))
    Lr = w.double() @ (S @ (H @ (T.T @ z.double())))
    gx, gth = torch.autograd.grad(Lr, [x, th])
    scale = float((w.double().abs() @ (S.abs() @ (H.abs() @ (T.abs().T @ z.double().abs())))).detach())
    assert abs(L - float(Lr)) <= tol * scale
    assert abs(dtheta[0] - float(gth)) <= tol * max(abs(float(gth)), scale)
    assert (dX.double() - gx).norm() <= tol * gx.norm()
