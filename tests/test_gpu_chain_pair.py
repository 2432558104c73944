"""The SM-pair chain kernel (the default of the kind::f16 forms for d >= 2) at the edges of its tiles:
point counts around 128 and 256, ranks whose padding differs (quads of 4, output rows that are
odd, even, multiples of 4 and of 32), n that is no multiple of 4, one-quad steps, and output
buffers that are not 16-byte aligned. U and V are compared with the library's FP64 form on the same
(FP32) points and seeded cores; the tolerances are those of the forms' other tests."""
import numpy as np
import pytest

from paper_2406_06344_gb300 import workloads as W

pytestmark = pytest.mark.gpu

TOL = {"fp16x3": 1e-5, "bf16x3": 3e-5, "fp16": 2e-3, "bf16": 2e-2}


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2406_06344_gb300 import pttk as P
    P.load()
    return torch, P


def _tt(P, d, n, ranks, seed):
    rng = np.random.default_rng(seed)
    dth = len(ranks) - 1 - 2 * d
    cores = [rng.standard_normal((ranks[k], n, ranks[k + 1])) / np.sqrt(ranks[k] * n) for k in range(len(ranks) - 1)]
    box = ((0.0, 1.0),) * d
    th = ((0.5, 2.0), (0.5, 2.5))[:dth]
    return P.TT.from_cores(W.MATERN_NU if dth == 2 else W.GAUSS, d, box, ((2.0, 3.0),) + box[1:], dth, th, n, cores)


def _check(env, d, n, ranks, ns, nt, form, offset=0):
    torch, P = env
    tt = _tt(P, d, n, ranks, 11)
    dth = len(ranks) - 1 - 2 * d
    theta = (1.1, 1.3)[:dth]
    rng = np.random.default_rng(12)
    X = torch.tensor(rng.random((ns, d)), device="cuda", dtype=torch.float32)
    Y = torch.tensor(rng.random((nt, d)) + np.array([2.0] + [0.0] * (d - 1)), device="cuda", dtype=torch.float32)
    rs, rt = ranks[d], ranks[d + dth]
    U = torch.full((ns * rs + offset,), float("nan"), device="cuda")[offset:].view(ns, rs)
    V = torch.full((nt * rt + offset,), float("nan"), device="cuda")[offset:].view(nt, rt)
    P.instantiate(tt, theta, X, Y, form, U=U, V=V)
    tt.check()
    U64, _, V64 = P.instantiate(tt, theta, X.double(), Y.double(), "fp64")
    for got, want in ((U, U64), (V, V64)):
        if want.numel():
            assert (got.double() - want).norm() <= TOL[form] * want.norm()


@pytest.mark.parametrize("ns,nt", [(1, 0), (0, 1), (127, 129), (128, 256), (255, 257), (1000, 511), (40001, 39999)])
@pytest.mark.parametrize("d,n,ranks", [(2, 20, (1, 10, 63, 63, 12, 1)), (3, 12, (1, 9, 44, 177, 300, 180, 49, 10, 1))])
def test_point_counts(env, d, n, ranks, ns, nt):
    _check(env, d, n, ranks, ns, nt, "fp16x3")


@pytest.mark.parametrize("form", ["fp16x3", "bf16x3", "fp16", "bf16"])
@pytest.mark.parametrize("d,n,ranks", [
    (2, 2, (1, 1, 1, 1, 1, 1)), (2, 5, (1, 4, 6, 64, 17, 1)), (2, 8, (1, 8, 250, 16, 2, 1)), (2, 13, (1, 13, 31, 33, 3, 1)),
    (2, 24, (1, 24, 48, 34, 16, 1)), (2, 28, (1, 7, 30, 36, 5, 1)), (2, 31, (1, 7, 30, 36, 5, 1)),
    (3, 4, (1, 3, 5, 16, 18, 4, 2, 1)), (3, 7, (1, 5, 17, 61, 40, 62, 16, 7, 1)), (3, 12, (1, 12, 64, 192, 100, 128, 33, 1, 1)),
    (3, 10, (1, 10, 52, 100, 30, 101, 4, 6, 1)), (3, 16, (1, 9, 40, 96, 30, 160, 41, 9, 1))])
def test_ranks_and_orders(env, d, n, ranks, form):
    _check(env, d, n, ranks, 700, 300, form)


@pytest.mark.parametrize("offset", [1, 2, 3])
def test_unaligned_output(env, offset):
    _check(env, 2, 20, (1, 10, 63, 62, 12, 1), 600, 500, "fp16x3", offset)
