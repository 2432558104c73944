"""The symmetric FP64 kernel product (each pair of points evaluated once) against a dense product in
torch at the edges of its tiles (64 and 256 points, super tiles), for every kernel and dimension, with
values that underflow, and with a NaN point. Tolerance: the product's own rounding, 1e-13 of
sum_j |K_ij v_j| + s2 |v_i| (N eps is below that for these N)."""
import math

import numpy as np
import pytest

from paper_2406_06344_gb300 import workloads as W

pytestmark = pytest.mark.gpu

KERNELS = [W.GAUSS, W.MATERN32, W.EXPONENTIAL, W.MATERN52]


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2406_06344_gb300 import pttk as P
    P.load()
    return torch, P


def _dense(torch, kind, X, l):
    r2 = ((X[:, None, :] - X[None, :, :]) ** 2).sum(-1)
    r = r2.sqrt()
    if kind == W.GAUSS:
        return torch.exp(-r2 / (l * l))
    if kind == W.MATERN32:
        a = math.sqrt(3.0) * r / l
        return (1 + a) * torch.exp(-a)
    if kind == W.EXPONENTIAL:
        return torch.exp(-r / l)
    a = math.sqrt(5.0) * r / l
    return (1 + a + a * a / 3) * torch.exp(-a)


def _check(env, kind, d, N, l, scale=1.0):
    torch, P = env
    rng = np.random.default_rng(N + d)
    X = torch.tensor(scale * rng.random((N, d)), device="cuda")
    v = torch.tensor(rng.standard_normal(N), device="cuda")
    K = _dense(torch, kind, X, l)
    out = P.gp_kv(kind, X, [l], 0.3, v)
    ref = K @ v + 0.3 * v
    bound = K @ v.abs() + 0.3 * v.abs()
    assert ((out - ref).abs() <= 1e-13 * bound + 1e-300).all()


@pytest.mark.parametrize("N", [1, 2, 31, 32, 33, 63, 64, 65, 127, 129, 1000, 5700, 8500, 9000, 9217])
def test_sizes(env, N):
    _check(env, W.GAUSS, 3, N, 0.6)


@pytest.mark.parametrize("kind", KERNELS)
@pytest.mark.parametrize("d", range(1, 9))
def test_kernels_and_dimensions(env, kind, d):
    _check(env, kind, d, 700, 0.5)


@pytest.mark.parametrize("kind", KERNELS)
def test_values_that_underflow(env, kind):
    _check(env, kind, 2, 300, 0.01, scale=30.0)


def test_super_tiles(env):
    """25,000 points: super tiles of two 256-point tiles; sampled rows."""
    torch, P = env
    rng = np.random.default_rng(5)
    N = 25000
    X = torch.tensor(rng.random((N, 3)), device="cuda")
    v = torch.tensor(rng.standard_normal(N), device="cuda")
    out = P.gp_kv(W.MATERN32, X, [0.7], 0.1, v)
    for rows in torch.tensor([0, 255, 256, 511, 512, 513, 12799, 12800, 24575, 24999], device="cuda").split(5):
        r = ((X[rows][:, None, :] - X[None]) ** 2).sum(-1).sqrt()
        a = math.sqrt(3.0) * r / 0.7
        K = (1 + a) * torch.exp(-a)
        assert ((out[rows] - (K @ v + 0.1 * v[rows])).abs() <= 1e-13 * (K @ v.abs() + 1)).all()


def test_nan_point_reaches_every_row(env):
    torch, P = env
    X = torch.rand(100, 2, dtype=torch.float64, device="cuda")
    X[40, 1] = float("nan")
    out = P.gp_kv(W.GAUSS, X, [0.5], 0.1, torch.ones(100, dtype=torch.float64, device="cuda"))
    assert out.isnan().all()
