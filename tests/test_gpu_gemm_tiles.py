"""The FP64 products of TT rounding over ranks that take every tile of the GEMM, its transposed form and its
slices: a random TT added to itself rounds back to its own ranks and to twice its tensor (1e-12: the
rounding's QR stops at 1e-13 of the norm here, and nothing of the tensor itself is that small)."""
import numpy as np
import pytest

import oracle.pttk_oracle as o
from paper_2406_06344_gb300 import workloads as W
from tests.test_oracle_pins import tt_sum

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mid", [(1, 2, 2, 1), (2, 6, 5, 3), (3, 11, 13, 4), (6, 22, 31, 7), (9, 39, 45, 8),
                                 (10, 66, 79, 10)])
def test_doubled_tt_rounds_back(mid):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2406_06344_gb300 import pttk as P
    P.load()
    n, ranks = 10, (1, *mid, 1)
    rng = np.random.default_rng(sum(mid))
    cores = [rng.standard_normal((ranks[k], n, ranks[k + 1])) / np.sqrt(ranks[k] * n) for k in range(5)]
    tt = P.TT.from_cores(W.GAUSS, 2, ((0.0, 1.0),) * 2, ((2.0, 3.0), (0.0, 1.0)), 1, ((0.5, 2.0),), n, tt_sum(cores, cores))
    rt = tt.round(1e-9)
    assert rt.ranks == list(ranks)
    X2 = 2.0 * o.tt_full(cores)
    assert o.rel_fro(X2, o.tt_full(rt.cores())) <= 1e-12
