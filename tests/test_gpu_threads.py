"""Two host threads on streams of their own make calls that launch the same kernels with different amounts of shared memory and
take their scratch from the same pool: every call succeeds and gives bit for bit what it gives alone."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_two_threads():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2406_06344_gb300 import pttk as P
    P.load()
    box = ((0.0, 1.0),) * 3, ((2.0, 3.0), (0.0, 1.0), (0.0, 1.0)), 2, ((0.5, 2.0), (0.5, 2.5))
    rng = np.random.default_rng(5)

    def case(n, r, ns):
        cores = [rng.standard_normal((r[k], n, r[k + 1])) / np.sqrt(r[k] * n) for k in range(8)]
        tt = P.TT.from_cores(P.MATERN_NU, 3, *box, n, cores)
        X = torch.tensor(rng.uniform(0, 1, (ns, 3)), device="cuda", dtype=torch.float32)
        Y = X + torch.tensor([2.0, 0.0, 0.0], device="cuda")
        w = torch.tensor(rng.standard_normal(ns), device="cuda", dtype=torch.float32)
        Z = torch.tensor(rng.uniform(0, 1, (25000 if n == 12 else 300, 2)), device="cuda")
        z = torch.ones(Z.shape[0], device="cuda", dtype=torch.float64)

        def call(stream):
            s = stream.cuda_stream
            loss, dth, dX = P.grad(tt, [1.1, 1.3], X, Y, w, w, "fp32", stream=s)
            U, M, V = P.instantiate(tt, [1.1, 1.3], X, Y, "fp32", stream=s)
            out = P.apply(U, M, V, w, stream=s)
            kv = P.gp_kv(P.GAUSS, Z, [0.7], 0.1, z, stream=s)
            stream.synchronize()
            return [torch.tensor([loss, *dth]), dX.clone(), out.clone(), kv.clone()]
        return call

    # both gradients run the reverse kernel for R_2 up to 48
    calls = [case(12, [1, 9, 44, 60, 80, 60, 44, 9, 1], 1500), case(5, [1, 3, 33, 20, 20, 20, 33, 3, 1], 700)]
    streams = [torch.cuda.Stream() for _ in calls]
    want = []
    for call, stream in zip(calls, streams):
        with torch.cuda.stream(stream):
            want.append(call(stream))
    torch.cuda.synchronize()
    errors = []

    def work(i):
        try:
            with torch.cuda.stream(streams[i]):
                for _ in range(300):
                    got = calls[i](streams[i])
                    assert all(torch.equal(a, b) for a, b in zip(got, want[i]))
        except Exception as e:  # noqa: BLE001
            errors.append(repr(e))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
