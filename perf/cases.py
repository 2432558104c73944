"""Performance cases: the work that a program using this library has it do, through the public binding.

Every case is a dict of plain values with a "kind":

  online    instantiate + apply for one theta, in one of the precision forms: the loop body of every user of
            the method (new points or a new theta, then products with K~)
  batched   one pttk_batch plan over many instances of their own theta and point sets
  adjoint   the differentiable loss w^T K~ z with its gradients in theta and X (a training step's inner part)
  grid      the offline stage's first half alone: the Chebyshev coefficient tensor of a kernel
  offline   build_offline for a new kernel or new boxes, then one FP64 instantiate + apply with the result
  gp_kv     (K + s2 I) v with the entries evaluated on the fly (the operator of a conjugate-gradient solve)
  gp_lml    log marginal likelihood and its theta-gradient through PTTK-Global (a step of a length-scale fit)

The online, batched and adjoint cases take tensor trains of seeded left-orthonormal cores (what the TT-SVD
hands over) with the ranks that the workloads of workloads.py have at tolerance 1e-10, so that U, M and V
are determined by the inputs: an SVD leaves the cores free up to rotations. The offline cases return what does
not depend on that freedom: the ranks and a product with K~.
"""
import math

import numpy as np
import torch

from paper_2406_06344_gb300 import pttk as P
from paper_2406_06344_gb300 import workloads as W

KERNELS = {name: code for code, name in W.KERNEL_NAMES.items()}
LENGTH_ONLY = ("gaussian", "matern32", "exponential", "matern52", "multiquadric")

# TT ranks at tolerance 1e-10 of the d = 1 Gaussian, d = 2 Matern-3/2 and d = 3 general-nu Matern workloads
R1, R2, R3 = "1,12,12,1", "1,10,63,63,12,1", "1,9,44,177,480,180,49,10,1"


def listed():
    return [
        # the smallest call: 2,000 points a side, where launches and host work are what a user waits for
        {"name": "online_d1_n2k_fp64", "kind": "online", "d": 1, "dtheta": 1, "n": 16, "ranks": R1, "ns": 2000, "nt": 2000, "form": "fp64"},
        # a small ragged d = 3 call: fewer tiles than the GPU has SMs, neither count a multiple of a tile
        {"name": "online_d3_n3k_fp16x3", "kind": "online", "d": 3, "dtheta": 2, "n": 12, "ranks": R3, "ns": 3001, "nt": 1777, "form": "fp16x3"},
        # the d = 2 workload in FP32 and in plain FP64
        {"name": "online_d2_n200k_fp32", "kind": "online", "d": 2, "dtheta": 1, "n": 20, "ranks": R2, "ns": 200000, "nt": 200000, "form": "fp32"},
        {"name": "online_d2_n200k_fp64", "kind": "online", "d": 2, "dtheta": 1, "n": 20, "ranks": R2, "ns": 200000, "nt": 200000, "form": "fp64"},
        # the headline: d = 3, a million points a side, the split tensor-core form
        {"name": "online_d3_n1m_fp16x3", "kind": "online", "d": 3, "dtheta": 2, "n": 12, "ranks": R3, "ns": 1000000, "nt": 1000000, "form": "fp16x3"},
        # 1024 instances of 1k to 100k points a side on one d = 2 tensor train
        {"name": "batched_d2_1024", "kind": "batched", "d": 2, "dtheta": 1, "n": 20, "ranks": R2, "instances": 1024, "lo": 1000, "hi": 100000, "form": "fp16x3"},
        # forward and backward on 500k points a side
        {"name": "adjoint_d3_n500k", "kind": "adjoint", "d": 3, "dtheta": 2, "n": 12, "ranks": R3, "ns": 500000, "nt": 500000, "form": "fp16x3"},
        # the 12^8 grid of the general-nu Matern kernel in FP64
        {"name": "grid_d3_nu_fp64", "kind": "grid", "kernel": "matern_nu", "d": 3, "n": 12, "form": "fp64"},
        # whole offline stages: 20^5 and 12^8
        {"name": "offline_d2_matern32", "kind": "offline", "kernel": "matern32", "d": 2, "n": 20, "tol": 1e-10, "points": 2000},
        {"name": "offline_d3_nu", "kind": "offline", "kernel": "matern_nu", "d": 3, "n": 12, "tol": 1e-10, "points": 2000},
        # one product of a conjugate-gradient solve
        {"name": "gp_kv_d3_n20k_fp64", "kind": "gp_kv", "kernel": "gaussian", "d": 3, "points": 20000, "form": "fp64"},
        # one step of a length-scale fit
        {"name": "gp_lml_d2_n12k", "kind": "gp_lml", "kernel": "gaussian", "d": 2, "n": 16, "tol": 1e-9, "points": 12000},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_tt(rng, d):
    """n and the ranks of a tensor train shaped like those of the workloads."""
    if d == 1:
        n = rng.randint(10, 24)
        return n, "1,%d,%d,1" % (rng.randint(7, n), rng.randint(7, n))
    if d == 2:
        n = rng.randint(12, 24)
        return n, "1,%d,%d,%d,%d,1" % (rng.randint(7, 12), rng.randint(24, 72), rng.randint(24, 72), rng.randint(7, 12))
    n = rng.randint(8, 12)
    return n, "1,%d,%d,%d,%d,%d,%d,%d,1" % (
        rng.randint(6, min(n, 10)), rng.randint(24, 52), rng.randint(72, 184), rng.randint(160, 480), rng.randint(72, 184), rng.randint(24, 52), rng.randint(6, min(n, 10)))


def draw(rng):
    kind = rng.choice(["online", "online", "online", "online", "batched", "adjoint", "grid", "offline", "offline", "gp_kv", "gp_lml"])
    d = rng.choice([1, 2, 2, 3, 3])
    if kind in ("online", "adjoint", "batched"):
        d = max(d, 2) if kind == "batched" else d
        n, ranks = _draw_tt(rng, d)
        c = {"kind": kind, "d": d, "dtheta": 2 if d == 3 else 1, "n": n, "ranks": ranks}
        if kind == "online":
            form = rng.choice(["fp64", "fp32", "fp16x3", "fp16x3", "tf32x3", "fp16"])
            hi = 100000 if form == "fp64" else 1000000
            return {**c, "ns": _log_int(rng, 500, hi), "nt": _log_int(rng, 500, hi), "form": form}
        if kind == "adjoint":
            return {**c, "ns": _log_int(rng, 1000, 500000), "nt": _log_int(rng, 1000, 500000), "form": rng.choice(["fp32", "fp16x3"])}
        return {**c, "instances": _log_int(rng, 16, 1024), "lo": 1000, "hi": _log_int(rng, 2000, 20000), "form": rng.choice(["fp32", "fp16x3", "fp16x3"])}
    if kind == "grid":
        n = {1: rng.randint(12, 32), 2: rng.randint(8, 24), 3: rng.randint(6, 10)}[d]
        return {"kind": kind, "kernel": rng.choice(["matern_nu"] + list(LENGTH_ONLY)), "d": d, "n": n, "form": rng.choice(["fp64", "fp32"])}
    if kind == "offline":
        n = {1: rng.randint(10, 28), 2: rng.randint(10, 22), 3: rng.randint(6, 10)}[d]
        return {"kind": kind, "kernel": rng.choice(["matern_nu"] + list(LENGTH_ONLY)), "d": d, "n": n, "tol": 10.0 ** rng.uniform(-11, -9), "points": _log_int(rng, 500, 3000)}
    if kind == "gp_kv":
        return {"kind": kind, "kernel": rng.choice(LENGTH_ONLY), "d": d, "points": _log_int(rng, 1000, 30000), "form": rng.choice(["fp64", "fp32"])}
    return {"kind": kind, "kernel": "gaussian", "d": rng.choice([1, 2, 2]), "n": rng.randint(14, 18), "tol": 1e-9, "points": _log_int(rng, 1000, 12000)}


# ---------------------------------------------------------------------------------------------------------------

def _boxes(d):
    """The workloads' boxes: the unit cube against the unit cube moved along the first axis (d = 3: by 3)."""
    first = (3.0, 4.0) if d == 3 else (2.0, 3.0)
    return ((0.0, 1.0),) * d, (first,) + ((0.0, 1.0),) * (d - 1)


def _theta_box(dtheta, kernel=None):
    if dtheta == 2:
        return ((0.5, 2.0), (0.5, 2.5))
    return ((0.5, 2.0),)


def _dtheta(c):
    return 2 if c["kernel"] == "matern_nu" else 1


def _ranks(c):
    return [int(r) for r in c["ranks"].split(",")]


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _uniform(g, box, count, dtype):
    lo = torch.tensor([b[0] for b in box], dtype=torch.float64, device="cuda")
    hi = torch.tensor([b[1] for b in box], dtype=torch.float64, device="cuda")
    return (lo + (hi - lo) * torch.rand(count, len(box), generator=g, dtype=torch.float64, device="cuda")).to(dtype)


def _thetas(g, box, count):
    return _uniform(g, box, count, torch.float64)


def _cores(g, c):
    """Left-orthonormal cores on the device, core k of shape r_{k-1} x n x r_k. Small ranks times n below the
    next rank (seldom drawn) leave plain scaled columns."""
    r, n = _ranks(c), c["n"]
    out = []
    for k in range(len(r) - 1):
        Z = torch.randn(r[k] * n, r[k + 1], generator=g, dtype=torch.float64, device="cuda")
        Q = torch.linalg.qr(Z)[0] if r[k] * n >= r[k + 1] else Z / math.sqrt(r[k] * n)
        out.append(Q.reshape(n, r[k], r[k + 1]).transpose(0, 1).contiguous())
    return out


def _tt(c, cores):
    src, tgt = _boxes(c["d"])
    return P.TT.from_cores(W.MATERN_NU if c["dtheta"] == 2 else W.GAUSS, c["d"], src, tgt, c["dtheta"], _theta_box(c["dtheta"]), c["n"],
                           [G.cpu().numpy() for G in cores])


def _dtype(form):
    return torch.float64 if form == "fp64" else torch.float32


def _sizes(c):
    """Instance sizes of a plan (log-uniform): part of the case, the same for every seed, like the other cases' sizes."""
    rng = np.random.default_rng(W.SEED_SIZES)
    lo, hi = math.log(c["lo"]), math.log(c["hi"])
    two = [np.floor(np.exp(rng.uniform(lo, hi, c["instances"]))).astype(np.int64) for _ in range(2)]
    return [np.concatenate([[0], np.cumsum(s)]).astype(np.int64) for s in two]


def _inputs(case, seed):
    """The seeded inputs of a case, shared by prepare and exact."""
    c, g = case, _gen(seed)
    s = {"kind": c["kind"]}
    if c["kind"] in ("online", "adjoint", "batched"):
        d, dt = c["d"], _dtype(c["form"])
        src, tgt = _boxes(d)
        s["cores"] = _cores(g, c)
        if c["kind"] == "batched":
            s["xoff"], s["yoff"] = _sizes(c)
            ns, nt, nth = int(s["xoff"][-1]), int(s["yoff"][-1]), c["instances"]
        else:
            ns, nt, nth = c["ns"], c["nt"], 1
        s["X"], s["Y"] = _uniform(g, src, ns, dt), _uniform(g, tgt, nt, dt)
        s["thetas"] = _thetas(g, _theta_box(c["dtheta"]), nth)
        if c["kind"] != "batched":
            s["w"] = torch.randn(nt, generator=g, dtype=dt, device="cuda")
        if c["kind"] == "adjoint":
            s["ws"] = torch.randn(ns, generator=g, dtype=dt, device="cuda")
        return s
    if c["kind"] in ("grid", "offline"):
        d, dth = c["d"], _dtheta(c)
        src, tgt = _boxes(d)
        # a user's own ranges: the workloads' boxes, moved and stretched a little
        u = torch.rand(2, generator=g, dtype=torch.float64, device="cuda").tolist()
        s["tgt"] = ((tgt[0][0] + 0.25 * u[0], tgt[0][1] + 0.25 * u[0] + 0.1 * u[1]),) + tgt[1:]
        s["src"], s["theta_box"] = src, _theta_box(dth)
        if c["kind"] == "offline":
            s["X"], s["Y"] = _uniform(g, src, c["points"], torch.float64), _uniform(g, s["tgt"], c["points"], torch.float64)
            s["theta"] = _thetas(g, s["theta_box"], 1)[0].tolist()
            s["w"] = torch.randn(c["points"], generator=g, dtype=torch.float64, device="cuda")
        return s
    d = c["d"]
    s["box"] = ((0.0, 1.0),) * d
    s["X"] = _uniform(g, s["box"], c["points"], torch.float64)
    s["v"] = torch.randn(c["points"], generator=g, dtype=torch.float64, device="cuda")
    s["theta"] = [0.5 + 0.5 * torch.rand(1, generator=g, dtype=torch.float64, device="cuda").item()]
    return s


def prepare(case, seed):
    c, s = case, _inputs(case, seed)
    s["case"] = c
    if c["kind"] in ("online", "adjoint", "batched"):
        r, dt = _ranks(c), _dtype(c["form"])
        s["tt"] = _tt(c, s.pop("cores"))
        rs, rt = r[c["d"]], r[c["d"] + c["dtheta"]]
        ns, nt = s["X"].shape[0], s["Y"].shape[0]
        if c["kind"] == "adjoint":
            s["theta"] = s["thetas"][0].cpu().requires_grad_(True)
            s["X"].requires_grad_(True)
            return s
        lead = (c["instances"],) if c["kind"] == "batched" else ()
        s["U"] = torch.empty(ns, rs, dtype=dt, device="cuda")
        s["M"] = torch.empty(*lead, rs, rt, dtype=dt, device="cuda")
        s["V"] = torch.empty(nt, rt, dtype=dt, device="cuda")
        if c["kind"] == "batched":
            s["plan"] = P.Batch(s["tt"], s["xoff"], s["yoff"], c["form"])
        else:
            s["theta"] = s["thetas"][0].tolist()
            s["out"] = torch.empty(ns, dtype=dt, device="cuda")
    elif c["kind"] == "grid":
        s["C"] = torch.empty(c["n"] ** (2 * c["d"] + _dtheta(c)), dtype=_dtype(c["form"]), device="cuda")
    elif c["kind"] == "gp_lml":
        tt = P.TT.build_offline(KERNELS[c["kernel"]], c["d"], s["box"], s["box"], 1, ((0.4, 1.2),), c["n"], c["tol"])
        s["global"] = P.Global(tt, s["X"])
    return s


def run(s):
    c = s["case"]
    kind = c["kind"]
    if kind == "online":
        U, M, V = P.instantiate(s["tt"], s["theta"], s["X"], s["Y"], c["form"], U=s["U"], M=s["M"], V=s["V"])
        return {"U": U, "M": M, "V": V, "Kw": P.apply(U, M, V, s["w"], out=s["out"])}
    if kind == "batched":
        U, M, V = s["plan"].instantiate(s["thetas"], s["X"], s["Y"], U=s["U"], M=s["M"], V=s["V"])
        return {"U": U, "M": M, "V": V}
    if kind == "adjoint":
        loss = P.pttk_loss(s["theta"], s["X"], s["Y"], s["ws"], s["w"], s["tt"], c["form"])
        dtheta, dX = torch.autograd.grad(loss, [s["theta"], s["X"]])
        return {"loss": loss, "dtheta": dtheta, "dX": dX}
    if kind == "grid":
        return P.grid_coeffs(KERNELS[c["kernel"]], c["d"], s["src"], s["tgt"], _dtheta(c), s["theta_box"], c["n"], c["form"], out=s["C"])
    if kind == "offline":
        tt = P.TT.build_offline(KERNELS[c["kernel"]], c["d"], s["src"], s["tgt"], _dtheta(c), s["theta_box"], c["n"], c["tol"])
        U, M, V = P.instantiate(tt, s["theta"], s["X"], s["Y"], "fp64")
        return {"ranks": np.array(tt.ranks), "Kw": P.apply(U, M, V, s["w"])}
    if kind == "gp_kv":
        return P.gp_kv(KERNELS[c["kernel"]], s["X"], s["theta"], 0.1, s["v"], prec=c["form"])
    lml, grad = P.gp_lml(s["global"], s["theta"], 1.0, s["v"])
    return {"lml": lml, "grad": grad}


def _chain_flops(r, n, d, dtheta, ns, nt):
    D = 2 * d + dtheta
    src = sum(r[k] * r[k + 1] for k in range(d))
    tgt = sum(r[k] * r[k + 1] for k in range(d + dtheta, D))
    return 2.0 * n * (src * ns + tgt * nt)


def work(case):
    c = case
    if c["kind"] in ("online", "adjoint", "batched"):
        r, n, d, dth = _ranks(c), c["n"], c["d"], c["dtheta"]
        e = 8 if c["form"] == "fp64" else 4
        if c["kind"] == "batched":
            mean = (c["hi"] - c["lo"]) / math.log(c["hi"] / c["lo"])
            ns = nt = mean * c["instances"]
            nth = c["instances"]
        else:
            ns, nt, nth = c["ns"], c["nt"], 1
        rs, rt = r[d], r[d + dth]
        flops = _chain_flops(r, n, d, dth, ns, nt)
        flops += nth * 2.0 * (n * sum(r[k] * r[k + 1] for k in range(d, d + dth)) + (rs * r[d + 1] * rt if dth == 2 else 0))
        cores = 8.0 * n * sum(a * b for a, b in zip(r, r[1:]))
        if c["kind"] == "adjoint":
            # the reverse pass: both products of every source step once more, but for the last (rank one)
            flops += 4.0 * n * ns * (sum(r[k] * r[k + 1] for k in range(d - 1)) + r[d - 1])
            return {"bytes": e * (ns * (2 * d + 1) + nt * (d + 1)) + cores, "flops": flops}
        nbytes = e * (ns * (d + rs) + nt * (d + rt) + nth * rs * rt) + cores
        if c["kind"] == "online":
            nbytes += e * (nt + ns)
            flops += 2.0 * (ns * rs + nt * rt + rs * rt)
        return {"bytes": nbytes, "flops": flops}
    if c["kind"] in ("grid", "offline"):
        D = 2 * c["d"] + _dtheta(c)
        entries = float(c["n"]) ** D
        flops = entries * (30.0 + 2.0 * c["n"] * D)
        if c["kind"] == "grid":
            return {"bytes": entries * (8 if c["form"] == "fp64" else 4), "flops": flops}
        return {"bytes": 8.0 * c["points"] * (2 * c["d"] + 2), "flops": flops + 20.0 * entries * c["n"]}
    N = float(c["points"])
    if c["kind"] == "gp_kv":
        return {"bytes": 8 * N * (c["d"] + 2), "flops": N * N * (3.0 * c["d"] + 20.0)}
    k = 2.0 * c["n"] ** c["d"] / 4
    return {"bytes": 8 * N * (k + 1), "flops": 2 * N * k + 10 * k ** 3}


# ---------------------------------------------------------------------------------------------------------------
# The same results in 64 bits, by plain torch.

def _cheb(x, lo, hi, n):
    xh = (2.0 * x.double() - lo - hi) / (lo - hi)
    T = [torch.ones_like(xh), xh]
    for _ in range(2, n):
        T.append(2.0 * xh * T[-1] - T[-2])
    return torch.stack(T[:n], dim=-1)


def _chain(cores, pts, box, source):
    """Rows of U (source) or V: the cores contracted with the points' Chebyshev vectors, 20,000 points at a time."""
    d, n = len(box), cores[0].shape[1]
    out = []
    for p in pts.detach().split(20000):
        if source:
            S = torch.ones(p.shape[0], 1, dtype=torch.float64, device=p.device)
            for i in range(d):
                G = cores[i]
                A = (S[:, :, None] * _cheb(p[:, i], *box[i], n)[:, None, :]).reshape(p.shape[0], -1)
                S = A @ G.reshape(-1, G.shape[2])
        else:
            S = torch.ones(p.shape[0], 1, dtype=torch.float64, device=p.device)
            for i in reversed(range(d)):
                G = cores[len(cores) - d + i]
                A = (_cheb(p[:, i], *box[i], n)[:, :, None] * S[:, None, :]).reshape(p.shape[0], -1)
                S = A @ G.reshape(G.shape[0], -1).T
        out.append(S)
    return torch.cat(out)


def _H(cores, d, dtheta, theta, box, n):
    H = None
    for j in range(dtheta):
        Hj = torch.einsum("ajb,j->ab", cores[d + j], _cheb(theta[j], *box[j], n))
        H = Hj if H is None else H @ Hj
    return H


def _kappa(kernel, r, theta):
    l = theta[0]
    if kernel == "gaussian":
        return torch.exp(-(r / l) ** 2)
    if kernel == "matern32":
        a = math.sqrt(3.0) * r / l
        return (1.0 + a) * torch.exp(-a)
    if kernel == "exponential":
        return torch.exp(-r / l)
    if kernel == "matern52":
        a = math.sqrt(5.0) * r / l
        return (1.0 + a + a * a / 3.0) * torch.exp(-a)
    if kernel == "multiquadric":
        return torch.sqrt(1.0 + (r / l) ** 2)
    # general-nu Matern, K_nu(z) = int_0^inf exp(-z cosh t) cosh(nu t) dt by the trapezoidal rule
    nu = theta[1]
    z = torch.sqrt(2.0 * nu) * r / l if torch.is_tensor(nu) else math.sqrt(2.0 * nu) * r / l
    acc = torch.zeros_like(z)
    h = 0.02
    for k in range(0, 451):  # z >= 0.5 here: the integrand is below 1e-17 of its largest well before t = 9
        t = k * h
        w = 0.5 if k == 0 else 1.0
        cn = torch.cosh(nu * t) if torch.is_tensor(nu) else math.cosh(nu * t)
        acc = acc + w * torch.exp(-z * math.cosh(t)) * cn
    lg = torch.lgamma(nu) if torch.is_tensor(nu) else math.lgamma(nu)
    cnu = torch.exp(math.log(2.0) * (1.0 - nu) - lg) if torch.is_tensor(nu) else math.exp(math.log(2.0) * (1.0 - nu) - lg)
    return cnu * z ** nu * acc * h


def _exact_grid(c, s):
    """The kernel at the tensor Chebyshev nodes and its transform along every mode; i_1 varies fastest."""
    d, dth, n = c["d"], _dtheta(c), c["n"]
    D = 2 * d + dth
    i = torch.arange(n, dtype=torch.float64, device="cuda")
    zeta = torch.cos((2 * i + 1) * math.pi / (2 * n))
    boxes = list(s["src"]) + list(s["theta_box"]) + list(s["tgt"])
    nodes = [0.5 * (a - b) * zeta + 0.5 * (a + b) for a, b in boxes]

    def axis(j):
        return nodes[j].reshape([n if k == D - 1 - j else 1 for k in range(D)])  # dimension D-1-j: i_1 is the last

    r2 = sum((axis(j) - axis(d + dth + j)) ** 2 for j in range(d))
    F = _kappa(c["kernel"], torch.sqrt(r2), [axis(d + j) for j in range(dth)]).expand([n] * D)
    A = torch.cos(i[:, None] * math.pi * (2 * i[None, :] + 1) / (2 * n)) * (2.0 / n)
    A[0] *= 0.5
    for k in range(D):
        F = torch.movedim(torch.tensordot(A, F, dims=([1], [k])), 0, k)
    return F.reshape(-1).contiguous()


def exact(case, seed):
    c, s = case, _inputs(case, seed)
    if c["kind"] in ("online", "adjoint", "batched"):
        cores, d, dth, n = s["cores"], c["d"], c["dtheta"], c["n"]
        src, tgt = _boxes(d)
        th = _theta_box(dth)
        if c["kind"] == "adjoint":
            theta = s["thetas"][0].clone().requires_grad_(True)
            b = sum(v.T @ w.double() for v, w in ((_chain(cores, y, tgt, False), w) for y, w in zip(s["Y"].split(20000), s["w"].split(20000))))
            grads, loss = [], 0.0
            dtheta = torch.zeros_like(theta)
            for x, w in zip(s["X"].split(20000), s["ws"].split(20000)):
                x = x.double().requires_grad_(True)
                S = torch.ones(x.shape[0], 1, dtype=torch.float64, device=x.device)
                for i in range(d):
                    G = cores[i]
                    A = (S[:, :, None] * _cheb(x[:, i], *src[i], n)[:, None, :]).reshape(x.shape[0], -1)
                    S = A @ G.reshape(-1, G.shape[2])
                L = w.double() @ (S @ (_H(cores, d, dth, theta, th, n) @ b))
                gt, gx = torch.autograd.grad(L, [theta, x])
                grads.append(gx)
                dtheta += gt
                loss += L.item()
            return {"loss": torch.tensor(loss, dtype=torch.float64), "dtheta": dtheta.cpu(), "dX": torch.cat(grads)}
        U, V = _chain(cores, s["X"], src, True), _chain(cores, s["Y"], tgt, False)
        if c["kind"] == "batched":
            return {"U": U, "M": torch.stack([_H(cores, d, dth, t, th, n) for t in s["thetas"]]), "V": V}
        M = _H(cores, d, dth, s["thetas"][0], th, n)
        return {"U": U, "M": M, "V": V, "Kw": U @ (M @ (V.T @ s["w"].double()))}
    if c["kind"] == "grid":
        if c["n"] ** (2 * c["d"] + _dtheta(c)) > 2.5e7:
            return None  # a 64-bit quadrature of K_nu at every entry takes too long
        return _exact_grid(c, s)
    if c["kind"] == "offline":
        K = _kappa(c["kernel"], torch.cdist(s["X"], s["Y"], compute_mode="donot_use_mm_for_euclid_dist"), s["theta"])
        return {"ranks": None, "Kw": K @ s["w"]}
    if c["kind"] == "gp_kv":
        out = [_kappa(c["kernel"], torch.cdist(x, s["X"], compute_mode="donot_use_mm_for_euclid_dist"), s["theta"]) @ s["v"] for x in s["X"].split(4000)]
        return torch.cat(out) + 0.1 * s["v"]
    # the likelihood of the exact kernel (the low-rank one differs from it by its own accuracy)
    N, l = c["points"], s["theta"][0]
    r2 = torch.cdist(s["X"], s["X"], compute_mode="donot_use_mm_for_euclid_dist") ** 2
    K = torch.exp(-r2 / l ** 2)
    dK = K * (2.0 * r2 / l ** 3)
    K.diagonal().add_(1.0)
    Lc = torch.linalg.cholesky(K)
    alpha = torch.cholesky_solve(s["v"][:, None], Lc)[:, 0]
    lml = -0.5 * (s["v"] @ alpha) - torch.log(Lc.diagonal()).sum() - 0.5 * N * math.log(2.0 * math.pi)
    trace = (torch.cholesky_inverse(Lc) * dK).sum()
    grad = 0.5 * (alpha @ (dK @ alpha)) - 0.5 * trace
    return {"lml": float(lml), "grad": grad.reshape(1).cpu().numpy()}
