"""Performance cases: what a user of the shifted-system solver runs.

Every case goes through the public binding (``paper_1708_06290_gb300.ssv``).
Systems are the random systems of the workloads, A = -2 I + G / sqrt(n) with
G, B, C i.i.d. N(0, 1), made on the GPU from the case's seed; shifts are drawn
log-uniformly on the imaginary axis (frequency sweeps) or as a grid over
[-4, 0] x [-2, 2] moved by a seeded fraction of its pitch (pseudospectra).
A handle that a program keeps between calls (a reduced system) is state;
outputs are returned whole.

Kinds (key "kind"):
  solve     Handle.solve on a kept handle (any precision, modes g / tf / x)
  step      reduction of (A, B, C) and the solve of all shifts, one pass of the
            whole path (the benchmark's step)
  reduce    reduction alone; returns the reduced triple (H, R, Ct)
  norms     Handle.tf_norm2: ||C (sigma I - A)^{-1} B||_2 on a grid
  tangential  Handle.solve_rhs and Handle.solve_trans at the same shifts, the
            two solves of one interpolatory model-reduction iteration
  many      solve_many: one serving micro-batch over several kept handles
  batch     a kept BatchPlan's run over many small systems
"""
import math

import torch

from paper_1708_06290_gb300 import ssv


def listed():
    return [
        # the small frequency sweep (n = 256, m = p = 2, 64 shifts) with the
        # defaults (FP64): the smallest calls, where latency counts
        dict(name="sweep_small_fp64", kind="solve", n=256, m=2, p=2, s=64, shifts="axis",
             precision="fp64", mode="g", arith="fp64"),
        # the FP64 workload: n = 2000, m = p = 8, 1000 frequencies
        dict(name="sweep_fp64", kind="solve", n=2000, m=8, p=8, s=1000, shifts="axis",
             precision="fp64", mode="g", arith="fp64"),
        # the benchmark's step: reduction and 2000 certified grid shifts at
        # n = 5000, m = p = 16; the largest case
        dict(name="step_mixed", kind="step", n=5000, m=16, p=16, s=2000, shifts="grid",
             precision="mixed", mode="g", arith="tensor"),
        # one certified request on a preloaded system of the serving set
        # (n = 4000, m = 16): few shifts, the chip is not filled by them alone
        dict(name="request_mixed", kind="solve", n=4000, m=16, p=16, s=40, shifts="axis",
             precision="mixed", mode="g", arith="tensor"),
        # full solution vectors X, ragged n and a narrow odd m
        dict(name="vectors_mixed", kind="solve", n=1999, m=3, p=5, s=150, shifts="axis",
             precision="mixed", mode="x", arith="tensor"),
        # transfer-function values without certification: the tensor-core sweep
        # alone, medium n and m
        dict(name="transfer_split", kind="solve", n=2500, m=8, p=6, s=600, shifts="axis",
             precision="split", mode="tf", arith="tensor"),
        # structured pseudospectrum on the 50 x 40 grid of a medium system
        dict(name="norms_grid", kind="norms", n=1000, m=4, p=4, s=2000, shifts="grid",
             precision="mixed", arith="tensor"),
        # one model-reduction iteration: tangential and transposed solves
        dict(name="tangential_fp64", kind="tangential", n=1500, m=4, p=3, s=24, shifts="axis",
             arith="tensor"),
        # a serving micro-batch: requests on three preloaded systems at once
        dict(name="microbatch_mixed", kind="many", systems="1000,1,24 2000,4,60 4000,16,16",
             precision="mixed", arith="tensor"),
        # many small systems of uneven size in one replayable plan
        dict(name="batch_dfloat", kind="batch",
             systems="211,1,300 2750,8,24 640,2,90 1333,4,55 900,8,128 2101,2,41 417,4,17 1750,1,210 "
                     "1024,2,64 2944,4,33 305,8,480 1500,1,100",
             precision="dfloat", arith="tensor"),
        # the reduction alone, tensor-core products
        dict(name="reduce_tensor", kind="reduce", n=3000, m=4, p=4, arith="tensor"),
        # the reduction alone, the default arithmetic, at the FP64 workload's size
        dict(name="reduce_fp64", kind="reduce", n=2000, m=8, p=8, arith="fp64"),
    ]


def _between(rng, lo, hi):
    """A whole number spread over [lo, hi] by its logarithm."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "step", "reduce", "norms", "tangential", "many", "batch"])
    arith = "tensor"
    if kind in ("many", "batch"):
        k = rng.randint(2, 4) if kind == "many" else rng.randint(6, 16)
        top = 4000 if kind == "many" else 3000
        systems = ["%d,%d,%d" % (_between(rng, 200, top),
                                 rng.choice([1, 4, 16] if kind == "many" else [1, 2, 4, 8]),
                                 _between(rng, 1 if kind == "many" else 16, 64)) for _ in range(k)]
        return dict(kind=kind, systems=" ".join(systems),
                    precision="mixed" if kind == "many" else rng.choice(["fp64", "dfloat"]), arith=arith)
    n = _between(rng, 200, 4000)
    m = rng.choice([1, 2, 3, 4, 5, 8, 12, 16])
    p = rng.choice([1, 2, m, m, m + 3])
    if kind == "reduce":
        return dict(kind=kind, n=n, m=m, p=p, arith=rng.choice(["fp64", "tensor"]))
    if kind == "tangential":
        return dict(kind=kind, n=min(n, 2000), m=m, p=p, s=_between(rng, 2, 100), shifts="axis", arith=arith)
    # shifts: log-uniform up to 1000, the work bounded by the listed largest
    s = _between(rng, 1, 1000)
    if kind == "norms":
        return dict(kind=kind, n=min(n, 2000), m=m, p=p, s=max(16, s), shifts="grid",
                    precision=rng.choice(["mixed", "split"]), arith=arith)
    if kind == "step":
        return dict(kind=kind, n=n, m=m, p=p, s=s, shifts=rng.choice(["axis", "grid"]), precision="mixed",
                    mode="g", arith=arith)
    prec = rng.choice(["fp64", "mixed", "mixed", "split", "dfloat"])
    mode = rng.choice(["g", "tf", "x"])
    if mode == "x":
        s = min(s, 200)
    # an FP64 sweep of n = 4000, m = 16 takes about 0.7 ms a shift
    if prec == "fp64":
        s = min(s, max(1, int(1.2e10 / (float(n) * n * m))))
    return dict(kind=kind, n=n, m=m, p=p, s=s, shifts="axis", precision=prec, mode=mode, arith=arith)


# ---- inputs -----------------------------------------------------------------

def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _systems(case):
    """(n, m, shifts) of every system of a many / batch case ("n,m,s n,m,s ...")."""
    return [tuple(int(v) for v in q.split(",")) for q in case["systems"].split()]


def _normal(g, rows, cols):
    """Column-major rows x cols, i.i.d. N(0, 1)."""
    return torch.randn((cols, rows), dtype=torch.float64, device="cuda", generator=g).t()


def _system(n, m, p, g):
    A = _normal(g, n, n)
    A.mul_(1.0 / math.sqrt(n)).diagonal().sub_(2.0)
    return A, _normal(g, n, m), _normal(g, p, n)


def _shifts(case, s, g):
    u = torch.rand(s, dtype=torch.float64, device="cuda", generator=g)
    if case.get("shifts", "axis") == "axis":
        w = torch.sort(torch.pow(10.0, 6.0 * u - 3.0)).values
        return torch.complex(torch.zeros_like(w), w)
    # a grid, real index fastest, moved by a fraction of its pitch
    nre = max(1, int(round(math.sqrt(1.25 * s))))
    nim = (s + nre - 1) // nre
    k = torch.arange(s, device="cuda")
    o = torch.rand(2, dtype=torch.float64, device="cuda", generator=g)
    re = -4.0 + 4.0 * ((k % nre) + o[0]) / nre
    im = -2.0 + 4.0 * (torch.div(k, nre, rounding_mode="floor") + o[1]) / nim
    return torch.complex(re, im)


def _complex_normal(g, rows, cols):
    return torch.complex(_normal(g, rows, cols), _normal(g, rows, cols)).t().contiguous().t()


def _inputs(case, seed):
    """Everything that is drawn, in a fixed order."""
    g = _generator(seed)
    if case["kind"] in ("many", "batch"):
        out = []
        for n, m, s in _systems(case):
            A, B, C = _system(n, m, m, g)
            out.append((A, B, C, _shifts(case, s, g)))
        return out
    A, B, C = _system(case["n"], case["m"], case["p"], g)
    d = dict(A=A, B=B, C=C)
    if "s" in case:
        d["sigma"] = _shifts(case, case["s"], g)
    if case["kind"] == "tangential":
        d["b"] = _complex_normal(g, case["m"], case["s"])
        d["c"] = _complex_normal(g, case["p"], case["s"])
    return d


def prepare(case, seed):
    kind = case["kind"]
    x = _inputs(case, seed)
    if kind in ("many", "batch"):
        hs = [ssv.reduce(A, B, C, arith=case["arith"]) for A, B, C, _ in x]
        sg = [q[3] for q in x]
        st = dict(case=case, handles=hs, sigma=sg)
        if kind == "batch":
            st["plan"] = ssv.BatchPlan(hs, sg, mode="g", precision=case["precision"])
        return st
    st = dict(x, case=case)
    if kind not in ("step", "reduce"):
        st["handle"] = ssv.reduce(x["A"], x["B"], x["C"], arith=case["arith"])
        for k in ("A", "B", "C"):
            del st[k]
    return st


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "solve":
        out, status, _ = state["handle"].solve(state["sigma"], mode=case["mode"], precision=case["precision"])
        return {"out": out, "status": status}
    if kind == "step":
        h = ssv.reduce(state["A"], state["B"], state["C"], arith=case["arith"])
        out, status, _ = h.solve(state["sigma"], mode=case["mode"], precision=case["precision"])
        h.close()
        return {"out": out, "status": status}
    if kind == "reduce":
        h = ssv.reduce(state["A"], state["B"], state["C"], arith=case["arith"])
        H, R, Ct = h.reduced()
        h.close()
        return {"H": H, "R": R, "Ct": Ct}
    if kind == "norms":
        norms, status = state["handle"].tf_norm2(state["sigma"], precision=case["precision"])
        return {"norms": norms, "status": status}
    if kind == "tangential":
        x, sx = state["handle"].solve_rhs(state["sigma"], state["b"], mode="x")
        y, sy = state["handle"].solve_trans(state["sigma"], state["c"], mode="x")
        return {"x": x, "y": y, "sx": sx, "sy": sy}
    if kind == "many":
        outs, sts = ssv.solve_many(state["handles"], state["sigma"], mode="g", precision=case["precision"])
        return {"out": outs, "status": sts}
    plan = state["plan"]
    plan.run()
    return {"out": plan.outs, "status": plan.statuses}


# ---- work and exact values ---------------------------------------------------

def _solve_flops(n, m, p, s):
    """Eliminating m subdiagonals of a shifted m-Hessenberg matrix: the fresh
    real columns against m complex ones, 2 n^2 m real operations a shift, and
    the rows of Ct."""
    return s * (2.0 * n * n * m + 4.0 * n * m * p)


def _reduce_flops(n, m, p):
    """The two-sided Householder reduction and the rows of C."""
    return 10.0 / 3.0 * n ** 3 + 4.0 * n * n * (m + p)


def work(case):
    kind = case["kind"]
    if kind in ("many", "batch"):
        b = f = 0.0
        for n, m, s in _systems(case):
            f += _solve_flops(n, m, m, s)
            b += 8.0 * (n * n / 2.0 + 2.0 * n * m) + 16.0 * s * (m * m + 1)
        return {"bytes": b, "flops": f}
    n, m, p, s = case["n"], case["m"], case["p"], case.get("s", 0)
    reduced = 8.0 * (n * (n + 1) / 2.0 + n * m + m * m / 2.0 + p * n)
    full = 8.0 * (n * n + n * m + p * n)
    if kind == "reduce":
        return {"bytes": full + 8.0 * (n * n + n * m + p * n), "flops": _reduce_flops(n, m, p)}
    if kind == "tangential":
        return {"bytes": reduced + 8.0 * n * n + 16.0 * s * (2 * n + m + p + 1),
                "flops": 2.0 * _solve_flops(n, m, 0, s) + 16.0 * s * n * n}
    if kind == "norms":
        return {"bytes": reduced + 24.0 * s, "flops": _solve_flops(n, m, p, s)}
    if kind == "step":
        return {"bytes": full + 16.0 * s * (p * m + 1),
                "flops": _reduce_flops(n, m, p) + _solve_flops(n, m, p, s)}
    rows = n if case["mode"] == "x" else p
    f = _solve_flops(n, m, 0 if case["mode"] == "x" else p, s)
    b = reduced
    if case["mode"] == "x":
        f += 8.0 * s * m * n * n  # X = Q Xhat by the n reflectors
        b += 8.0 * n * n / 2.0
    return {"bytes": b + 16.0 * s * (rows * m + 1), "flops": f}


def _lu_seconds(n):
    """A complex LU of order n with its solves, in FP64 on the GPU."""
    return 2e-3 + 8.0 / 3.0 * float(n) ** 3 / 0.6e12


def _resolvent(A, sigma, B):
    M = A.to(torch.complex128)
    M.diagonal().sub_(sigma)
    return torch.linalg.solve(M, B)


def _transfer(A, B, C, sigma, sign=1.0):
    """C (A - sigma_j I)^{-1} B, p x (s m), one block per shift."""
    Bc, Cc = B.to(torch.complex128), C.to(torch.complex128)
    return torch.cat([sign * (Cc @ _resolvent(A, z, Bc)) for z in sigma], dim=1)


def _exact_reduced(A, B, C):
    """Unblocked Householder reduction to controller-Hessenberg form: B to upper
    triangular, A to upper m-Hessenberg, C along; beta = -sign(alpha) ||x||."""
    A, B, C = A.clone(), B.clone(), C.clone()
    n, m = B.shape

    def reflector(x):
        v = x.clone()
        s = torch.where(v[0] >= 0, 1.0, -1.0).to(v.dtype)
        v[0] += s * torch.linalg.vector_norm(v)
        return v, 2.0 / torch.dot(v, v)

    def both(v, tau, lo, M, col):
        M[lo:, col:] -= tau * torch.outer(v, v @ M[lo:, col:])
        A[:, lo:] -= tau * torch.outer(A[:, lo:] @ v, v)
        C[:, lo:] -= tau * torch.outer(C[:, lo:] @ v, v)

    for j in range(min(m, n - 1)):
        v, tau = reflector(B[j:, j])
        A[j:, :] -= tau * torch.outer(v, v @ A[j:, :])
        both(v, tau, j, B, j)
    for j in range(max(0, n - m - 1)):
        v, tau = reflector(A[j + m:, j])
        both(v, tau, j + m, A, j)
    return torch.triu(A, -m), torch.triu(B), C


def exact(case, seed):
    kind = case["kind"]
    if kind in ("many", "batch"):
        if sum(s * _lu_seconds(n) for n, m, s in _systems(case)) > 15.0:
            return None
        x = _inputs(case, seed)
        return {"out": [_transfer(A, B, C, sg) for A, B, C, sg in x], "status": [None] * len(x)}
    n = case["n"]
    if kind == "reduce":
        if n > 3000:
            return None
        x = _inputs(case, seed)
        H, R, Ct = _exact_reduced(x["A"], x["B"], x["C"])
        return {"H": H, "R": R, "Ct": Ct}
    if case["s"] * _lu_seconds(n) * (2 if kind == "tangential" else 1) > 15.0:
        return None
    x = _inputs(case, seed)
    A, B, C, sg = x["A"], x["B"], x["C"], x["sigma"]
    Bc, Cc = B.to(torch.complex128), C.to(torch.complex128)
    if kind == "tangential":
        xs = [_resolvent(A, sg[j], Bc @ x["b"][:, j:j + 1]) for j in range(case["s"])]
        ys = [_resolvent(A.t(), sg[j], Cc.t() @ x["c"][:, j:j + 1]) for j in range(case["s"])]
        return {"x": torch.cat(xs, dim=1), "y": torch.cat(ys, dim=1), "sx": None, "sy": None}
    if kind == "norms":
        g = [torch.linalg.svdvals(Cc @ _resolvent(A, z, Bc))[0] for z in sg]
        return {"norms": torch.stack(g), "status": None}
    if case["mode"] == "x":
        return {"out": torch.cat([_resolvent(A, z, Bc) for z in sg], dim=1), "status": None}
    return {"out": _transfer(A, B, C, sg, -1.0 if case["mode"] == "tf" else 1.0), "status": None}
