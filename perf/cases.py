"""The work this library is timed on: whole solves, gradients, batches and transforms.

Every case goes through the public entry points of ``paper_2312_09376_gb300``
the way a program calls them: the system, the right-hand sides, the workspace
and the plan are in hand, one pass is one call (or one call and its backward).

Sizes are those of the repository's own configurations, tests and benchmark
(n = 67, 1003, 4001, 8197, 20001, 40003; 2048 systems of order 48 .. 700; 256
systems of order 32 .. 256); ``draw`` spreads over the same ranges.  Matrices
are N(0, 1), or D_r G D_c with diagonal entries 10^U(-s, s) (``spread`` s).  Solves
refine to a backward error of 1e-15, near the end of double arithmetic, so that
two correct solvers' results for one input agree to nine digits and more.
"""
import math

import torch

from paper_2312_09376_gb300 import _lib, autograd

TOL = 1e-15


def listed():
    return [
        # a layer-sized dense system inside a training step: host and launch latency
        {"name": "grad f64 n=67", "do": "grad", "prec": "f64", "n": 67, "nrhs": 3, "depth": 2, "spread": 0.0},
        # the plain method on one small system, in the default precision
        {"name": "solve f64 n=1003", "do": "solve", "prec": "f64", "n": 1003, "nrhs": 1, "depth": 2,
         "spread": 0.0, "kind": "scaled"},
        # the same system in the mixed precision
        {"name": "solve df64tc7 n=1003", "do": "solve", "prec": "df64tc7", "n": 1003, "nrhs": 1, "depth": 2,
         "spread": 0.0, "kind": "scaled"},
        # an ordinary double solve
        {"name": "solve f64 n=4001", "do": "solve", "prec": "f64", "n": 4001, "nrhs": 1, "depth": 2,
         "spread": 0.0, "kind": "scaled"},
        # differentiation: X = solve(A, B) and both gradients, default precision
        {"name": "grad f64 n=8197", "do": "grad", "prec": "f64", "n": 8197, "nrhs": 32, "depth": 2, "spread": 0.0},
        # the same in mixed precision
        {"name": "grad df64tc7 n=8197", "do": "grad", "prec": "df64tc7", "n": 8197, "nrhs": 32, "depth": 2,
         "spread": 0.0},
        # a large system at depth 3, an odd order
        {"name": "solve df64tc n=20001 d=3", "do": "solve", "prec": "df64tc", "n": 20001, "nrhs": 1, "depth": 3,
         "spread": 0.0, "kind": "scaled"},
        # the benchmark's system: scaled rows and columns, mixed precision
        {"name": "solve df64tc7 n=40003", "do": "solve", "prec": "df64tc7", "n": 40003, "nrhs": 1, "depth": 2,
         "spread": 0.5, "kind": "scaled"},
        # thousands of uneven systems in one planned launch, both precisions
        {"name": "batch f64 2048", "do": "batch", "prec": "f64", "count": 2048, "lo": 48, "hi": 700, "rhs": 8,
         "depth": 2},
        {"name": "batch f32 2048", "do": "batch", "prec": "f32", "count": 2048, "lo": 48, "hi": 700, "rhs": 8,
         "depth": 2},
        # a batched layer and its backward, planned anew in each step
        {"name": "batch grad f32 256", "do": "batch_grad", "prec": "f32", "count": 256, "lo": 32, "hi": 256, "rhs": 4,
         "depth": 2},
        # the two-sided transform alone, double out
        {"name": "transform f64 n=16385", "do": "transform", "prec": "f64", "n": 16385, "depth": 2},
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    do = rng.choice(["solve", "solve", "solve", "grad", "grad", "batch", "batch_grad", "transform"])
    if do == "solve":
        prec = rng.choice(["f64", "df64tc7", "df64tc"])
        return {"do": do, "prec": prec, "n": _log_int(rng, 64, 8200 if prec == "f64" else 24000),
                "nrhs": rng.choice([1, 1, 1, 2, 5, 16]), "depth": rng.choice([1, 2, 2, 3]),
                "spread": rng.choice([0.0, 0.0, round(rng.uniform(0.1, 0.5), 2)]),
                "kind": rng.choice(["scaled", "scaled", "scaled", "rotation"])}
    if do == "grad":
        return {"do": do, "prec": rng.choice(["f64", "df64tc7"]), "n": _log_int(rng, 33, 8000),
                "nrhs": _log_int(rng, 1, 32), "depth": rng.choice([1, 2]), "spread": 0.0}
    if do == "batch":
        lo = rng.randint(16, 100)
        return {"do": do, "prec": rng.choice(["f64", "f32"]), "count": _log_int(rng, 64, 2048), "lo": lo,
                "hi": rng.randint(lo + 50, 700), "rhs": rng.randint(1, 8), "depth": rng.choice([1, 2])}
    if do == "batch_grad":
        lo = rng.randint(16, 60)
        return {"do": do, "prec": rng.choice(["f64", "f32"]), "count": _log_int(rng, 32, 256), "lo": lo,
                "hi": rng.randint(lo + 40, 256), "rhs": rng.randint(1, 6), "depth": rng.choice([1, 2])}
    return {"do": do, "prec": rng.choice(["f64", "f64", "f32"]), "n": _log_int(rng, 500, 20001),
            "depth": rng.choice([1, 2, 2, 3])}


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _randn(g, rows, cols):
    """A column-major rows x cols matrix of N(0, 1) entries."""
    return torch.randn((cols, rows), generator=g, device="cuda", dtype=torch.float64).T


def _system(case, seed):
    g = _generator(seed)
    n = case["n"]
    A, B = _randn(g, n, n), _randn(g, n, case["nrhs"])
    if case["spread"]:
        for shape in ((n, 1), (1, n)):
            u = torch.rand(shape, generator=g, device="cuda", dtype=torch.float64)
            A.mul_(torch.pow(10.0, case["spread"] * (2 * u - 1)))
    return A, B, g


def _orders(case):
    """Orders and right-hand-side counts of a batch: the case's own, the same for every seed."""
    r = torch.Generator().manual_seed(7)
    n = torch.randint(case["lo"], case["hi"] + 1, (case["count"],), generator=r).tolist()
    return n, torch.randint(1, case["rhs"] + 1, (case["count"],), generator=r).tolist()


def _batch(case, seed):
    n, k = _orders(case)
    g = _generator(seed)
    a = torch.randn(sum(m * m for m in n), generator=g, device="cuda", dtype=torch.float64)
    b = torch.randn(sum(m * c for m, c in zip(n, k)), generator=g, device="cuda", dtype=torch.float64)
    return n, k, a, b, g


def _views(flat, rows, cols):
    parts = torch.split(flat, [r * c for r, c in zip(rows, cols)])
    return [p.view(c, r).T for p, r, c in zip(parts, rows, cols)]


def prepare(case, seed):
    _lib.load()
    s = dict(case)
    if case["do"] == "solve":
        s["A"], s["B"], _ = _system(case, seed)
        n, nrhs = case["n"], case["nrhs"]
        s["opts"] = _lib.make_opts(case["depth"], 1, case["prec"], 30, TOL, True, kind=case["kind"])
        s["X"] = _lib.colmajor(n, nrhs)
        s["work"] = torch.empty(_lib.rbt_solve_workspace(s["opts"], n, nrhs), dtype=torch.uint8, device="cuda")
    elif case["do"] == "grad":
        A, B, g = _system(case, seed)
        s["A"], s["B"] = A.requires_grad_(), B.requires_grad_()
        s["W"] = _randn(g, case["n"], case["nrhs"])
    elif case["do"] == "batch":
        n, k, a, b, _ = _batch(case, seed)
        s["x"] = torch.zeros_like(b)
        opts = _lib.make_opts(case["depth"], 1000, case["prec"], 30, TOL, True)
        s["plan"] = _lib.rbt_solve_batched_plan(opts, _views(a, n, n), _views(b, n, k), _views(s["x"], n, k))
    elif case["do"] == "batch_grad":
        n, k, a, b, g = _batch(case, seed)
        w = torch.randn(b.shape, generator=g, device="cuda", dtype=torch.float64)
        s["A"], s["B"], s["W"] = _views(a, n, n), _views(b, n, k), _views(w, n, k)
    else:
        n, g = case["n"], _generator(seed)
        s["A"] = _randn(g, n, n)
        s["U"], s["V"] = _lib.colmajor(n, case["depth"]), _lib.colmajor(n, case["depth"])
        _lib.rbt_generate(n, case["depth"], 1, s["U"], s["V"])
        s["out"] = _lib.colmajor(n, n, dtype=_lib.PREC_DTYPE[_lib.PREC[case["prec"]]])
    return s


def _flat(tensors):
    return torch.cat([t.T.reshape(-1) for t in tensors])


def run(s):
    if s["do"] == "solve":
        status, _ = _lib.rbt_solve(s["opts"], s["n"], s["A"], s["B"], s["X"], s["work"])
        return {"X": s["X"], "status": status}
    if s["do"] == "grad":
        X = autograd.solve(s["A"], s["B"], depth=s["depth"], prec=s["prec"], tol=TOL)
        gA, gB = torch.autograd.grad(X, (s["A"], s["B"]), s["W"])
        return {"X": X.detach(), "grad_A": gA, "grad_B": gB}
    if s["do"] == "batch":
        _lib.rbt_solve_batched_run(s["plan"])
        return {"X": s["x"]}
    if s["do"] == "batch_grad":
        Xs, plan = autograd.solve_batched(s["A"], s["B"], depth=s["depth"], prec=s["prec"], tol=TOL)
        gB, gA = autograd.solve_batched_backward(plan, s["W"])
        return {"X": _flat(Xs), "grad_A": _flat(gA), "grad_B": _flat(gB)}
    if s["prec"] == "f64":
        _lib.rbt_apply_2sided(s["n"], s["depth"], s["U"], s["V"], s["A"], s["out"])
    else:
        _lib.rbt_apply_2sided_wp(s["n"], s["depth"], s["U"], s["V"], s["A"], s["out"], s["prec"])
    return {"out": s["out"]}


def work(case):
    if case["do"] in ("solve", "grad"):
        n, r = case["n"], case["nrhs"]
        bytes_ = 8 * n * n + 16 * n * r
        flops = 2 * n ** 3 / 3 + 2 * n * n * r
        if case["do"] == "grad":
            bytes_ += 8 * n * n + 16 * n * r
            flops += 4 * n * n * r
        return {"bytes": bytes_, "flops": flops}
    if case["do"] in ("batch", "batch_grad"):
        sizes = list(zip(*_orders(case)))
        bytes_ = sum(8 * n * n + 16 * n * r for n, r in sizes)
        flops = sum(2 * n ** 3 / 3 + 2 * n * n * r for n, r in sizes)
        if case["do"] == "batch_grad":
            bytes_ *= 2
            flops += sum(4 * n * n * r for n, r in sizes)
        return {"bytes": bytes_, "flops": flops}
    n, d = case["n"], case["depth"]
    return {"bytes": n * n * (16 if case["prec"] == "f64" else 12), "flops": 4 * d * n * n}


def _layer(X, w, h, n):
    """(B_k R_k)^T X along dimension 0: butterflies of half size h on each 2 h rows, then the diagonal w."""
    Y = torch.empty_like(X)
    for r0 in range(0, n, 2 * h):
        top, mid, end = r0, min(n, r0 + h), min(n, r0 + 2 * h)
        m = end - mid
        a, b = X[top:top + m], X[mid:end]
        Y[top:top + m] = (a + b) * math.sqrt(0.5)
        Y[mid:end] = (a - b) * math.sqrt(0.5)
        Y[top + m:mid] = X[top + m:mid]
    return Y * w[:, None]


def _two_sided(A, U, V):
    n, d = U.shape
    ds = min(d, math.ceil(math.log2(n)))
    m = 2 ** ds * -(-n // 2 ** ds)
    for W in (U, V):
        for k in range(d, 0, -1):
            A = _layer(A, W[:, k - 1], m >> k, n) if k <= ds else A * W[:, k - 1, None]
        A = A.T
    return A


def exact(case, seed):
    if case["do"] in ("solve", "grad"):
        if case["n"] > 24000:
            return None  # about 40 seconds in 64 bits
        A, B, g = _system(case, seed)
        LU, piv = torch.linalg.lu_factor(A)

        def solved(R, adjoint):
            """The solution and one step of refinement."""
            M = A.T if adjoint else A
            X = torch.linalg.lu_solve(LU, piv, R, adjoint=adjoint)
            return X + torch.linalg.lu_solve(LU, piv, R - M @ X, adjoint=adjoint)

        X = solved(B, False)
        if case["do"] == "solve":
            return {"X": X, "status": None}
        Y = solved(_randn(g, case["n"], case["nrhs"]), True)
        return {"X": X, "grad_A": -Y @ X.T, "grad_B": Y}
    if case["do"] in ("batch", "batch_grad"):
        n, k, a, b, g = _batch(case, seed)
        As, Xs = _views(a, n, n), []
        for A, B in zip(As, _views(b, n, k)):
            Xs.append(torch.linalg.solve(A, B))
        if case["do"] == "batch":
            return {"X": _flat(Xs)}
        w = torch.randn(b.shape, generator=g, device="cuda", dtype=torch.float64)
        Ys = [torch.linalg.solve(A.T, W) for A, W in zip(As, _views(w, n, k))]
        return {"X": _flat(Xs), "grad_A": _flat([-Y @ X.T for X, Y in zip(Xs, Ys)]), "grad_B": _flat(Ys)}
    n, d = case["n"], case["depth"]
    U, V = (_coefficients(n, d, side) for side in (0, 1))
    return {"out": _two_sided(_randn(_generator(seed), n, n), U, V)}


def _coefficients(n, d, side, seed=1):
    """exp(r / 20), r uniform on [-1, 1) from SplitMix64 of (seed, side, layer, row)."""
    import numpy as np

    W = np.empty((n, d))
    with np.errstate(over="ignore"):
        for k in range(1, d + 1):
            z = np.uint64(seed ^ (side << 62) ^ (k << 48)) ^ np.arange(n, dtype=np.uint64)
            z = z + np.uint64(0x9E3779B97F4A7C15)
            z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
            z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
            z = z ^ (z >> np.uint64(31))
            W[:, k - 1] = np.exp((2 * ((z >> np.uint64(11)).astype(np.float64) * 2.0 ** -53) - 1) / 20)
    return torch.from_numpy(W).cuda()
