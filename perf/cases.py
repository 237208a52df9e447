"""The work that programs have this library do, as cases to measure.

A case is a dict of plain values.  `prepare` makes what a program holds before
the call (inputs on the device or the host, and the handle, batch or server it
keeps), `run` is one call through the public entry points with the whole result
read back, as a program reads it.  Every LP is a dense one of the kind the
solver is for:  maximize c^T x,  A x <= b,  x >= 0,  A ~ U[1, 10),
b ~ U[100, 1000), c ~ U[1, 10)  (kind "diag": A ~ U[0, 1) with a strong
diagonal, whose final basis holds every structural variable).
"""
import math
import random

import numpy as np
import torch

import paper_2211_10979_gb300 as tsx

DEV = "cuda"


# ------------------------------------------------------------------ cases
def listed():
    return [
        # one small LP, solved over and over by a program that waits for each:
        # latency is everything
        {"name": "single_256", "kind": "single", "m": 256, "n": 256, "precision": "fp64"},
        # a one-off solve from NumPy arrays: upload, check, solve, read-out, release
        {"name": "oneshot_700x500", "kind": "oneshot", "m": 700, "n": 500, "precision": "fp64"},
        # medium LPs, too large for one cluster's shared memory, too small to be
        # bound by memory; the second with odd sizes and more rows than columns
        {"name": "single_1024", "kind": "single", "m": 1024, "n": 1024, "precision": "fp64"},
        {"name": "single_2049x1531", "kind": "single", "m": 2049, "n": 1531, "precision": "fp64"},
        # the large dense LP the library is benchmarked on, and its aspect-ratio case
        {"name": "single_8192", "kind": "single", "m": 8192, "n": 8192, "precision": "fp64"},
        {"name": "single_4096x16384", "kind": "single", "m": 4096, "n": 16384, "precision": "fp64"},
        # float tableau with FP64 recovery: a medium odd LP, a large one, and one
        # whose recovery refactorises a basis of 2048 structural variables
        {"name": "fp32_1500x2001", "kind": "single", "m": 1500, "n": 2001, "precision": "fp32"},
        {"name": "fp32_12288", "kind": "single", "m": 12288, "n": 12288, "precision": "fp32"},
        {"name": "fp32_diag_2048", "kind": "diag", "m": 2048, "n": 2048, "precision": "fp32"},
        # thousands of small LPs at once, m and n in [16, 128]
        {"name": "batch_4096", "kind": "batch", "count": 4096, "lo": 16, "hi": 128, "precision": "fp64"},
        # many medium LPs of mixed sizes in one call
        {"name": "many_96", "kind": "many", "count": 96, "lo": 180, "hi": 3000, "precision": "fp64"},
        # a server that gets a burst of requests of every size it serves
        {"name": "serve_200", "kind": "serve", "count": 200, "lo": 32, "hi": 4096, "precision": "fp32"},
    ]


def _log_int(rng, lo, hi):
    return int(math.floor(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.999)))))


def draw(rng):
    kind = rng.choice(["single", "single", "single", "single", "oneshot", "diag", "batch", "many", "serve"])
    if kind == "single":
        precision = rng.choice(["fp64", "fp64", "fp32"])
        top = 12288 if precision == "fp32" else 8192
        m = _log_int(rng, 33, top)
        n = min(_log_int(rng, 33, 16384), max(33, top * top // m))   # no tableau above the largest listed
        return {"kind": kind, "m": m, "n": n, "precision": precision}
    if kind == "oneshot":
        return {"kind": kind, "m": _log_int(rng, 33, 1999), "n": _log_int(rng, 33, 1999),
                "precision": rng.choice(["fp64", "fp32"])}
    if kind == "diag":
        m = _log_int(rng, 100, 2047)
        return {"kind": kind, "m": m, "n": m, "precision": rng.choice(["fp64", "fp32"])}
    if kind == "batch":
        return {"kind": kind, "count": _log_int(rng, 65, 4095), "lo": 16, "hi": _log_int(rng, 33, 128),
                "precision": "fp64"}
    if kind == "many":
        return {"kind": kind, "count": _log_int(rng, 5, 95), "lo": 180, "hi": _log_int(rng, 500, 3000),
                "precision": rng.choice(["fp64", "fp32"])}
    return {"kind": kind, "count": _log_int(rng, 21, 199), "lo": 32, "hi": _log_int(rng, 500, 4096),
            "precision": "fp32"}


# ----------------------------------------------------------------- inputs
def _shapes(case, seed):
    """(m, n) of the LPs of a case.  Lists: m and n uniform in [lo, hi] for a
    batch, log-uniform otherwise; the sizes belong to the case and only the
    data to the seed, so that every seed is the same amount of work."""
    if "count" not in case:
        return [(case["m"], case["n"])]
    rng = random.Random(f"{case['kind']} {case['count']} {case['lo']} {case['hi']}")
    lo, hi = case["lo"], case["hi"]
    one = (lambda: rng.randint(lo, hi)) if case["kind"] == "batch" else (lambda: _log_int(rng, lo, hi))
    return [(one(), one()) for _ in range(case["count"])]


def _inputs(case, seed):
    """A, b, c of every LP, FP64 on the device, from the seed alone."""
    g = torch.Generator(device=DEV)
    g.manual_seed(1_000_003 * int(seed) + 17)
    out = []
    for m, n in _shapes(case, seed):
        A = torch.rand(m, n, dtype=torch.float64, device=DEV, generator=g)
        if case["kind"] == "diag":
            A.diagonal().add_(4.0 * max(m, n))
        else:
            A.mul_(9.0).add_(1.0)
        b = torch.rand(m, dtype=torch.float64, device=DEV, generator=g).mul_(900.0).add_(100.0)
        c = torch.rand(n, dtype=torch.float64, device=DEV, generator=g).mul_(9.0).add_(1.0)
        out.append((A, b, c))
    torch.cuda.synchronize()
    return out


def prepare(case, seed):
    lps = _inputs(case, seed)
    prec = tsx.LP_PREC_FP32 if case["precision"] == "fp32" else tsx.LP_PREC_FP64
    kind = case["kind"]
    if kind in ("single", "diag"):
        return {"kind": "single", "opts": tsx.options(precision=prec), "problem": tsx.Problem(*lps[0], device=True)}
    if kind == "oneshot":
        return {"kind": kind, "precision": prec, "host": tuple(t.cpu().numpy() for t in lps[0])}
    if kind == "batch":
        m = np.array([A.shape[0] for A, _, _ in lps], dtype=np.int32)
        n = np.array([A.shape[1] for A, _, _ in lps], dtype=np.int32)
        A, b, c = (torch.cat([lp[k].reshape(-1) for lp in lps]) for k in range(3))
        torch.cuda.synchronize()
        return {"kind": kind, "batch": tsx.Batch(m=m, n=n, A=A, b=b, c=c, device=True)}
    if kind == "many":
        return {"kind": kind, "opts": tsx.options(precision=prec),
                "problems": [tsx.Problem(*lp, device=True) for lp in lps]}
    return {"kind": kind, "lps": lps, "server": tsx.Server(precision=prec)}


# -------------------------------------------------------------------- run
def _packed(status, iters, x, y, obj, basis=None):
    out = {"status": np.asarray(status, dtype=np.int64), "iters": np.asarray(iters, dtype=np.int64),
           "x": np.concatenate(x), "y": np.concatenate(y), "obj": np.asarray(obj, dtype=np.float64)}
    if basis is not None:
        out["basis"] = np.concatenate(basis)
    return out


def _solutions(sols):
    return _packed([s.status for s in sols], [s.iters for s in sols], [s.x for s in sols], [s.y for s in sols],
                   [s.obj for s in sols], [s.basis for s in sols])


def run(state):
    kind = state["kind"]
    if kind == "single":
        state["problem"].solve(state["opts"])
        return _solutions([state["problem"].solution()])
    if kind == "oneshot":
        return _solutions([tsx.solve(*state["host"], precision=state["precision"])])
    if kind == "batch":
        state["batch"].solve()
        r = state["batch"].results()
        return _packed(r.status, r.iters, r.x, r.y, r.obj)
    if kind == "many":
        tsx.solve_many(state["problems"], state["opts"])
        return _solutions([p.solution() for p in state["problems"]])
    sv = state["server"]
    tickets = [sv.submit_device(A.shape[0], A.shape[1], A, b, c) for A, b, c in state["lps"]]
    for t in tickets:
        sv.wait(t)
    rs = [sv.result(t) for t in tickets]
    return _packed([r.status for r in rs], [r.iters for r in rs], [r.x for r in rs], [r.y for r in rs],
                   [r.obj for r in rs])


# ------------------------------------------------------------------- work
def _pivots(case, m, n):
    """Pivots of an LP of this kind, fitted to measured runs (256^2: 38,
    8192^2: 2.8k, 16384^2: 6.5k; a diagonal LP takes about one per variable)."""
    if case["kind"] == "diag":
        return float(n)
    return max(1.0, 38.0 * (math.sqrt(m * n) / 256.0) ** 1.24)


def work(case):
    """The inputs read and the results written once, and the multiply-adds of
    the pivots: one per entry of the condensed tableau and pivot."""
    nbytes = flops = 0.0
    for m, n in _shapes(case, 0):
        nbytes += 8.0 * (m * n + 2 * m + 2 * n) + 4.0 * m
        flops += 2.0 * (m + 1) * (n + 1) * _pivots(case, m, n)
        if case["kind"] == "diag" and case["precision"] == "fp32":
            flops += 2.0 * float(n) ** 3   # the recovery's inverse of the final basis
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """x, y and the objective against the same LP solved in 64 bits from its
    final basis: the tableau's rounding, which grows along the pivots.  Seen
    over these cases: 1e-15 at 256^2 to 2e-13 at 8192^2 (FP64), 6e-14 with
    the recovery.  The pivots, the basis and the statuses are whole numbers and
    stay the same."""
    return {"rel": 1e-12, "differ": 0.0}


# ------------------------------------------------------------------ exact
def _simplex(A, b, c):
    """Final basis of the condensed-tableau simplex in plain torch, FP64: the
    nonbasic variable of each column and the basic one of each row."""
    m, n = A.shape
    T = torch.zeros(m + 1, n + 1, dtype=torch.float64, device=A.device)
    T[0, :n] = -c
    T[1:, :n] = A
    T[1:, n] = b
    col = list(range(n))
    row = list(range(n, n + m))
    inf = torch.tensor(float("inf"), dtype=torch.float64, device=A.device)
    for _ in range(50 * (m + n)):
        q = torch.argmin(T[0, :n])
        f = T.index_select(1, q.view(1)).view(-1)
        ratio = torch.where(f[1:] > 1e-9, T[1:, n] / f[1:], inf)
        p = torch.argmin(ratio) + 1
        qi, pi, low = (int(v) for v in torch.stack([q, p, (T[0, :n].index_select(0, q.view(1)).view(()) < -1e-9).long()]))
        if not low:
            return col, row
        piv = T[pi, qi].clone()
        f[pi] = 0.0
        T[:, qi] = 0.0
        T[pi, qi] = 1.0
        r = T[pi] / piv
        T.addr_(f, r, alpha=-1.0)
        T[pi] = r
        col[qi], row[pi - 1] = row[pi - 1], col[qi]
    raise RuntimeError("the reference did not finish")


def _solve_basis(A, b, c, col, row):
    """x, y, objective of a basis from the inputs: x_S of A_RS x_S = b_R and
    y_R of A_RS^T y_R = c_S, S the basic structurals, R the rows whose slack is
    nonbasic."""
    m, n = A.shape
    S = torch.tensor(sorted(v for v in row if v < n), dtype=torch.long, device=A.device)
    R = torch.tensor(sorted(v - n for v in col if v >= n), dtype=torch.long, device=A.device)
    x = torch.zeros(n, dtype=torch.float64, device=A.device)
    y = torch.zeros(m, dtype=torch.float64, device=A.device)
    if len(S):
        M = A[R][:, S]
        x[S] = torch.linalg.solve(M, b[R])
        y[R] = torch.linalg.solve(M.T, c[S])
    return x.cpu().numpy(), y.cpu().numpy(), float(c @ x)


def exact(case, seed):
    shapes = _shapes(case, seed)
    # about 0.2 ms of launches and a few passes over the tableau a pivot
    cost = sum(_pivots(case, m, n) * (3e-4 + 4 * 8.0 * m * n / 4e12) for m, n in shapes)
    if cost > 16.0:
        return None
    x, y, obj = [], [], []
    for A, b, c in _inputs(case, seed):
        got = _solve_basis(A, b, c, *_simplex(A, b, c))
        x.append(got[0])
        y.append(got[1])
        obj.append(got[2])
    out = {"status": None, "iters": None, "x": np.concatenate(x), "y": np.concatenate(y),
           "obj": np.asarray(obj, dtype=np.float64)}
    if case["kind"] in ("single", "diag", "oneshot", "many"):
        out["basis"] = None
    return out
