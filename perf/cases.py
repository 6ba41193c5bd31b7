"""The work that users of this library have it do, as timed cases.

A case names a graph (family, size, weights), an entry point and its options.
The entry points are the ones a program calls: a whole solve (setup plus
cascade), a re-solve on a resident hierarchy, k eigenpairs, a batch of small
graphs, warm requests to the server, and the step entry points on device
buffers.  Sizes and families follow the configurations of bench.py and of the
tests: 2D and 3D grids, random geometric, Barabasi-Albert and Chung-Lu graphs.

    listed()             the cases
    draw(rng)            one more case of the same ranges
    prepare(case, seed)  what a program holds before the call
    run(state)           one call and its outputs
    work(case)           bytes and operations the call cannot do without
    exact(case, seed)    what run() returns, from plain 64-bit torch and numpy
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1412_0565_gb300 import cmg, inputs

DEV = "cuda"


# ------------------------------------------------------------------ cases
def listed():
    return [
        # one small graph from host memory, setup and solve: latency and launches
        {"name": "solve_grid2d_4k", "kind": "solve", "family": "grid2d", "n": 4096, "weights": "uniform",
         "precision": "fp64", "mem": "host"},
        # the median graph of a request stream (sizes 1e3 .. 2e6), host memory
        {"name": "solve_rgg_45k", "kind": "solve", "family": "rgg", "n": 44721, "weights": "uniform",
         "precision": "fp64", "mem": "host"},
        # the headline: 1M vertices on the device, FP64 and FP32 sweeps
        {"name": "solve_grid3d_1m", "kind": "solve", "family": "grid3d", "n": 1000000, "weights": "uniform",
         "precision": "fp64", "mem": "device"},
        {"name": "solve_grid3d_1m_fp32", "kind": "solve", "family": "grid3d", "n": 1000000, "weights": "uniform",
         "precision": "fp32", "mem": "device"},
        # power-law graph: hub rows, dense coarse levels, FP32 sweeps
        {"name": "solve_chunglu_250k_fp32", "kind": "solve", "family": "chung_lu", "n": 250000,
         "weights": "lognormal", "precision": "fp32", "mem": "device"},
        # recursive bisection, parameter studies: another solve on a kept hierarchy
        {"name": "resolve_ba_20k", "kind": "resolve", "family": "ba", "n": 20000, "weights": "uniform",
         "precision": "fp64", "start": "seed"},
        # spectral embedding: several eigenpairs on a kept hierarchy
        {"name": "eigenpairs4_rgg_8k", "kind": "eigenpairs", "family": "rgg", "n": 8000, "weights": "uniform", "k": 4},
        # many small graphs at once, FP32 sweeps (the batched form's use)
        {"name": "batch_128_fp32", "kind": "batch", "graphs": 128, "lo": 500, "hi": 8192, "precision": "fp32"},
        # requests for resident graphs of mixed sizes, four workers
        {"name": "serve_warm_8", "kind": "serve", "graphs": 8, "lo": 1000, "hi": 100000, "precision": "fp32"},
        # coarsening alone, on device buffers
        {"name": "hec_grid3d_262k", "kind": "hec", "family": "grid3d", "n": 262144, "weights": "uniform"},
        # smoothing alone: a latency-critical loop that must not allocate ...
        {"name": "sweeps_noalloc_rgg_10k", "kind": "sweeps", "family": "rgg", "n": 10000, "weights": "uniform",
         "k": 16, "noalloc": True},
        # ... and a graph larger than L2
        {"name": "sweeps_grid3d_2m", "kind": "sweeps", "family": "grid3d", "n": 2097152, "weights": "uniform",
         "k": 20, "noalloc": False},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


# largest graph per family in a drawn case (the listed ones bound the cost)
_MOST = {"grid2d": 1000000, "grid3d": 1000000, "rgg": 300000, "ba": 100000, "chung_lu": 250000}


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "solve", "resolve", "resolve", "eigenpairs", "batch", "serve", "hec",
                       "sweeps", "sweeps"])
    family = rng.choice(sorted(_MOST))
    weights = "lognormal" if family == "chung_lu" else "uniform"
    if kind == "batch":
        lo = _log(rng, 100, 2000)
        return {"kind": kind, "graphs": rng.randint(33, 128), "lo": lo, "hi": _log(rng, 2 * lo, 8192),
                "precision": rng.choice(["fp64", "fp32"])}
    if kind == "serve":
        return {"kind": kind, "graphs": rng.randint(2, 8), "lo": 1000, "hi": _log(rng, 4000, 100000),
                "precision": rng.choice(["fp64", "fp32"])}
    c = {"kind": kind, "family": family, "n": _log(rng, 200, _MOST[family]), "weights": weights}
    if kind == "solve":
        c.update(precision=rng.choice(["fp64", "fp64", "fp32"]), mem=rng.choice(["host", "device"]))
    elif kind == "resolve":
        c.update(precision=rng.choice(["fp64", "fp32"]), start=rng.choice(["seed", "seed", "vector"]))
    elif kind == "eigenpairs":
        # vertex sets with a geometry to embed, as in the listed case
        c.update(family=rng.choice(["grid2d", "grid3d", "rgg"]), n=_log(rng, 200, 8000), weights="uniform",
                 k=rng.randint(2, 6))
    elif kind == "sweeps":
        small = c["n"] <= 100000
        c.update(k=rng.randint(1, 20), noalloc=small and rng.random() < 0.5)
    return c


# ------------------------------------------------------------------ inputs
def _weighted(g, weights, seed):
    """The graph with weights drawn from `seed`, one per edge: the vertices
    and edges of a case stay the same from seed to seed."""
    rp, col, _ = g
    n = len(rp) - 1
    rows = np.repeat(np.arange(n, dtype=np.int64), np.diff(rp))
    up = rows < col
    rng = np.random.default_rng(seed)
    m = int(up.sum())
    we = rng.lognormal(0.0, 1.0, size=m) if weights == "lognormal" else rng.uniform(0.5, 1.5, size=m)
    w = np.empty(2 * m)
    w[up] = we
    low = np.nonzero(~up)[0]
    w[low[np.argsort(col[low] * np.int64(n) + rows[low])]] = we
    return rp, col, w


def _graph(family, n, weights, seed, form=1412):
    if family == "grid2d":
        a = max(2, int(math.sqrt(n)))
        return inputs.grid2d(a, max(2, -(-n // a)), weights, seed=seed)
    if family == "grid3d":
        a = max(2, round(n ** (1.0 / 3.0)))
        return inputs.grid3d(a, a, max(2, round(n / (a * a))), weights, seed=seed)
    if family == "rgg":
        g = inputs.rgg(n, 8.0, seed=form, weights="unit")
    elif family == "ba":
        g = inputs.barabasi_albert(n, 4, seed=form, weights="unit")
    else:
        g = inputs.chung_lu(n, seed=form, weights="unit")
    return _weighted(g, weights, seed)


def _case_graph(case, seed):
    return _graph(case["family"], case["n"], case["weights"], 1000 + seed)


def _batch_graphs(case, seed):
    """Sizes log-uniform in [lo, hi], families round-robin (as the mixed batch
    of the benchmark)."""
    rng = np.random.default_rng(case["graphs"])
    sizes = np.exp(rng.uniform(math.log(case["lo"]), math.log(case["hi"]), size=case["graphs"])).astype(np.int64)
    fam = ("rgg", "grid2d", "ba")
    return [_graph(fam[i % 3], int(v), "uniform", 1000 * seed + i, form=i) for i, v in enumerate(sizes)]


def _dev(g):
    return tuple(torch.from_numpy(x).to(DEV) for x in g)


def _rp32(g):
    return torch.from_numpy(g[0].astype(np.int32)).to(DEV)


def prepare(case, seed):
    kind = case["kind"]
    st = {"kind": kind, "case": case, "seed": seed}
    if kind == "batch":
        rp, col, w, offs = inputs.concat_csr(_batch_graphs(case, seed))
        st["csr"], st["offs"] = _dev((rp, col, w)), offs
        return st
    if kind == "serve":
        # a running server whose graphs are resident: every graph has been
        # solved once, alone (min_batch above the graph count)
        s = cmg.Server(workers=4, min_batch=4096, precision=case["precision"], seed=1412)
        ids = [s.add_graph(*g) for g in _batch_graphs(case, seed)]
        for t in [s.submit(i, want_vector=False) for i in ids]:
            s.wait(t)
        st["server"], st["ids"] = s, ids
        return st
    g = _case_graph(case, seed)
    n = len(g[0]) - 1
    if kind == "solve":
        st["csr"] = _dev(g) if case["mem"] == "device" else g
        return st
    if kind in ("resolve", "eigenpairs"):
        st["h"] = cmg.Hierarchy(*_dev(g), seed=1412, precision=case.get("precision", "fp64"))
        st["n"] = n
        if case.get("start") == "vector":
            st["x0"] = torch.from_numpy(np.random.default_rng(seed).standard_normal(n)).to(DEV)
        return st
    st["csr"] = (_rp32(g),) + _dev(g)[1:]
    if kind == "hec":
        st["rank"] = torch.from_numpy(np.random.default_rng(seed).permutation(n).astype(np.int32)).to(DEV)
    else:
        st["x"] = torch.from_numpy(np.random.default_rng(seed).standard_normal(n)).to(DEV)
    return st


# ------------------------------------------------------------------ the calls
def _per_level(values):
    """One value per level, for the most levels a hierarchy can have."""
    out = np.zeros(cmg.CMG_MAX_LEVELS, dtype=np.int64)
    out[:len(values)] = values
    return out


def _report(u, lam, stats):
    return {"u": u, "lambda2": lam, "residual": stats["residual"], "n": _per_level(stats["n"]),
            "nnz": _per_level(stats["nnz"]), "sweeps": _per_level(stats["sweeps"])}


def run(st):
    kind, case = st["kind"], st["case"]
    if kind == "solve":
        n = len(st["csr"][0]) - 1
        out = torch.empty(n, dtype=torch.float64, device=DEV) if case["mem"] == "device" else None
        with cmg.Hierarchy(*st["csr"], seed=st["seed"], precision=case["precision"]) as h:
            return _report(*h.fiedler(out))
    if kind == "resolve":
        out = torch.empty(st["n"], dtype=torch.float64, device=DEV)
        if "x0" in st:
            return _report(*st["h"].fiedler(out, x0=st["x0"]))
        return _report(*st["h"].fiedler(out, seed=st["seed"]))
    if kind == "eigenpairs":
        out = torch.empty((case["k"], st["n"]), dtype=torch.float64, device=DEV)
        U, lam, res, stats = st["h"].eigenpairs(case["k"], seed=st["seed"], U_out=out)
        return {"U": U, "lambda": lam, "residual": res, "sweeps": _per_level(stats["sweeps"])}
    if kind == "batch":
        out = torch.empty(int(st["offs"][-1]), dtype=torch.float64, device=DEV)
        with cmg.Batch(st["offs"], *st["csr"], seed=st["seed"], precision=case["precision"]) as b:
            u, lam, res, status = b.fiedler(out)
        return {"u": u, "lambda2": lam, "residual": res, "status": status}
    if kind == "serve":
        s = st["server"]
        tickets = [s.submit(i, seed=st["seed"] + 1) for i in st["ids"]]
        got = [s.wait(t) for t in tickets]
        return {"u": [u for u, _ in got], "lambda2": np.array([r["lambda2"] for _, r in got]),
                "residual": np.array([r["residual"] for _, r in got])}
    if kind == "hec":
        agg, c = cmg.hec_aggregate(*st["csr"], st["rank"])
        return {"agg": agg, "count": c}
    f = cmg.power_sweeps_noalloc if case["noalloc"] else cmg.power_sweeps
    u, cos = f(*st["csr"], st["x"], case["k"])
    return {"u": u, "cos": cos}


# ------------------------------------------------------------------ work
def _size(family, n):
    """Vertices and stored entries of a family's graph, about."""
    if family == "grid2d":
        return n, 4 * n - 4 * int(math.sqrt(n))
    if family == "grid3d":
        return n, 6 * n - 6 * round(n ** (2.0 / 3.0))
    if family == "chung_lu":
        return n, 16 * n
    return n, 8 * n


def work(case):
    """One reading of the graph and one writing of the result; the operations
    of the sweeps where their number is given."""
    kind = case["kind"]
    if kind in ("batch", "serve"):
        mean = (case["hi"] - case["lo"]) / math.log(case["hi"] / case["lo"])
        n, nnz = int(mean * case["graphs"]), int(6.7 * mean * case["graphs"])
        return {"bytes": 12 * nnz + 16 * n, "flops": 0}
    n, nnz = _size(case["family"], case["n"])
    if kind == "eigenpairs":
        return {"bytes": 12 * nnz + 8 * n * (1 + case["k"]), "flops": 0}
    if kind == "hec":
        return {"bytes": 12 * nnz + 12 * n, "flops": 0}
    if kind == "sweeps":
        return {"bytes": 12 * nnz + 20 * n, "flops": case["k"] * (2 * nnz + 9 * n)}
    return {"bytes": 12 * nnz + 16 * n, "flops": 0}


# ------------------------------------------------------------------ 64-bit reference
# The method as its paper states it (arXiv 1412.0565, Alg. 1-3), sequential
# coarsening in numpy and power iteration in torch, with the library's keyed
# visit order and Gaussian start.
_U = np.uint64


def _mix(x):
    with np.errstate(over="ignore"):
        z = x + _U(0x9E3779B97F4A7C15)
        z = (z ^ (z >> _U(30))) * _U(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> _U(27))) * _U(0x94D049BB133111EB)
        return z ^ (z >> _U(31))


def _ranks(n, seed, level):
    """Keyed 4-round Feistel permutation of [0, 2^k), walked onto [0, n)."""
    k = 2
    while (1 << k) < n:
        k += 2
    half, mask = _U(k // 2), _U((1 << (k // 2)) - 1)
    base = (seed ^ (level * 0x9E3779B97F4A7C15)) & 0xFFFFFFFFFFFFFFFF
    keys = [_mix(np.array([base ^ t], dtype=_U))[0] for t in range(4)]
    x = np.arange(n, dtype=_U)
    todo = np.ones(n, dtype=bool)
    while todo.any():
        L, R = x[todo] >> half, x[todo] & mask
        for t in range(4):
            L, R = R, L ^ (_mix(R ^ keys[t]) & mask)
        x[todo] = (L << half) | R
        todo[todo] = x[todo] >= n
    return x.astype(np.int64)


def _gaussian(n, seed):
    i = np.arange(n, dtype=_U)
    base = _U(seed ^ 0xC0A45E)
    a, b = _mix(base ^ (_U(2) * i)), _mix(base ^ (_U(2) * i + _U(1)))
    u1, u2 = ((v >> _U(11)).astype(np.float64) + 1.0 for v in (a, b))
    return np.sqrt(-2.0 * np.log(u1 * 2.0 ** -53)) * np.cos(2.0 * np.pi * (u2 * 2.0 ** -53))


def _hec(rp, col, w, rank):
    """Alg. 2: visit in rank order; an unmapped vertex joins its heaviest
    neighbour's aggregate or opens one with it."""
    n = len(rp) - 1
    rows = np.repeat(np.arange(n), np.diff(rp))
    top = np.maximum.reduceat(w, rp[:-1])
    at = np.nonzero(w == top[rows])[0]
    heavy = np.empty(n, dtype=np.int64)
    heavy[rows[at[::-1]]] = col[at[::-1]]    # the lowest column wins
    order = np.empty(n, dtype=np.int64)
    order[rank] = np.arange(n)
    heavy, agg, c = heavy.tolist(), [-1] * n, 0
    for v in order.tolist():
        if agg[v] < 0:
            m = heavy[v]
            if agg[m] < 0:
                agg[v] = agg[m] = c
                c += 1
            else:
                agg[v] = agg[m]
    return np.array(agg, dtype=np.int64), c


def _coarse(rp, col, w, agg, c):
    n = len(rp) - 1
    a, b = agg[np.repeat(np.arange(n), np.diff(rp))], agg[col]
    cross = a != b
    key, ww = a[cross] * c + b[cross], w[cross]
    o = np.argsort(key, kind="stable")
    key, ww = key[o], ww[o]
    head = np.nonzero(np.concatenate(([True], key[1:] != key[:-1])))[0]
    rows = key[head] // c
    out = np.zeros(c + 1, dtype=np.int64)
    np.cumsum(np.bincount(rows, minlength=c), out=out[1:])
    return out, key[head] % c, np.add.reduceat(ww, head)


def _levels(g, seed):
    rp, col, w = g[0], g[1].astype(np.int64), g[2]
    lv, maps = [(rp, col, w)], []
    while len(lv[-1][0]) - 1 > 25 and len(lv) < 64:
        rp, col, w = lv[-1]
        agg, c = _hec(rp, col, w, _ranks(len(rp) - 1, seed, len(maps)))
        if c < 2:
            break
        maps.append(agg)
        lv.append(_coarse(rp, col, w, agg, c))
    return lv, maps


class _Op:
    """B_g = g I - L of one level."""

    def __init__(self, rp, col, w):
        t = [torch.from_numpy(np.ascontiguousarray(x)).to(DEV) for x in (rp, col, w)]
        n = len(rp) - 1
        self.A = torch.sparse_csr_tensor(t[0], t[1].long(), t[2], size=(n, n))
        self.d = self.A @ torch.ones(n, dtype=torch.float64, device=DEV)
        self.g = float(2.0 * self.d.max())

    def mul(self, x):
        d = self.d if x.dim() == 1 else self.d[:, None]
        return self.g * x - d * x + self.A @ x

    def lap(self, x):
        d = self.d if x.dim() == 1 else self.d[:, None]
        return d * x - self.A @ x


def _iterate(op, x, most, k=None, tol=1e-8):
    """Alg. 3 from x: (unit vector, sweeps, last cosine)."""
    x = x - x.mean()
    x = x / x.norm()
    s, cos = 0, 0.0
    while s < (most if k is None else k):
        y = op.mul(x)
        y = y - y.mean()
        nrm = float(y.norm())
        s += 1
        if nrm <= 64 * 2.220446049250313e-16 * op.g:
            return x, s, 1.0
        y = y / nrm
        cos = float(y @ x)
        x = y
        if k is None and cos >= 1.0 - tol:
            break
    return x, s, cos


def _orthonormal(X):
    X = X - X.mean(0)
    Q, R = torch.linalg.qr(X)
    return Q * torch.sign(torch.diagonal(R))


def _iterate_block(op, X, most, tol=1e-8):
    X = _orthonormal(X)
    s = 0
    while s < most:
        Y = _orthonormal(op.mul(X))
        s += 1
        done = bool(((Y * X).sum(0) >= 1.0 - tol).all())
        X = Y
        if done:
            break
    return X, s


def _signed(u):
    return u if float(u[torch.argmax(u.abs())]) > 0 else -u


def _quotient(op, u):
    lu = op.lap(u)
    lam = float(u @ lu)
    return lam, float((lu - lam * u).norm())


def _cascade(lv, maps, seed, x0=None, k=0):
    """Alg. 1 Steps 2-3; k > 0: k vectors at once."""
    J = len(lv) - 1
    sweeps = [0] * (J + 1)
    x = None
    for j in range(0 if x0 is not None else J, -1, -1):
        n = len(lv[j][0]) - 1
        if x is None and x0 is not None:
            x = x0
        elif x is None:
            x = torch.from_numpy(np.stack([_gaussian(n, seed + i) for i in range(max(k, 1))], 1)).to(DEV)
            x = x if k else x[:, 0]
        else:
            x = x[torch.from_numpy(maps[j]).to(DEV)]
        op = _Op(*lv[j])
        most = 100000 if j == J else 20000
        if k:
            x, sweeps[j] = _iterate_block(op, x, most)
        else:
            x, sweeps[j], _ = _iterate(op, x, most)
    return op, x, sweeps


def _solve_exact(g, setup_seed, solve_seed, x0=None):
    lv, maps = _levels(g, setup_seed)
    op, u, sweeps = _cascade(lv, maps, solve_seed, x0)
    u = _signed(u)
    lam, res = _quotient(op, u)
    return _report(u, lam, {"residual": res, "n": [len(L[0]) - 1 for L in lv], "nnz": [len(L[1]) for L in lv],
                            "sweeps": sweeps})


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return None      # hundreds of sequential solves: minutes
    if kind == "serve":
        if case["hi"] > 20000 or case["graphs"] > 8:
            return None
        got = [_solve_exact(g, 1412, seed + 1) for g in _batch_graphs(case, seed)]
        return {"u": [r["u"].cpu().numpy() for r in got], "lambda2": np.array([r["lambda2"] for r in got]),
                "residual": np.array([r["residual"] for r in got])}
    g = _case_graph(case, seed)
    if kind == "solve":
        r = _solve_exact(g, seed, seed)
        return dict(r, u=r["u"].cpu().numpy()) if case["mem"] == "host" else r
    if kind == "resolve":
        x0 = None
        if case["start"] == "vector":
            x0 = torch.from_numpy(np.random.default_rng(seed).standard_normal(len(g[0]) - 1)).to(DEV)
        return _solve_exact(g, 1412, seed, x0)
    if kind == "eigenpairs":
        k = case["k"]
        lv, maps = _levels(g, 1412)
        op, X, sweeps = _cascade(lv, maps, seed, k=k)
        cols = [_signed(X[:, i]) for i in range(k)]
        lam, res = zip(*(_quotient(op, u) for u in cols))
        return {"U": torch.stack(cols).contiguous(), "lambda": np.array(lam), "residual": np.array(res),
                "sweeps": _per_level(sweeps)}
    if kind == "hec":
        rank = np.random.default_rng(seed).permutation(len(g[0]) - 1)
        agg, c = _hec(g[0], g[1], g[2], rank)
        return {"agg": torch.from_numpy(agg.astype(np.int32)).to(DEV), "count": c}
    x = torch.from_numpy(np.random.default_rng(seed).standard_normal(len(g[0]) - 1)).to(DEV)
    u, _, cos = _iterate(_Op(*g), x, case["k"], k=case["k"])
    return {"u": u, "cos": cos}
