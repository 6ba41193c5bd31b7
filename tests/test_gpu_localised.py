"""Fixed-point sweeps of vectors that live on a few vertices (a pendant path, a
vertex behind a weak edge): the fixed point has one unit for the whole vector,
so this is where it can fall behind FP64, whose units follow each entry.

Reference: the same sweeps in extended precision.  Bar on the vector: the
result's own three FP64 roundings of its largest entry (the mean, the scale, the
store), and the sweeps' roundings of half a unit of 2^-62 of the largest entry
per row, 0.29 of one as a standard deviation, added up undamped over the sweeps
with their standard deviation times two."""
import numpy as np
import pytest

from paper_1412_0565_gb300 import cmg, inputs

pytestmark = pytest.mark.gpu


def with_tail(n, tail, weight, seed):
    """Barabasi-Albert graph with a path of `tail` vertices hanging from vertex 5,
    every edge of it of the given weight."""
    rp, col, w = inputs.barabasi_albert(n, 4, seed=seed)
    rows = np.repeat(np.arange(n), np.diff(rp))
    up = rows < col
    u = np.concatenate([rows[up], [5], np.arange(n, n + tail - 1)])
    v = np.concatenate([col[up], np.arange(n, n + tail)])
    return inputs.csr_from_edges(n + tail, u, v, np.concatenate([w[up], np.full(tail, weight)]))


def sweeps(rp, col, w, g, x, k):
    x = x.astype(np.longdouble)
    w, rows = w.astype(np.longdouble), np.repeat(np.arange(len(rp) - 1), np.diff(rp))
    x = x - x.mean()
    for _ in range(k):
        x = x + np.add.reduceat(w * (x[col] - x[rows]), rp[:-1]) / np.longdouble(g)
    x = x - x.mean()
    return x / np.sqrt((x * x).sum())


@pytest.mark.parametrize("tail,weight", [(10, 1.0), (1, 0.01)])
@pytest.mark.parametrize("n", [600, 3000, 20000, 60000, 250000])
def test_localised_vectors_keep_fp64_accuracy(n, tail, weight):
    k = 100
    rp, col, w = with_tail(n, tail, weight, seed=n)
    N = n + tail
    x0 = 1e-6 * np.random.default_rng(n).standard_normal(N)
    x0[n:] += np.sin(np.arange(1, tail + 1) / tail)
    with cmg.Hierarchy(rp, col, w, seed=1412, max_levels=1, schedule="replay", replay_sweeps=[k]) as h:
        g = h.level_csr(0)[3]
        u, lam, st = h.fiedler(x0=x0)
    assert st["sweeps"] == [k]
    ref = sweeps(rp, col, w, g, x0, k)
    u = u.astype(np.longdouble)
    if (u * ref).sum() < 0:
        u = -u
    err = float(np.sqrt(((u - ref) ** 2).sum()))
    assert err <= 3 * 2.0 ** -53 + 2 * 0.29 * 2.0 ** -62 * np.sqrt(k * N)
