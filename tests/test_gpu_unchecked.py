"""validate = 0 on weights that differ by direction: the fixed-point sweeps rely on
a symmetric matrix (they keep the mean and the sums by it), so such a graph keeps
the FP64 kernels, which iterate the operator as it is."""
import numpy as np
import pytest

from paper_1412_0565_gb300 import cmg, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("a,b", [(30, 31), (70, 80)])
def test_weights_that_differ_by_direction_keep_fp64_sweeps(a, b):
    """400 sweeps from a ramp, whose mean drifts from sweep to sweep, against plain
    numpy: 8 roundings of 2^-53 a sweep, on a vector whose constant part has grown to
    at most 100 times the rest."""
    rp, col, w = inputs.grid2d(a, b, "uniform", seed=2)
    n = a * b
    rows = np.repeat(np.arange(n), np.diff(rp))
    w = np.where(rows < col, 3.0 * w, w)
    x0 = np.linspace(-1.0, 1.0, n)
    k = 400
    with cmg.Hierarchy(rp, col, w, seed=1412, validate=0, max_levels=1, schedule="replay", replay_sweeps=[k]) as h:
        forms = h.level_forms()[0]
        g = h.level_csr(0)[3]
        u, lam, st = h.fiedler(x0=x0)
    assert not forms[0].startswith(("fix", "rows"))
    x = x0 - x0.mean()
    for _ in range(k):
        x = x + np.add.reduceat(w * (x[col] - x[rows]), rp[:-1]) / g
        x -= x.mean()
    x /= np.linalg.norm(x)
    if np.dot(u, x) < 0:
        u = -u
    assert np.linalg.norm(u - x) <= 100 * 8 * 2.0 ** -53 * k


@pytest.mark.parametrize("a,b", [(30, 31), (70, 80)])
def test_an_unchecked_graph_inside_the_contract_keeps_its_kernels(a, b):
    g = inputs.grid2d(a, b, "uniform", seed=2)
    got = []
    for v in (0, 1):
        with cmg.Hierarchy(*g, seed=1412, validate=v) as h:
            got.append((h.level_forms(), h.fiedler()[0]))
    assert got[0][0] == got[1][0] and got[0][0][0][0].startswith(("fix", "rows"))
    assert np.array_equal(got[0][1], got[1][1])
