"""The fixed-point sweeps of small FP64 levels against the oracle, at the edges of
their plan (one item per warp of 8 or 16 steps, items dealt by entries, one CTA
or a cluster) and of their arithmetic (weights over many orders of magnitude,
constant-magnitude and localised vectors, annihilated iterates, start vectors
of any scale and with infinities)."""
import numpy as np
import pytest

import oracle
from paper_1412_0565_gb300 import cmg, inputs

pytestmark = pytest.mark.gpu


def aligned_err(u, ref):
    if np.dot(u, ref) < 0:
        u = -u
    return np.linalg.norm(u - ref) / np.linalg.norm(ref)


def check(g, **kw):
    with cmg.Hierarchy(*g, seed=1412, **kw) as h:
        kinds = h.level_kernels()[0]
        u, lam, st = h.fiedler()
        u2, lam2, _ = h.fiedler()
    assert np.array_equal(u, u2) and lam == lam2
    ref_u, ref_lam, _, oh, ref = oracle.fiedler(*g, seed=1412)
    assert st["sweeps"] == ref["sweeps"].tolist()
    assert aligned_err(u, ref_u) <= 1e-10
    assert abs(lam - ref_lam) <= 1e-12 * abs(ref_lam)
    return kinds


def two_cliques(m, weak):
    iu = np.triu_indices(m, 1)
    u = np.concatenate([iu[0], iu[0] + m, [0]])
    v = np.concatenate([iu[1], iu[1] + m, [m]])
    w = np.concatenate([np.ones(2 * iu[0].size), [weak]])
    return inputs.csr_from_edges(2 * m, u, v, w)


def spread(n, extra, decades, seed):
    """Random connected graph with weights over `decades` orders of magnitude."""
    rp, col, w = inputs.random_connected(n, extra, seed=seed)
    rows = np.repeat(np.arange(n), np.diff(rp))
    up = rows < col
    rng = np.random.default_rng(seed)
    return inputs.csr_from_edges(n, rows[up], col[up], 10.0 ** rng.uniform(-decades, 0, size=int(up.sum())))


CASES = {
    "one_warp": lambda: inputs.path(20),
    "one_cta": lambda: inputs.grid2d(18, 13, "uniform", seed=1),
    "steps_8_edge": lambda: inputs.random_connected(470, 400, seed=2),
    "steps_16": lambda: inputs.random_connected(900, 9000, seed=3),
    "row_of_512": lambda: inputs.hub_grid(30, 30, 512, seed=4, hub_scale=1e-2),
    "row_of_513": lambda: inputs.hub_grid(30, 30, 513, seed=4, hub_scale=1e-2),
    "by_entries": lambda: inputs.barabasi_albert(1500, 24, seed=5),
    "most_rows": lambda: inputs.grid2d(64, 64, "uniform", seed=6),
    "odd_rows": lambda: inputs.rgg(4000, 8.0, seed=7),
    "constant_magnitude": lambda: two_cliques(130, 1e-3),
    "weights_over_8_decades": lambda: spread(700, 2100, 8.0, 8),
}


@pytest.mark.parametrize("clusters", [True, False])
@pytest.mark.parametrize("name", sorted(CASES))
def test_fixed_point_levels_match_oracle(monkeypatch, name, clusters):
    if not clusters:
        monkeypatch.setenv("CMG_CLUSTER", "0")
    kinds = check(CASES[name]())
    if clusters:
        assert kinds[0] in (0, 5)


@pytest.mark.parametrize("power", [-600, 600])
def test_scaled_weights_give_the_same_vector(power):
    """Weights times a power of two: the same hierarchy, sweeps and vector (the
    oracle's own squares leave the doubles' range here)."""
    rp, col, w = inputs.grid2d(20, 21, "uniform", seed=9)
    u, lam, st = cmg.fiedler(rp, col, w, seed=1412)
    u2, lam2, st2 = cmg.fiedler(rp, col, w * 2.0 ** power, seed=1412)
    assert st2["sweeps"] == st["sweeps"] and np.array_equal(u2, u)
    assert lam2 == lam * 2.0 ** power


def test_annihilated_iterate_keeps_the_previous_one():
    """n = 2: B_g maps the mean-free vector to 0 in the first sweep."""
    u, lam, st = cmg.fiedler(*inputs.path(2), seed=1412)
    assert st["sweeps"] == [1] and st["cos_final"] == [1.0]
    assert abs(abs(u[0]) - np.sqrt(0.5)) <= 1e-13 and lam == pytest.approx(2.0, rel=1e-12)


@pytest.mark.parametrize("scale", [1e-250, 1e-3, 1.0, 1e30, 1e250])
def test_start_vectors_of_any_scale(scale):
    """Only the direction of a start vector counts."""
    g = inputs.grid2d(30, 31, "uniform", seed=3)
    x0 = np.random.default_rng(1).standard_normal(930)
    oh = oracle.Hierarchy(*g, seed=1412)
    r = oh.solve(start_level=0, x0=x0)
    with cmg.Hierarchy(*g, seed=1412) as h:
        u, lam, st = h.fiedler(x0=x0 * scale)
    assert st["sweeps"] == r["sweeps"].tolist()
    assert aligned_err(u, r["u"]) <= 1e-10


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_start_vector_that_is_not_finite(bad):
    g = inputs.grid2d(20, 20, "uniform", seed=3)
    x0 = np.random.default_rng(1).standard_normal(400)
    x0[7] = bad
    with cmg.Hierarchy(*g, seed=1412, max_sweeps=50) as h:
        u, lam, st = h.fiedler(x0=x0)
    assert np.isnan(u).any() and st["status"] == "WARN_MAXITER"


def test_no_sweeps_returns_the_projected_start():
    g = inputs.grid2d(25, 20, "uniform", seed=3)
    x0 = np.random.default_rng(2).standard_normal(500) + 3.0
    with cmg.Hierarchy(*g, seed=1412, schedule="replay", replay_sweeps=[0] * 64) as h:
        u, lam, st = h.fiedler(x0=x0)
    ref = x0 - x0.mean()
    assert st["sweeps"][0] == 0
    assert aligned_err(u, ref / np.linalg.norm(ref)) <= 1e-12


def test_unchecked_weights_outside_the_contract_keep_fp64_sweeps():
    """validate=0 takes weights that are not positive; the fixed-point sweeps rely
    on positive ones, so such a graph keeps the FP64 kernels: the signed operator
    is iterated as it is (one sweep against plain numpy)."""
    rp, col, w = inputs.grid2d(12, 11, "uniform", seed=2)
    rows = np.repeat(np.arange(132), np.diff(rp))
    w = np.where((rows + col) % 7 == 3, -0.1 * w, w)
    x0 = np.random.default_rng(3).standard_normal(132)
    with cmg.Hierarchy(rp, col, w, seed=1412, validate=0, max_levels=1, schedule="replay", replay_sweeps=[1]) as h:
        g = h.level_csr(0)[3]
        u, lam, st = h.fiedler(x0=x0)
    x = x0 - x0.mean()
    d = np.zeros(132)
    np.add.at(d, rows, w)
    y = (g - d) * x
    np.add.at(y, rows, w * x[col])
    y -= y.mean()
    assert aligned_err(u, y / np.linalg.norm(y)) <= 1e-12
