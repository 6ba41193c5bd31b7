"""Every form of the sweep kernels of a single graph, named by the library and
checked against the same sweeps in extended precision: the fixed-point kernels at
the lines of their plans, the levels that leave them, and the FP32 slice kernel
with its layout resident.

Bars on the vector after k sweeps.  Fixed point: three FP64 roundings of the
result's entries and two of its scale, and half a unit of 2^-62 of the largest
entry per row and sweep (0.29 of one as a standard deviation, times two).  FP64 kernels: 2^-52 of the vector for
each of four roundings a sweep, and the same again for the rows' sums."""
import numpy as np
import pytest

from paper_1412_0565_gb300 import cmg, inputs
from test_gpu_localised import sweeps
from test_gpu_rows import EDGES, ladder

pytestmark = pytest.mark.gpu

K = 7
CASES = {
    # name: (graph, form of level 0, environment)
    "registers_8_steps": (lambda: inputs.grid2d(18, 13, "uniform", seed=1), "fix_registers", {}),
    "registers_16_steps": (lambda: inputs.random_connected(900, 9000, seed=3), "fix_registers", {}),
    "shared": (lambda: inputs.random_connected(3000, 24000, seed=4), "fix_shared", {}),
    "resident": (lambda: inputs.grid2d(100, 101, "uniform", seed=2), "rows_resident", {}),
    "resident_edges_odd": (lambda: ladder(60002, EDGES + [7, 3], 2), "rows_resident", {}),
    "resident_longest_row": (lambda: ladder(60000, [4090, 2000], 3), "rows_resident", {}),
    "resident_most_16_bit_columns": (lambda: ladder(65533, [40, 50, 60], 5), "rows_resident", {}),
    "resident_32_bit_columns": (lambda: ladder(65534, [40, 50, 60], 5), "rows_resident", {}),
    "staged_edges": (lambda: ladder(6000, EDGES, 1), "rows_staged", {}),
    "staged_edges_odd": (lambda: ladder(6002, EDGES + [7, 3], 2), "rows_staged", {}),
    "staged_longest_row": (lambda: ladder(9000, [4090, 2000], 3), "rows_staged", {}),
    "staged": (lambda: inputs.random_connected(3000, 150000, seed=6), "rows_staged", {}),
    "staged_odd": (lambda: inputs.random_connected(3001, 150000, seed=7), "rows_staged", {}),
    "streamed": (lambda: inputs.random_connected(60001, 1900000, seed=8), "rows_streamed", {}),
    "streamed_32_bit_columns": (lambda: inputs.grid3d(70, 71, 72, "uniform", seed=9), "rows_streamed", {}),
    "streamed_most_rows": (lambda: ladder((1 << 20) - 3, [40, 50, 60], 5), "rows_streamed", {}),
    "evict_first": (lambda: inputs.random_connected(60001, 7300000, seed=10), "rows_evict_first", {}),
    "evict_first_32_bit_columns": (lambda: inputs.random_connected(70001, 6300000, seed=11), "rows_evict_first", {}),
    "row_too_long": (lambda: ladder(9000, [4200], 4), "slice", {}),
    "one_row_too_many": (lambda: ladder((1 << 20) - 2, [40, 50, 60], 5), "slice", {}),
    "slice_by_choice": (lambda: ladder(6000, EDGES, 1), "slice", {"CMG_STAGE": "0"}),
    "staged_slice_by_choice": (lambda: ladder(6000, EDGES, 1), "slice_staged", {"CMG_STAGE": "1"}),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_each_form_runs_where_it_is_named(monkeypatch, name):
    make, form, env = CASES[name]
    for k, v in env.items():
        monkeypatch.setenv(k, v)
    rp, col, w = make()
    n = len(rp) - 1
    x0 = np.random.default_rng(n).standard_normal(n) + 0.5
    with cmg.Hierarchy(rp, col, w, seed=1412, max_levels=1, schedule="replay", replay_sweeps=[K]) as h:
        forms, ctas = h.level_forms()
        g = h.level_csr(0)[3]
        u, lam, st = h.fiedler(x0=x0)
        u2 = h.fiedler(x0=x0)[0]
    assert forms == [form]
    assert (ctas[0] > 0) == (form.startswith("fix") or form.startswith("rows"))
    assert np.array_equal(u, u2)
    ref = sweeps(rp, col, w, g, x0, K)
    u = u.astype(np.longdouble)
    if (u * ref).sum() < 0:
        u = -u
    err = float(np.sqrt(((u - ref) ** 2).sum()))
    if form.startswith("slice"):
        bar = 8 * 2.0 ** -52 * K
    else:
        bar = 5 * 2.0 ** -53 + 2 * 0.29 * 2.0 ** -62 * np.sqrt(K * n) * float(np.abs(ref).max()) * np.sqrt(K)
    assert err <= bar


DENSE = {
    "slices": lambda: inputs.random_connected(6000, 1500000, seed=9),
    # rows of 5,200 entries are cut into chunks that go to several CTAs
    "chunks": lambda: inputs.csr_from_edges(6000, *dense_with_hubs(6000, 1400000, 9, 5200, seed=10)),
}


def dense_with_hubs(n, m, hubs, degree, seed):
    rng = np.random.default_rng(seed)
    u = np.concatenate([np.arange(n - 1), rng.integers(0, n, m)] + [np.full(degree, h) for h in range(hubs)])
    v = np.concatenate([np.arange(1, n), rng.integers(0, n, m)]
                       + [hubs + rng.choice(n - hubs, degree, replace=False) for _ in range(hubs)])
    lo, hi = np.minimum(u, v), np.maximum(u, v)
    key = np.unique(lo[lo < hi].astype(np.int64) * n + hi[lo < hi])
    return key // n, key % n, rng.uniform(0.5, 1.5, key.size)


@pytest.mark.parametrize("name", sorted(DENSE))
def test_resident_fp32_layout_gives_the_streamed_bits(monkeypatch, name):
    rp, col, w = DENSE[name]()
    x0 = np.random.default_rng(1).standard_normal(6000)
    got = {}
    for mode, form in (("0", "slice_staged"), ("1", "slice_resident")):
        monkeypatch.setenv("CMG_RESIDENT", mode)
        with cmg.Hierarchy(rp, col, w, seed=1412, precision="fp32", max_levels=1, schedule="replay",
                           replay_sweeps=[40]) as h:
            assert h.level_forms()[0] == [form]
            got[mode] = h.fiedler(x0=x0)
    assert np.array_equal(got["0"][0], got["1"][0]) and got["0"][1] == got["1"][1]


@pytest.mark.parametrize("switch", ["0", "128", "1000", "2000", "9000"])
def test_cluster_switch_keeps_smaller_levels_on_one_cta(monkeypatch, switch):
    """CMG_CLUSTER=<rows>: no level of fewer rows takes a cluster, whatever the plan
    would have given it; larger levels take the plan's."""
    rp, col, w = inputs.grid2d(64, 64, "uniform", seed=3)
    with cmg.Hierarchy(rp, col, w, seed=1412) as h:
        free = h.level_forms()[1]
        u0 = h.fiedler()[0]
    monkeypatch.setenv("CMG_CLUSTER", switch)
    with cmg.Hierarchy(rp, col, w, seed=1412) as h:
        forms, ctas = h.level_forms()
        kinds, n = h.level_kernels()[0], h.sizes()[0]
        u = h.fiedler()[0]
    least = int(switch) if int(switch) else 1 << 30
    assert any(c > 1 and rows < 512 for c, rows in zip(free, n))
    for f, c, k, rows, plan in zip(forms, ctas, kinds, n, free):
        if f.startswith("fix"):
            assert c == (plan if rows >= least else 1)
            assert k == (5 if c > 1 else 0)
    assert np.linalg.norm(u - u0) <= 1e-10
