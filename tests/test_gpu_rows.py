"""The row kernel (resident and streaming) against the oracle, at the edges of
its plan: lanes per row change at 8 / 16, 16 / 32, ... entries, an item is 32
lanes, and a row of more than 4,096 entries leaves the level to the slice
kernel."""
import numpy as np
import pytest

import oracle
from paper_1412_0565_gb300 import cmg, inputs

pytestmark = pytest.mark.gpu


def aligned_err(u, ref):
    if np.dot(u, ref) < 0:
        u = -u
    return np.linalg.norm(u - ref) / np.linalg.norm(ref)


def ladder(n, degrees, seed):
    """A weighted cycle of n vertices plus one star per entry of `degrees`
    (centre k joined to that many cycle vertices): rows of chosen lengths."""
    rng = np.random.default_rng(seed)
    u = [np.arange(n)]
    v = [(np.arange(n) + 1) % n]
    for k, d in enumerate(degrees):
        u.append(np.full(d, n + k))
        v.append(rng.choice(n, size=d, replace=False))
    u, v = np.concatenate(u), np.concatenate(v)
    w = rng.uniform(0.5, 1.5, size=u.size)
    w[n:] *= 0.05       # the stars do not set the shift
    return inputs.csr_from_edges(n + len(degrees), u, v, w)


EDGES = [8, 9, 16, 17, 31, 32, 33, 63, 64, 65, 127, 128, 129, 255, 256, 257, 511, 513, 1000]
CASES = {
    "edges": lambda: ladder(6000, EDGES, 1),
    "edges_odd": lambda: ladder(6001, EDGES + [7, 3], 2),
    "longest_item_row": lambda: ladder(9000, [4090, 2000], 3),
    "beyond_the_items": lambda: ladder(9000, [4200], 4),
    "dense_levels": lambda: inputs.barabasi_albert(9000, 4, seed=5),
    "streaming": lambda: inputs.grid3d(90, 90, 90, "uniform", seed=6),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_row_kernel_fp64_matches_oracle(monkeypatch, name):
    """FP64 bars of the whole method (1e-10 on the vector, 1e-12 on lambda2,
    the same sweeps), and bit-identical repeats."""
    monkeypatch.setenv("CMG_CLUSTER", "0")   # every level beyond one CTA takes the row kernel
    rp, col, w = CASES[name]()
    with cmg.Hierarchy(rp, col, w, seed=1412) as h:
        assert h.level_kernels()[0][0] == 1
        u, lam, st = h.fiedler()
        u2, lam2, _ = h.fiedler()
    assert np.array_equal(u, u2) and lam == lam2
    ref_u, ref_lam, _, oh, ref = oracle.fiedler(rp, col, w, seed=1412)
    assert st["sweeps"] == ref["sweeps"].tolist()
    assert aligned_err(u, ref_u) <= 1e-10
    assert abs(lam - ref_lam) <= 1e-12 * abs(ref_lam)


def test_resident_fp32_levels_give_the_slice_kernels_bits(monkeypatch):
    """FP32 levels held in shared memory keep the slice kernel's CTAs, warps and
    order: bit for bit the vector of the slice kernel reading its layout from
    L2 (CMG_RESIDENT=0)."""
    rp, col, w = inputs.chung_lu(80000, seed=21)
    got = {}
    for mode in ("0", "1"):
        monkeypatch.setenv("CMG_RESIDENT", mode)
        with cmg.Hierarchy(rp, col, w, seed=1412, precision="fp32") as h:
            assert "fp32" in h.level_precision()
            u, lam, st = h.fiedler()
        got[mode] = (u, st["sweeps"])
    assert got["0"][1] == got["1"][1]
    assert np.array_equal(got["0"][0], got["1"][0])
