"""g(r) histogram at the edges of its kernel: windows that name every cell of a
row once, runs of home cells cut by the box, one bin and the most bins (bin
edges closer than binary32 resolves), a crowded cell.  Counts are whole numbers
and must be equal."""
import numpy as np
import pytest

import oracle as O
from paper_1804_06205_gb300 import workloads as W

pytestmark = pytest.mark.gpu

BOXES = [((7.0, 7.9, 9.3), 3.0), ((3.0, 3.5, 4.0), 1.0), ((13.2, 5.0, 5.7), 2.0), ((16.0, 11.0, 9.0), 2.5)]


def _positions(L, n, crowd, seed):
    rng = np.random.default_rng(seed)
    L = np.asarray(L)
    pos = rng.uniform(0, 1, (n, 3)) * L
    pos[: n // 8] = np.floor(pos[: n // 8])          # on faces: distances at bin edges
    pos[n - crowd:] = rng.uniform(0.1, 0.9, (crowd, 3))
    return np.where(pos >= L, 0.0, pos)


@pytest.mark.parametrize("L,rmax", BOXES)
@pytest.mark.parametrize("nbins", [1, 60, 4096])
def test_counts_fp64(L, rmax, nbins):
    from paper_1804_06205_gb300 import dpd as D
    w = W.fluid(L, seed=3)
    pos = _positions(L, w.n, min(w.n // 2, 150), 4)
    g = D.System.from_workload(w, precision=D.DPD_FP64)
    g.set_state(pos, w.vel, 0)
    s = O.System(w.L, w.types, w.a, w.gamma, w.kT, w.dt, w.lam)
    assert np.array_equal(g.gr_counts(rmax, nbins), O.gr_counts(s, O.wrap(s, pos), rmax, nbins))


@pytest.mark.parametrize("nbins", [1, 75, 4096])
def test_counts_fp32(nbins):
    """Against all pairs of the exact cells and offsets (cell edges are 1)."""
    from paper_1804_06205_gb300 import dpd as D
    L, rmax = np.array([9.0, 7.0, 8.0]), 3.0
    w = W.fluid(L, seed=5)
    g = D.System.from_workload(w, precision=D.DPD_FP32)
    g.set_state(_positions(L, w.n, 100, 6), w.vel, 0)
    g.step(2)
    rec = np.frombuffer(g.get_checkpoint()[80:], dtype=np.dtype([("key", "<u4"), ("o", "<f4", 3), ("vf", "<f4", 6)]))
    key = rec["key"].astype(np.int64)
    cell = np.stack([key % 9, key // 9 % 7, key // 63], 1)
    o = rec["o"].astype(np.float64)
    i, j = np.triu_indices(w.n, 1)
    dc = cell[i] - cell[j]
    dc = dc - (L * np.rint(dc / L)).astype(np.int64)
    d = (o[i] - o[j]) + dc
    r = np.sqrt((d[:, 0] ** 2 + d[:, 1] ** 2) + d[:, 2] ** 2)
    dr = rmax / nbins
    bins = np.floor(r[r < rmax] / dr).astype(np.int64)
    want = np.bincount(bins[bins < nbins], minlength=nbins)
    assert np.array_equal(g.gr_counts(rmax, nbins).astype(np.int64), want)
