"""Crowded cells in the gather by cell (systems of at least 262,144 beads in id order:
set_state, a restored checkpoint): cells at the limit up to which eight threads rank a
cell's beads (64), one more, and one of thousands, whose beads are ranked a thread per
bead.  Cells are compared with the oracle's and a run resumed by a checkpoint with the
same run gone on with, bit for bit."""
import numpy as np
import pytest

import oracle as O
from paper_1804_06205_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,big", [(262_144, 2_000), (262_145, 0)])   # 0: no cell is left over
def test_crowded_cells_by_cell(n, big):
    from paper_1804_06205_gb300 import dpd as D
    w = W.fluid((45.0, 44.2, 45.0), n=n, seed=61)
    rng = np.random.default_rng(62)
    h = w.L / np.floor(w.L)
    crowds = (9, 16, 17, 40, 50) + ((64, 65, 66, 300, big) if big else ())
    at = 0
    for k, beads in enumerate(crowds):
        cell = np.array([3 + 4 * k, 5, 44])          # apart from one another
        w.pos[at:at + beads] = (cell % np.floor(w.L) + rng.uniform(0.02, 0.98, (beads, 3))) * h
        at += beads
    w.pos = w.pos[rng.permutation(n)]                 # the crowds' ids everywhere
    s = O.System(w.L, w.types, w.a, w.gamma, w.kT, w.dt, w.lam)
    key = O.cell_keys(s, O.wrap(s, w.pos))
    order, start = O.cell_sort(s, key)
    assert np.diff(start).max() >= max(crowds)
    for prec in (D.DPD_FP32, D.DPD_FP64):
        g = D.System.from_workload(w, precision=prec)
        g.set_state(w.pos, w.vel * 0.1, 0)
        gk, go, gs = g.cells()
        assert np.array_equal(gk, key) and np.array_equal(go, order) and np.array_equal(gs, start)
        ck = g.get_checkpoint()
        g.set_checkpoint(ck)                          # sorted on demand, from id order
        gk, go, gs = g.cells()
        assert np.array_equal(gk, key) and np.array_equal(go, order) and np.array_equal(gs, start)
        g.step(1)
        on = g.get_state()[:3] + g.cells()
        g.set_checkpoint(ck)                          # sorted by the step
        g.step(1)
        for x, y in zip(g.get_state()[:3] + g.cells(), on):
            assert np.array_equal(x, y)
        g.close()
