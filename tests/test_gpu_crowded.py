"""Crowded cells in the gather by cell (systems of at least 65,536 beads in id order:
set_state, a restored checkpoint): cells at the limit up to which eight threads rank a
cell's beads (64), one more, and one of thousands, whose beads are ranked a thread per
bead.  Cells are compared with the oracle's and a run resumed by a checkpoint with the
same run gone on with, bit for bit.  Refused states, whose non-finite beads belong in
no cell, cost no more than others."""
import numpy as np
import pytest

import oracle as O
from paper_1804_06205_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,n,big", [((45.0, 44.2, 45.0), 262_145, 2_000),
                                     ((45.0, 44.2, 45.0), 262_144, 0),     # 0: no cell is left over
                                     ((28.0, 28.7, 28.2), 65_536, 1_000),
                                     ((28.0, 28.7, 28.2), 65_535, 1_000)])  # by bead
def test_crowded_cells_by_cell(L, n, big):
    from paper_1804_06205_gb300 import dpd as D
    w = W.fluid(L, n=n, seed=61)
    rng = np.random.default_rng(62)
    h = w.L / np.floor(w.L)
    crowds = (9, 16, 17, 40, 50) + ((64, 65, 66, 300, big) if big else ())
    at = 0
    for k, beads in enumerate(crowds):
        cell = np.array([2 + 2 * k, 5, 44])          # apart from one another
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


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
def test_refused_state_costs_what_a_state_costs(prec, value):
    """Non-finite positions have no cell.  All in one cell, the pair pass before the
    refusal would test every pair of them, in one block: a thousand times what a
    state of this size takes (and its square at a million beads)."""
    import time
    from paper_1804_06205_gb300 import dpd as D
    w = W.fluid(18.8, n=20_000, seed=63)
    bad = np.full_like(w.pos, value)
    g = D.System.from_workload(w, precision=prec)
    best = []
    for pos in (w.pos, bad):
        best.append(np.inf)
        for _ in range(3):
            t = time.perf_counter()
            if pos is bad:
                with pytest.raises(D.DPDError) as e:
                    g.set_state(pos, w.vel, 0)
                assert e.value.code == D.DPD_EINVAL
                with pytest.raises(D.DPDError):
                    g.get_state()                     # no state to read
            else:
                g.set_state(pos, w.vel, 0)
            best[-1] = min(best[-1], time.perf_counter() - t)
    assert best[1] < 20 * best[0], best
    g.set_state(w.pos, w.vel, 0)                      # the handle stays usable
    g.step(3)
    ref = D.System.from_workload(w, precision=prec)
    ref.set_state(w.pos, w.vel, 0)
    ref.step(3)
    for x, y in zip(g.get_state()[:3], ref.get_state()[:3]):
        assert np.array_equal(x, y)
    g.close()
    ref.close()


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("where", ["pos", "vel"])
def test_refused_state_leaves_no_error(prec, where):
    """A non-finite value of one bead, in a system with bonds: refused, and the handle
    takes the next state."""
    from paper_1804_06205_gb300 import dpd as D
    w = W.serving_system(4, edge=8.0, a_ab=30.0)
    g = D.System.from_workload(w, precision=prec)
    bonded = int(w.bonds["i"][0])
    for value in (np.nan, np.inf):
        pos, vel = w.pos.copy(), w.vel.copy()
        (pos if where == "pos" else vel)[bonded, 1] = value
        with pytest.raises(D.DPDError) as e:
            g.set_state(pos, vel, 0)
        assert e.value.code == D.DPD_EINVAL
        g.set_state(w.pos, w.vel, 0)
        g.step(2)
        assert np.isfinite(g.get_state()[0]).all()
    g.close()
