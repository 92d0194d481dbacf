"""The cell division's rows of ids, lists behind them and scans, at their edges:
cells of 0 to 8, 9 and hundreds of beads, boxes of one and of several scan tiles
on both sides of the one-launch scan's limit (8 tiles of 2,048 cells), and a box
so empty that its cells keep lists only.  Cells are compared with the oracle's
(bit-exact), and steps with the persistent kernel (the same bits)."""
import numpy as np
import pytest

import oracle as O
from paper_1804_06205_gb300 import workloads as W

pytestmark = pytest.mark.gpu

#        box                 beads   crowded cells: (count, beads each)
SYSTEMS = [((5.0, 4.0, 3.0), 700, ()),
           ((12.7, 12.9, 12.2), None, ((1, 400), (6, 9), (5, 8))),     # 1,728 cells, one tile
           ((26.0, 25.3, 25.0), 30_000, ((3, 33),)),                   # 16,250 cells, 8 tiles
           ((26.0, 25.3, 26.0), 30_000, ((3, 33),)),                   # 16,900 cells, 9 tiles
           ((20.0, 20.0, 20.0), 1_500, ((2, 40),)),                    # 5.3 cells per bead
           ((45.0, 44.2, 45.0), 262_144, ((2, 30), (30, 9)))]          # restored by cell


@pytest.mark.parametrize("k", range(len(SYSTEMS)))
def test_cells_and_steps(k):
    from paper_1804_06205_gb300 import dpd as D
    L, n, crowd = SYSTEMS[k]
    w = W.fluid(L, n=n, seed=40 + k)
    rng = np.random.default_rng(50 + k)
    h = w.L / np.floor(w.L)
    at = 0
    for count, beads in crowd:
        for _ in range(count):
            cell = rng.integers(0, np.floor(w.L).astype(int))
            w.pos[at:at + beads] = (cell + rng.uniform(0.02, 0.98, (beads, 3))) * h
            at += beads
    perm = rng.permutation(w.n)          # the crowd's ids everywhere
    w.pos = w.pos[perm]
    s = O.System(w.L, w.types, w.a, w.gamma, w.kT, w.dt, w.lam)
    key = O.cell_keys(s, O.wrap(s, w.pos))
    order, start = O.cell_sort(s, key)
    for prec in (D.DPD_FP32, D.DPD_FP64):
        end = []
        for persistent in (0, 1):
            g = D.System.from_workload(w, precision=prec, persistent=persistent)
            g.set_state(w.pos, w.vel * 0.1, 0)
            gk, go, gs = g.cells()
            assert np.array_equal(gk, key) and np.array_equal(go, order) and np.array_equal(gs, start)
            g.step(3)
            end.append(g.get_state()[:3] + g.cells())
            # a restored state comes in id order: the same steps from it
            ck = g.get_checkpoint()
            g.step(2)
            end[-1] += g.get_state()[:3]
            g.set_checkpoint(ck)
            g.step(2)
            for x, y in zip(g.get_state()[:3], end[-1][-3:]):
                assert np.array_equal(x, y)
        for x, y in zip(*end):
            assert np.array_equal(x, y)
