"""Bond records dealt out to a block's threads: beads with more records than a
block has threads, blocks with none, one, or more than one round of records,
and a last block that is not full, against the oracle and against the
persistent kernel (each bead walking its own records: the same bits)."""
import numpy as np
import pytest

import oracle as O
from paper_1804_06205_gb300 import workloads as W

pytestmark = pytest.mark.gpu

HUBS = [(0,), (1,), (255,), (257,), (700, 3, 300)]


def _star(hubs, seed):
    """Hub k has hubs[k] bond records, kinds in turn, with beads nearer than 2
    (the FP32 path takes a bond's nearest image from its cells, so a bond has to be
    shorter than half the box by a cell)."""
    w = W.fluid((7.0, 6.0, 6.4), seed=seed)
    rng = np.random.default_rng(seed)
    parts = []
    for h, m in enumerate(hubs):
        d = w.pos - w.pos[h]
        near = np.flatnonzero(np.linalg.norm(d - w.L * np.rint(d / w.L), axis=1) < 2.0)
        j = rng.choice(near[near >= 10], m)
        for q, kind in enumerate((W.KIND_HARMONIC, W.KIND_MORSE_PAPER, W.KIND_MORSE)):
            jj = j[q::3]
            parts.append(W.bond_records(np.full(jj.size, h), jj, kind, 0.4, 0.5, 0.8))
    w.bonds = W.concat_bonds(parts)
    return w


@pytest.mark.parametrize("hubs", HUBS)
def test_star_forces(hubs):
    from paper_1804_06205_gb300 import dpd as D
    w = _star(hubs, 7)
    s = O.System(w.L, w.types, w.a, w.gamma, w.kT, w.dt, w.lam, seed=w.seed, bonds=w.bonds)
    fo, _ = O.forces(s, w.pos, w.vel, 0)
    st = O.State(s, w.pos, w.vel, 0)
    st.run(2)
    for prec, tol in ((D.DPD_FP32, 1e-4), (D.DPD_FP64, 1e-10)):
        end = []
        for persistent in (0, 1):
            g = D.System.from_workload(w, precision=prec, persistent=persistent)
            g.set_state(w.pos, w.vel, 0)
            f0 = g.get_state()[2]
            assert np.abs(f0 - fo).max() <= tol * np.abs(fo).max()
            g.step(2)
            end.append(g.get_state())
            e = g.observables()["e_bond"]
            assert abs(e - st.observables()["e_bond"]) <= 10 * tol * max(1.0, abs(e))
        assert np.abs(end[0][2] - st.f).max() <= 2 * tol * np.abs(st.f).max()
        for x, y in zip(end[0][:3], end[1][:3]):
            assert np.array_equal(x, y)
