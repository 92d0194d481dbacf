"""The bonds/velocity kernel with and without the records dealt out to the block: a
system whose beads hold at most two records alone (not dealt on the FP32 path) and next
to one with a bead of many (dealt), and a system without bonds next to bonded ones, must
have the same bits, forces, observables and running means among them."""
import numpy as np
import pytest

from paper_1804_06205_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _hub(m=9):
    w = W.fluid((7.0, 6.0, 6.4), seed=71)
    d = w.pos - w.pos[5]
    near = np.argsort(np.linalg.norm(d - w.L * np.rint(d / w.L), axis=1))[1:m + 1]
    w.bonds = W.bond_records(np.full(m, 5), near, W.KIND_HARMONIC, 4.0, 0.3)
    return w


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("n", [1, 2])        # systems beside the hub's
def test_same_bits_dealt_and_not(prec, n):
    from paper_1804_06205_gb300 import dpd as D
    ws = [W.serving_system(5, edge=8.3, a_ab=31.0), W.fluid((6.0, 7.0, 8.2), seed=72)][:n]
    hub = _hub()
    b = D.Batch(8000, 4000, 4000, max_systems=4, precision=prec, threads=128)   # bricks
    ids = [b.add_workload(w) for w in ws + [hub]]
    for k in (1, 4):
        b.step(k)
    for w, i in zip(ws, ids):
        g = D.System.from_workload(w, precision=prec, threads=128)
        g.set_state(w.pos, w.vel, 0)
        for k in (1, 4):
            g.step(k)
        for x, y in zip(b.get_state(i)[:3], g.get_state()[:3]):
            assert np.array_equal(x, y)
        p, q = b.observables(i), g.observables()
        for k in ("e_bond", "p_bond", "e_pair", "kT"):
            assert p[k] == q[k], k
        s = D.System.from_workload(w, precision=prec, threads=128, sample_every=1)
        s.set_state(w.pos, w.vel, 0)
        s.step(5)
        assert s.observables()["e_bond"] == q["e_bond"]
        for x, y in zip(s.get_state()[:3], g.get_state()[:3]):
            assert np.array_equal(x, y)
        g.close()
        s.close()
    b.close()
