"""The observables' reductions by four, two and one block per chunk of 4,096 beads: the
numbers of chunks on both sides of the first switches (4 to 2 above 38, 2 to 1 above 76,
1 to 2 above 152), kinetic sums against plain
sums of the state read back, pair and bond sums against the oracle's."""
import numpy as np
import pytest

import oracle as O
from paper_1804_06205_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,tol", [(0, 1e-5), (1, 1e-11)])
@pytest.mark.parametrize("chunks", [38, 39, 76, 77, 152, 153])
def test_sums_at_the_switches(chunks, prec, tol):
    from paper_1804_06205_gb300 import dpd as D
    n = 4096 * (chunks - 1) + 1 + chunks % 2
    edge = (n / 3.0) ** (1.0 / 3.0)
    w = W.fluid(edge, n=n, ntypes=2, a_cross=30.0, seed=chunks)
    i = np.arange(0, n - 1, 7)
    near = np.linalg.norm(w.pos[i] - w.pos[i + 1], axis=1) < 3.0
    w.bonds = W.bond_records(i[near], i[near] + 1, W.KIND_HARMONIC, 0.5, 4.0)
    g = D.System.from_workload(w, precision=prec)
    g.set_state(w.pos, w.vel, 0)
    _, v, _, _ = g.get_state()
    o = g.observables()
    g.close()
    # n additions of numbers of order one, each rounded to 2^-53
    assert np.all(np.abs(np.asarray(o["momentum"]) - v.sum(axis=0)) <= 16 * n * 2.0 ** -53)
    assert abs(o["sum_v2"] - float((v * v).sum())) <= 64 * n * 2.0 ** -53
    s = O.System(w.L, w.types, w.a, w.gamma, w.kT, w.dt, w.lam, seed=w.seed, bonds=w.bonds)
    r = O.State(s, w.pos, w.vel, 0, mode=O.MODE_CELLS).observables()
    for k in ("e_pair", "p_cons", "e_bond", "p_bond"):
        assert abs(o[k] - r[k]) <= tol * max(abs(r[k]), 1e-3), k
