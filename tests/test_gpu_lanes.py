"""The pair kernel for few beads (lanes per bead) against the brick kernel
(threads set), bit for bit: boxes of three cells, odd and ragged ones, bricks cut
by the box, crowded cells (more hits and candidates than are queued or tested at
once), both sides of the bead counts where the lanes per bead change, both noises,
several types, and several systems in one launch."""
import numpy as np
import pytest

from paper_1804_06205_gb300 import workloads as W

pytestmark = pytest.mark.gpu

#        box                beads  types noise crowd
CASES = [((3.0, 3.0, 3.0), None, 1, 0, 0), ((3.9, 3.2, 4.7), 150, 3, 1, 0), ((12.3, 5.5, 3.1), None, 2, 0, 0),
         ((7.0, 9.0, 11.0), None, 2, 0, 400), ((5.0, 5.0, 5.0), 2000, 2, 1, 150), ((9.7, 30.1, 3.0), 40, 2, 0, 0),
         ((11.0, 11.0, 11.0), 4000, 2, 0, 0), ((11.0, 11.0, 11.0), 4001, 2, 0, 0),
         ((16.7, 16.7, 16.7), 14000, 2, 0, 60), ((16.7, 16.7, 16.7), 14001, 2, 0, 60),
         ((6.0, 6.0, 6.0), 1, 1, 0, 0), ((6.0, 6.0, 6.0), 2, 1, 0, 0)]


def _workload(k):
    L, n, nt, noise, crowd = CASES[k]
    w = W.fluid(L, n=n, ntypes=nt, a_cross=33.0, seed=60 + k)
    if crowd:
        rng = np.random.default_rng(k)
        w.pos[:crowd] = 1.0 + rng.uniform(0.0, 1.0, (crowd, 3))
        w.pos[crowd // 2] = w.pos[crowd // 2 - 1]          # a coincident pair
    return w, noise


@pytest.mark.parametrize("k", range(len(CASES)))
def test_same_bits_as_bricks(k):
    from paper_1804_06205_gb300 import dpd as D
    w, noise = _workload(k)
    dt = 0.04 if CASES[k][4] == 0 else 0.001
    out = []
    for threads in (0, 128):
        g = D.System(w.L, w.types, w.a, w.gamma, w.kT, dt, seed=w.seed, lam=w.lam, noise=noise, threads=threads)
        g.set_state(w.pos, w.vel, 5)
        f0 = g.get_state()[2]
        g.step(4)
        out.append((f0,) + g.get_state()[:3])
    for x, y in zip(*out):
        assert np.array_equal(x, y)


def test_same_bits_in_a_batch():
    from paper_1804_06205_gb300 import dpd as D
    ws = [_workload(k)[0] for k in (1, 2, 0, 5, 6)]
    out = []
    for threads in (0, 128):
        b = D.Batch(sum(w.n for w in ws), sum(int(np.prod(np.floor(w.L))) for w in ws), 1, threads=threads)
        ids = [b.add_workload(w, step=k) for k, w in enumerate(ws)]
        b.step(3)
        out.append([x for i in ids for x in b.get_state(i)[:3]])
    for x, y in zip(*out):
        assert np.array_equal(x, y)
