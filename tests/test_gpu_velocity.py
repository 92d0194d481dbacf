"""The velocity update inside the pair kernel against its own kernel (phases timed),
bit for bit: lanes per bead (32 and 16) and bricks of every block size, no bonds,
chains, beads with more bonds than the pair kernel takes, boxes cut by bricks, both
sides of the size up to which it is done, and several systems at once."""
import numpy as np
import pytest

from paper_1804_06205_gb300 import workloads as W

pytestmark = pytest.mark.gpu

#        box                 beads   chains threads
CASES = [((3.0, 3.0, 3.0), 1, 0, 0), ((9.3, 4.1, 3.2), None, 0, 0), ((10.0, 10.0, 10.0), None, 20, 0),
         ((15.5, 14.0, 15.0), None, 0, 0), ((15.5, 14.0, 15.0), None, 60, 0), ((17.3, 17.9, 18.0), None, 0, 0),
         ((17.3, 17.9, 18.0), None, 90, 64), ((17.3, 17.9, 18.0), None, 90, 256),
         ((37.0, 37.0, 39.0), 159999, 400, 0), ((37.0, 37.0, 39.0), 160001, 400, 0)]


def _bonds(chains, extra):
    """Chains of ten; extra: also their second and third neighbours."""
    i = (np.arange(chains)[:, None] * 10 + np.arange(7)[None, :]).ravel()
    i, j = (np.concatenate([i] * len(extra)), np.concatenate([i + d for d in extra]))
    m = i.size
    return dict(i=i.astype(np.int32), j=j.astype(np.int32), kind=np.full(m, 1, np.int32), r0=np.full(m, 0.4),
                k=np.full(m, 6.0), alpha=np.zeros(m))


def _run(make, timed):
    with make() as g:
        if timed:
            g.profile_begin(20)
        g.step(5)
        mid = g.get_state()[:3]
        g.step(1)
        g.step(4)
        return mid + g.get_state()[:3] + (np.frombuffer(g.get_checkpoint(), np.uint8),)


@pytest.mark.parametrize("extra", [(1,), (1, 2, 3)])
@pytest.mark.parametrize("k", range(len(CASES)))
def test_same_bits_as_its_own_kernel(k, extra):
    from paper_1804_06205_gb300 import dpd as D
    L, n, chains, threads = CASES[k]
    if not chains and extra != (1,):
        pytest.skip("no bonds")
    w = W.fluid(L, n=n, ntypes=2, a_cross=33.0, seed=30 + k)

    def make():
        g = D.System(w.L, w.types, w.a, w.gamma, w.kT, 0.01, seed=w.seed, lam=w.lam, threads=threads,
                     bonds=_bonds(chains, extra) if chains else None)
        g.set_state(w.pos, w.vel, 3)
        return g
    for x, y in zip(_run(make, False), _run(make, True)):
        assert np.array_equal(x, y)


def test_same_bits_in_a_batch():
    from paper_1804_06205_gb300 import dpd as D
    ws = [W.fluid(L, n=None, ntypes=2, a_cross=33.0, seed=k) for k, (L, *_) in enumerate(CASES[1:6])]
    out = []
    for timed in (False, True):
        b = D.Batch(sum(w.n for w in ws), sum(int(np.prod(np.floor(w.L))) for w in ws), 1)
        ids = [b.add_workload(w, step=k) for k, w in enumerate(ws)]
        if timed:
            b.profile_begin(20)
        b.step(3)
        b.step(2)
        out.append([x for i in ids for x in b.get_state(i)[:3]])
    for x, y in zip(*out):
        assert np.array_equal(x, y)
