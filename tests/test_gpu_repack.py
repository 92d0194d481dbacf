"""Observables of a system that a re-pack has moved in the pools, asked for before
the next step: a removal followed by an admission (or by one that is refused) moves
the survivors' beads and cells, and the sampled pair pass needs the cell starts of
the new place.  Compared bit for bit with the same system run alone, then stepped on."""
import numpy as np
import pytest

from paper_1804_06205_gb300 import workloads as W

pytestmark = pytest.mark.gpu

KEYS = ("kT", "p_total", "p_cons", "p_bond", "e_pair", "e_bond", "momentum")


def _same(a, b):
    for k in KEYS:
        assert np.array_equal(a[k], b[k]), k


@pytest.mark.parametrize("restored", [False, True])     # B's state comes by set_checkpoint
@pytest.mark.parametrize("refused", [False, True])      # the admission does not fit
@pytest.mark.parametrize("prec", [0, 1])
def test_observables_after_repack_before_a_step(prec, refused, restored):
    from paper_1804_06205_gb300 import dpd as D
    a = W.serving_system(1, edge=8.0, a_ab=27.0)
    b = W.serving_system(2, edge=9.7, a_ab=44.0)
    p = W.peptide_192k(L=9.0, nchains=8, chain_len=20, seed=31)
    c = W.serving_system(3, edge=12.0 if refused else 7.6, a_ab=33.0)
    ws = [a, b, p]
    bt = D.Batch(sum(w.n for w in ws), sum(int(np.prod(np.floor(w.L))) for w in ws),
                 sum(w.nbonds for w in ws), max_systems=4, precision=prec)
    ids = [bt.add_workload(w) for w in ws]
    bt.step(4)
    alone = []
    for w in (b, p):
        g = D.System.from_workload(w, precision=prec)
        g.set_state(w.pos, w.vel, 0)
        g.step(4)
        alone.append(g)
    if restored:
        for g, i in zip(alone, ids[1:]):
            bt.set_checkpoint(i, g.get_checkpoint())
    bt.remove(ids[0])                    # b and p move down by a's beads and cells
    late = bt.add_workload(c)
    assert (late is None) == refused
    for g, i in zip(alone, ids[1:]):
        _same(bt.observables(i), g.observables())
    bt.step(3)
    for g, i in zip(alone, ids[1:]):
        g.step(3)
        for x, y in zip(bt.get_state(i)[:3], g.get_state()[:3]):
            assert np.array_equal(x, y)
        _same(bt.observables(i), g.observables())
        g.close()
    bt.close()
