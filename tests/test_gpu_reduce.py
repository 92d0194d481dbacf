"""The reductions, two sums of a chunk per block: momentum and the sum of v^2 at the edges
of warps, blocks and chunks, against plain sums in 64 bits of the state read back."""
import numpy as np
import pytest

from paper_1804_06205_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 31, 33, 255, 256, 257, 4095, 4096, 4097, 8193, 156000])
def test_sums_against_the_state(n):
    from paper_1804_06205_gb300 import dpd as D
    edge = max(3.0, round((n / 3.0) ** (1.0 / 3.0), 3))
    w = W.fluid((edge, edge, edge), n=n, ntypes=1, seed=n % 97)
    with D.System(w.L, w.types, w.a, w.gamma, w.kT, 0.02, seed=w.seed, lam=w.lam) as g:
        g.set_state(w.pos, w.vel, 0)
        g.step(2)
        _, v, _, _ = g.get_state()
        o = g.observables()
        # n additions and products of numbers of order one, each rounded to 2^-53
        tol = n * 2.0 ** -53 * 16
        assert np.all(np.abs(np.asarray(o["momentum"]) - v.sum(axis=0)) <= tol)
        assert abs(o["sum_v2"] - float((v * v).sum())) <= 4 * tol
