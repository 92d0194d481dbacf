"""FP64 systems on both sides of the size from which the Box-Muller factors are
looked up: the same system must follow the same bits alone (computed, below the
size) and in a batch whose capacity is above it (looked up), for both noises; and
the four-blocks-per-SM variant (many bricks) the same as the persistent kernel."""
import numpy as np
import pytest

from paper_1804_06205_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("noise", [0, 1])
def test_lookup_equals_arithmetic(noise):
    from paper_1804_06205_gb300 import dpd as D
    w = W.fluid((8.0, 8.0, 9.0), ntypes=2, a_cross=30.0, seed=81)
    assert w.n < 2000
    g = D.System.from_workload(w, precision=D.DPD_FP64, noise=noise)
    g.set_state(w.pos, w.vel, 0)
    g.step(4)
    b = D.Batch(50_000, 50_000, 1, precision=D.DPD_FP64, noise=noise)
    i = b.add_workload(w)
    b.step(4)
    for x, y in zip(g.get_state()[:3], b.get_state(i)[:3]):
        assert np.array_equal(x, y)


def test_dense_variant():
    from paper_1804_06205_gb300 import dpd as D
    w = W.fluid(49.0, ntypes=2, a_cross=30.0, seed=82)      # 4,375 bricks of 7 x 2 x 2 cells
    out = []
    for kw in (dict(), dict(persistent=1)):
        g = D.System.from_workload(w, precision=D.DPD_FP64, **kw)
        g.set_state(w.pos, w.vel, 0)
        g.step(2)
        out.append(g.get_state()[:3])
    for x, y in zip(*out):
        assert np.array_equal(x, y)
