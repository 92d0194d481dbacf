"""Handles made, stepped and closed by several host threads at once: they share the
pair kernels' shared-memory limit, raised by the largest, and the FP64 tables, which
come and go with the handles.  Each run must have the bits of the same run alone."""
import threading

import numpy as np
import pytest

from paper_1804_06205_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def test_handles_from_several_threads():
    from paper_1804_06205_gb300 import dpd as D
    # different densities and so different brick sizes and shared memory
    ws = [W.fluid(10.0, n=3000, seed=91), W.fluid(9.3, n=4100, seed=92),
          W.fluid(7.1, n=2900, seed=93), W.fluid(8.0, n=6100, seed=94)]

    def run(w, k):
        g = D.System.from_workload(w, precision=D.DPD_FP64 if k % 3 else D.DPD_FP32)
        g.set_state(w.pos, w.vel, 0)
        g.step(35)
        out = g.get_state()[:3]
        g.close()
        return out

    got, errors = {}, []

    def work(t):
        try:
            for k in range(6):
                got[t, k] = run(ws[(t + k) % 4], k)
        except Exception as e:      # a thread's exception is the test's
            errors.append(e)

    threads = [threading.Thread(target=work, args=(t,)) for t in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for (t, k), out in got.items():
        for x, y in zip(out, run(ws[(t + k) % 4], k)):
            assert np.array_equal(x, y)
