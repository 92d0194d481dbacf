"""The 80 MB of Box-Muller tables are made only for FP64 handles that read them often
enough: not for uniform noise, few beads or few steps; handles share them, and they go
with the last.  Checked by the device's free memory, in a process of its own so that no
other handle has them; a handle's creation takes the memory that the header states.
And a run that starts without them and goes on with them has the
bits of one that never has them."""
import subprocess
import sys

import pytest

from paper_1804_06205_gb300 import workloads as W

pytestmark = pytest.mark.gpu

PROGRAM = """
import torch
from paper_1804_06205_gb300 import dpd as D, workloads as W
w, small = W.fluid(10.0, n=3000, seed=1), W.fluid(7.0, n=900, seed=2)
MB = 1 << 20
free = lambda: torch.cuda.mem_get_info(0)[0] / MB

def system(w, **kw):
    g = D.System.from_workload(w, precision=D.DPD_FP64, **kw)
    g.set_state(w.pos, w.vel, 0)
    return g

g = system(small)                                   # context and kernels are loaded
g.step(2); g.close()
base = free()
def taken(g):
    g.sync()
    return base - free()
a = system(w, noise=D.DPD_NOISE_UNIFORM)
a.step(200)
assert taken(a) < 40, taken(a)
s = system(small)
s.step(200)
assert taken(s) < 40, taken(s)
b = D.Batch(6000, 2000, 1, precision=D.DPD_FP64)
assert b.add_workload(w) is not None
b.step(5)
assert taken(b) < 40, taken(b)
b.step(60)
assert 80 < taken(b) < 120, taken(b)
c = system(w)
c.step(1)
assert taken(c) < 120, taken(c)                     # shared
b.close()
assert taken(c) > 80, taken(c)
c.close()
assert taken(a) < 40, taken(a)
print("ok")
"""


CREATED = """
import torch
from paper_1804_06205_gb300 import dpd as D, workloads as W
free = lambda: torch.cuda.mem_get_info(0)[0]
small, w = W.fluid(7.0, n=900, seed=2), W.fluid(70.0, n=1 << 20, seed=3)
for prec, per_bead in ((D.DPD_FP32, 152), (D.DPD_FP64, 264)):
    g = D.System.from_workload(small, precision=prec)       # context and kernels are loaded
    g.set_state(small.pos, small.vel, 0); g.step(2); g.close()
    base = free()
    g = D.System.from_workload(w, precision=prec)
    taken, said = base - free(), per_bead * w.n + 48 * 70 ** 3
    assert 0.97 * said < taken < 1.08 * said, (prec, taken / 2 ** 20, said / 2 ** 20)   # 2 MB pages
    g.close()
print("ok")
"""


@pytest.mark.parametrize("program", [PROGRAM, CREATED], ids=["tables", "created"])
def test_device_memory(program):
    pytest.importorskip("torch")
    r = subprocess.run([sys.executable, "-c", program], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout + r.stderr


@pytest.mark.parametrize("mode", [dict(), dict(use_graph=1), dict(persistent=1)])
def test_same_bits_when_the_tables_come_in(mode):
    import numpy as np
    from paper_1804_06205_gb300 import dpd as D
    w = W.fluid((8.0, 8.0, 9.0), ntypes=2, a_cross=30.0, seed=81)
    assert w.n < 2000
    g = D.System.from_workload(w, precision=D.DPD_FP64)      # never looked up
    g.set_state(w.pos, w.vel, 0)
    b = D.Batch(50_000, 50_000, 1, precision=D.DPD_FP64, **mode)
    i = b.add_workload(w)
    for k in (3, 10, 25, 2, 30):                             # from the third call on, at the latest
        g.step(k)
        b.step(k)
        for x, y in zip(g.get_state()[:3], b.get_state(i)[:3]):
            assert np.array_equal(x, y)
    g.close()
    b.close()
