"""dpd_cells_noalloc recorded by a stream capture (its kernels after the first become
programmatic edges) and replayed on other positions in the same buffers: cells as the
oracle's each time."""
import numpy as np
import pytest

import oracle as O
from paper_1804_06205_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,n", [((11.3, 9.0, 14.7), 4500), ((40.0, 41.5, 39.0), 200_003)])
def test_capture_and_replay(L, n):
    torch = pytest.importorskip("torch")
    from paper_1804_06205_gb300 import dpd as D
    w = W.fluid(L, n=n, seed=95)
    s = O.System(w.L, w.types, w.a, w.gamma, w.kT, w.dt, w.lam)
    ncell = int(np.prod(np.floor(w.L)))
    pos = torch.tensor(w.pos, dtype=torch.float64, device="cuda:0")
    key, order, start = (torch.zeros(k, dtype=torch.int32, device="cuda:0") for k in (n, n, ncell + 1))

    def call(stream):
        return D.cells_noalloc(pos.data_ptr(), n, w.L, key.data_ptr(), order.data_ptr(),
                               start.data_ptr(), stream.cuda_stream)

    assert call(torch.cuda.current_stream()) == D.DPD_OK      # looks the scratch up
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        assert call(torch.cuda.current_stream()) == D.DPD_OK
    rng = np.random.default_rng(96)
    for _ in range(3):
        p = rng.uniform(-0.5, 1.5, (n, 3)) * w.L
        pos.copy_(torch.tensor(p))
        key.fill_(-1), order.fill_(-1), start.fill_(-1)
        graph.replay()
        torch.cuda.synchronize()
        okey = O.cell_keys(s, O.wrap(s, p))
        oorder, ostart = O.cell_sort(s, okey)
        assert np.array_equal(key.cpu().numpy().view(np.uint32), okey)
        assert np.array_equal(order.cpu().numpy(), oorder)
        assert np.array_equal(start.cpu().numpy().view(np.uint32), ostart)
