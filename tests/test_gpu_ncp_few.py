"""Sweep cuts of few rows and a small top, whose rows are streamed in parts and
merged by one block each, around the lines of that route, against the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_2103_14915_gb300 import fg
from test_gpu_ncp_paths import DEV, graph, rows

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,nq,top", [(16385, 1, 256), (16388, 3, 257), (24577, 85, 20), (24577, 86, 20), (65540, 31, 64),
                                      (65540, 32, 64), (131072, 2, 256), (131073, 2, 256), (262144, 2, 128),
                                      (262144, 2, 129), (262145, 1, 5)])
@pytest.mark.parametrize("kind", ["sparse", "ties", "clustered"])
def test_same_sweep(n, nq, top, kind):
    g = graph(n)
    p = rows(n, kind, nq)
    ref = oracle.ncp_sweep(g, p, top)
    best = np.where(np.isnan(ref[1]), np.inf, ref[1]).min(0)
    st, h = fg.fg_graph_create(g.n, g.m, g.row_ptr, g.col, None, 0)
    fg.check(st)
    try:
        p_d = torch.from_numpy(p).to(DEV)
        order = torch.empty((nq, top), dtype=torch.int32, device=DEV)
        phi = torch.empty((nq, top), dtype=torch.float64, device=DEV)
        count = torch.empty(nq, dtype=torch.int32, device=DEV)
        ncp = torch.full((top,), 0.4, dtype=torch.float64, device=DEV)
        for again in (False, True):
            fg.check(fg.fg_ncp_sweep(h, p_d, nq, top, order, phi, count, ncp, again))
            fg.check(fg.fg_sync())
            assert np.array_equal(count.cpu().numpy(), ref[2])
            assert np.array_equal(order.cpu().numpy(), ref[0])
            assert np.array_equal(phi.cpu().numpy(), ref[1], equal_nan=True)
            assert np.array_equal(ncp.cpu().numpy(), best)
            ncp.copy_(torch.from_numpy(np.maximum(best, 0.5)))  # the second call lowers it again
    finally:
        fg.fg_graph_destroy(h)
