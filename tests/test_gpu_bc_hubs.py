"""BC where one hub is in a warp once per query: its arcs are taken a bounded
number at a time, so degrees around that number and its multiples, parallel
arcs included, must give the oracle's sums bit for bit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_2103_14915_gb300 import fg, inputs

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
PASS = 1 << 16  # arcs of a vertex at a time
LEAVES = 33     # vertices with an arc to the hub: the sources


@pytest.mark.parametrize("deg", [PASS - 1, PASS, PASS + 1, 2 * PASS, 2 * PASS + 31])
def test_a_hub_under_many_queries(deg):
    r = np.random.RandomState(deg)
    mid = 500
    hub, n = LEAVES + mid, LEAVES + mid + 2
    u = np.concatenate([np.arange(LEAVES), np.full(deg, hub), np.arange(LEAVES, LEAVES + mid)])
    v = np.concatenate([np.full(LEAVES, hub), r.randint(LEAVES, LEAVES + mid, deg), np.full(mid, n - 1)])
    order = np.argsort(u, kind="stable")
    rp = np.zeros(n + 1, np.int64)
    rp[1:] = np.cumsum(np.bincount(u, minlength=n))
    g = inputs.Graph(n, rp, v[order].astype(np.int32), None, True)
    srcs = np.concatenate([np.arange(LEAVES), [hub]]).astype(np.int32)
    ref, most, exact = oracle.bc(g, srcs, False)
    assert exact
    st, h = fg.fg_graph_create(g.n, g.m, g.row_ptr, g.col, None, 0)
    fg.check(st)
    try:
        s_d = torch.from_numpy(srcs).to(DEV)
        dist = torch.empty((len(srcs), n), dtype=torch.int32, device=DEV)
        bc = torch.empty(n, dtype=torch.float64, device=DEV)
        fg.check(fg.fg_bfs_batch(h, s_d, len(srcs), dist))
        fg.check(fg.fg_sync())
        st, info = fg.fg_bc_accumulate(h, s_d, len(srcs), dist, False, bc)
        fg.check(st)
        assert info.sigma_max == most and info.waves == 4
        assert np.array_equal(bc.cpu().numpy(), ref)
    finally:
        fg.fg_graph_destroy(h)
