"""The automatic group on graphs of few partitions: a window or a delta sends
SSSP on a road map with a lone hub to one query per warp, whose options they
are; other batches there, and graphs whose arcs are at hubs, go to groups."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_2103_14915_gb300 import fg, inputs

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
WINDOW = dict(sched=fg.FG_SCHED_PRIORITY, sched_window=25000)


def road_with_a_hub():
    g = inputs.grid(100, 90, seed=3, weights=(100, 10000))
    r = np.random.RandomState(1)
    u = np.repeat(np.arange(g.n), g.out_degree())
    x, w = r.choice(np.arange(1, g.n), 100, False), r.randint(100, 10001, 100)
    u, v, w = np.r_[u, np.zeros(100, int), x], np.r_[g.col, x, np.zeros(100, int)], np.r_[g.w, w, w]
    order = np.argsort(u, kind="stable")
    rp = np.zeros(g.n + 1, np.int64)
    rp[1:] = np.cumsum(np.bincount(u, minlength=g.n))
    return inputs.Graph(g.n, rp, v[order].astype(np.int32), w[order].astype(np.int32), True)


@pytest.mark.parametrize("graph", ["road", "rmat"])
def test_choice(graph):
    g = road_with_a_hub() if graph == "road" else inputs.rmat(12, 16, seed=5, weights=(1, 255))
    srcs = inputs.sources_uniform(g, 40, 2).astype(np.int32)
    sssp, bfs = oracle.sssp(g, srcs), oracle.bfs(g, srcs)
    st, h = fg.fg_graph_create(g.n, g.m, g.row_ptr, g.col, g.w, 0)
    fg.check(st)
    s_d = torch.from_numpy(srcs).to(DEV)
    out = torch.empty((len(srcs), g.n), dtype=torch.int32, device=DEV)
    try:
        for call, ref, opts, alone in ((fg.fg_sssp_batch, sssp, {}, False), (fg.fg_sssp_batch, sssp, WINDOW, True),
                                       (fg.fg_sssp_batch, sssp, dict(delta=20000), True),
                                       (fg.fg_bfs_batch, bfs, dict(sched=fg.FG_SCHED_PRIORITY, sched_window=24), False)):
            fg.check(call(h, s_d, len(srcs), out, None, fg.fg_default_opts(watchdog_ms=20000, **opts)))
            fg.check(fg.fg_sync())
            assert np.array_equal(out.cpu().numpy().view(np.uint32), ref), opts
            st, stats = fg.fg_stats(h)
            fg.check(st)
            assert (stats.group == 1) == (alone and graph == "road"), (opts, stats.group)
    finally:
        fg.fg_graph_destroy(h)
