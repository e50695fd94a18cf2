"""The automatic group on graphs of few partitions: a window or a delta sends
SSSP on a road map with a lone hub to one query per warp, whose options they
are; other batches there, and graphs whose arcs are at hubs, go to groups. A
graph of one partition goes to one query per warp where neither the reduced
graph nor BFS's masks speak for groups."""
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


@pytest.mark.parametrize("n,edges,groups", [(200, 1200, (False, False)), (1000, 9000, (False, True)),
                                            (1000, 40000, (True, True))])
def test_one_partition(n, edges, groups):
    """groups: of SSSP, BFS; the densest graph has a reduced one."""
    r = np.random.RandomState(n)
    u, v = (n * r.rand(edges) ** 3).astype(np.int64), r.randint(0, n, edges)
    u, v, w = np.r_[u, v], np.r_[v, u], np.tile(r.randint(1, 256, edges), 2)
    order = np.argsort(u, kind="stable")
    rp = np.zeros(n + 1, np.int64)
    rp[1:] = np.cumsum(np.bincount(u, minlength=n))
    g = inputs.Graph(n, rp, v[order].astype(np.int32), w[order].astype(np.int32), True)
    assert g.out_degree().max() > 64
    srcs = np.resize(np.arange(n), 300).astype(np.int32)
    st, h = fg.fg_graph_create(g.n, g.m, g.row_ptr, g.col, g.w, 0)
    fg.check(st)
    s_d = torch.from_numpy(srcs).to(DEV)
    out = torch.empty((len(srcs), g.n), dtype=torch.int32, device=DEV)
    try:
        for call, ref, grouped in ((fg.fg_sssp_batch, oracle.sssp(g, srcs), groups[0]),
                                   (fg.fg_bfs_batch, oracle.bfs(g, srcs), groups[1])):
            fg.check(call(h, s_d, len(srcs), out))
            fg.check(fg.fg_sync())
            assert np.array_equal(out.cpu().numpy().view(np.uint32), ref)
            st, stats = fg.fg_stats(h)
            fg.check(st)
            assert (stats.group > 1) == grouped
    finally:
        fg.fg_graph_destroy(h)
