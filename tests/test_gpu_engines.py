"""What the automatic choices of a batch lead to -- engine, query group, cut
partitions -- against the oracle: power-law graphs of few partitions and of
many, batch sizes around the lines of the group sizes, sizes that leave the
last partition of the cut ones ragged or empty, and graphs of different
partition sizes in use in turn."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_2103_14915_gb300 import fg, inputs

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def create(g, method=fg.FG_PART_AUTO, S=0):
    st, h = fg.fg_graph_create_ex(g.n, g.m, g.row_ptr, g.col, g.w, 0,
                                  fg.fg_default_graph_opts(partition_method=method, partition_vertices=S))
    fg.check(st)
    return h


def run(h, g, kind, srcs):
    s_d = torch.from_numpy(np.ascontiguousarray(srcs, dtype=np.int32)).to(DEV)
    out = torch.empty((len(srcs), g.n), dtype=torch.int32, device=DEV)
    f = fg.fg_sssp_batch if kind == "sssp" else fg.fg_bfs_batch
    fg.check(f(h, s_d, len(srcs), out, None, fg.fg_default_opts(watchdog_ms=20000)))
    fg.check(fg.fg_sync())
    return out.cpu().numpy().view(np.uint32), fg.fg_stats(h)[1].group


def cut_to(g, n):
    """The graph on the first n vertices."""
    u = np.repeat(np.arange(g.n), g.out_degree())
    keep = (u < n) & (g.col < n)
    rp = np.zeros(n + 1, np.int64)
    rp[1:] = np.cumsum(np.bincount(u[keep], minlength=n))
    return inputs.Graph(n, rp, np.ascontiguousarray(g.col[keep]), np.ascontiguousarray(g.w[keep]), g.directed)


@pytest.mark.parametrize("n", [1025, 2048, 4097, 16321, 16384])
@pytest.mark.parametrize("directed", [False, True])
def test_power_law(n, directed):
    g = cut_to(inputs.rmat((n - 1).bit_length(), 24, seed=31, directed=directed, weights=(1, 255)), n)
    assert g.out_degree().max() > 64
    srcs = np.concatenate([inputs.sources_uniform(g, 64, 6), [0, n - 1]])
    ref = {"sssp": oracle.sssp(g, srcs), "bfs": oracle.bfs(g, srcs)}
    h = create(g)
    try:
        for nq in (1, 9, 32, 33, 64, 66):
            for kind in ("sssp", "bfs"):
                got, group = run(h, g, kind, srcs[:nq])
                assert np.array_equal(got, ref[kind][:nq]), (kind, nq)
                assert group == (64 if nq > 64 else (8 if nq <= 32 else 16) if kind == "sssp" else
                                 next(G for G in (8, 16, 32, 64) if G >= nq))
    finally:
        fg.fg_graph_destroy(h)


def test_partition_sizes_in_turn():
    """A graph's launches keep working after another graph sized the same kernels for less shared memory."""
    g = inputs.rmat(12, 16, seed=33, weights=(1, 255))
    road = inputs.grid(60, 70, 500, 100, seed=3, weights=(100, 10000))
    srcs = inputs.sources_uniform(g, 40, 2)
    rsrc = inputs.sources_uniform(road, 40, 2)
    handles = [(create(x, fg.FG_PART_RANGE, S), x, s) for x, s in ((g, srcs), (road, rsrc)) for S in (4096, 32, 1024)]
    try:
        for _ in range(2):
            for h, x, s in handles:
                for kind in ("sssp", "bfs"):
                    ref = oracle.sssp(x, s) if kind == "sssp" else oracle.bfs(x, s)
                    assert np.array_equal(run(h, x, kind, s)[0], ref)
    finally:
        for h, _, _ in handles:
            fg.fg_graph_destroy(h)
