"""SSSP on a graph without the arcs that lie on no shortest path (built at graph
creation for power-law graphs) against the oracle and against one query per
warp, which runs on the whole graph: directed and undirected, relabelled,
zero and equal weights, parallel arcs and loops, sizes around the words of
the arc marks, and overflows on arcs that were left out."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_2103_14915_gb300 import fg, inputs

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def build(g, method=fg.FG_PART_AUTO, S=0):
    """(handle, whether arcs were left out)"""
    st, h = fg.fg_graph_create_ex(g.n, g.m, g.row_ptr, g.col, g.w, 0,
                                  fg.fg_default_graph_opts(partition_method=method, partition_vertices=S))
    fg.check(st)
    st, info = fg.fg_graph_info(h)
    fg.check(st)
    whole = 4 * (g.n + 1 + 2 * g.m) + (0 if info.partition_method == fg.FG_PART_RANGE else 8 * g.n)
    return h, info.device_bytes > whole


def rows(h, g, srcs, **opts):
    s_d = torch.from_numpy(np.ascontiguousarray(srcs, dtype=np.int32)).to(DEV)
    out = torch.empty((len(srcs), g.n), dtype=torch.int32, device=DEV)
    fg.check(fg.fg_sssp_batch(h, s_d, len(srcs), out, None, fg.fg_default_opts(watchdog_ms=20000, **opts)))
    st = fg.fg_sync()
    return st, out.cpu().numpy().view(np.uint32)


def from_arcs(n, u, v, w):
    """A directed multigraph: loops and parallel arcs stay."""
    order = np.argsort(u, kind="stable")
    rp = np.zeros(n + 1, np.int64)
    rp[1:] = np.cumsum(np.bincount(u, minlength=n))
    return inputs.Graph(n, rp, v[order].astype(np.int32), w[order].astype(np.int32), True)


def multigraph(m, lo, hi):
    """m arcs with skewed ends, loops and repeats among them."""
    r = np.random.RandomState(m + hi)
    n = 3001
    u, v = ((n * r.rand(m) ** 3).astype(np.int64) * 7 % n for _ in range(2))
    return from_arcs(n, u, v, r.randint(lo, hi + 1, m))


CASES = {
    "undirected": (lambda: inputs.rmat(13, 16, seed=3, weights=(1, 255)), True),
    "directed": (lambda: inputs.rmat(13, 16, seed=4, directed=True, weights=(1, 255)), True),
    "wide": (lambda: inputs.rmat(12, 24, seed=5, weights=(1, 1 << 20)), True),
    "zero": (lambda: multigraph(70001, 0, 9), True),
    "last_word_full": (lambda: multigraph(65536, 1, 100), True),
    "last_word_of_one": (lambda: multigraph(65537, 1, 100), True),
    "too_few_arcs": (lambda: multigraph(32767, 1, 100), False),
    "no_arc_can_be_beaten": (lambda: inputs.rmat(12, 16, seed=6, weights=(128, 256)), False),
}


@pytest.mark.parametrize("name", CASES)
def test_rows_are_exact(name):
    make, left_out = CASES[name]
    g = make()
    srcs = np.concatenate([inputs.sources_uniform(g, 66, 2), [int(np.argmax(g.out_degree()))]])
    ref = oracle.sssp(g, srcs)
    h, reduced = build(g, fg.FG_PART_RANGE)  # AUTO may grow partitions that keep most arcs inside
    try:
        assert reduced == left_out
        for G in (8, 16, 32, 64):
            st, got = rows(h, g, srcs, group=G)
            assert st == fg.FG_OK and np.array_equal(got, ref), G
        st, got = rows(h, g, srcs, group=32, sched=fg.FG_SCHED_PRIORITY, sched_window=64)
        assert st == fg.FG_OK and np.array_equal(got, ref)
        st, got = rows(h, g, srcs, group=1)
        assert st == fg.FG_OK and np.array_equal(got, ref)
    finally:
        fg.fg_graph_destroy(h)


@pytest.mark.parametrize("method,S", [(fg.FG_PART_RANGE, 32), (fg.FG_PART_DEGREE, 64)])
def test_partitioners(method, S):
    g = inputs.rmat(13, 16, seed=8, weights=(1, 255))
    srcs = inputs.sources_uniform(g, 20, 3)
    h, reduced = build(g, method, S)
    try:
        assert reduced
        st, got = rows(h, g, srcs)
        assert st == fg.FG_OK and np.array_equal(got, oracle.sssp(g, srcs))
    finally:
        fg.fg_graph_destroy(h)


def test_overflow_on_an_arc_that_was_left_out():
    """A far source sees the whole graph near 2^32 - 1. Where only arcs that lie
    on no shortest path pass the limit, the call reports it as it does with
    every arc in, and the distances are the same."""
    g0 = inputs.rmat(12, 16, seed=9, weights=(1, 255))
    hub = int(np.argmax(g0.out_degree()))
    d0 = oracle.sssp(g0, [hub])[0]
    ecc = int(d0[d0 != 0xFFFFFFFF].max())
    u = np.repeat(np.arange(g0.n), g0.out_degree())
    reached = d0[u] != 0xFFFFFFFF
    over = int((d0[u].astype(np.int64) + g0.w)[reached].max())  # the longest sum any arc makes
    assert over > ecc + 1
    no_walk = 255 * (g0.n + 1)  # a value on the way is a sum over fewer than n arcs
    for room, status in ((ecc + 1, fg.FG_ERR_OVERFLOW), (over, fg.FG_ERR_OVERFLOW), (no_walk, fg.FG_OK)):
        # source -> middle -> hub of total 2^32 - 1 - room
        far = 2**32 - 1 - room
        n, m1 = g0.n + 2, 2**31 - 1
        g = from_arcs(n, np.concatenate([u, [g0.n, g0.n + 1]]), np.concatenate([g0.col, [g0.n + 1, hub]]),
                      np.concatenate([g0.w, [m1, far - m1]]))
        h, reduced = build(g, fg.FG_PART_RANGE)
        try:
            assert reduced
            want = d0.astype(np.int64) + far
            want[d0 == 0xFFFFFFFF] = 0xFFFFFFFF
            for G in (1, 8, 64):
                st, got = rows(h, g, [g0.n], group=G)
                assert st == status, (room, G)
                assert np.array_equal(got[0, :g0.n].astype(np.int64), want), (room, G)
        finally:
            fg.fg_graph_destroy(h)


@pytest.mark.parametrize("weights,directed", [((1, 8), False), ((1, 255), True)])
def test_dependencies_are_the_same(weights, directed):
    """BC runs on the graph that SSSP runs on: the same tight arcs in the same
    order. Small weights tie many paths."""
    g = inputs.rmat(13, 16, seed=11, directed=directed, weights=weights)
    srcs = np.concatenate([inputs.sources_uniform(g, 6, 5), [int(np.argmax(g.out_degree()))]]).astype(np.int32)
    h, reduced = build(g, fg.FG_PART_RANGE)
    try:
        assert reduced
        s_d = torch.from_numpy(srcs).to(DEV)
        dist = torch.empty((len(srcs), g.n), dtype=torch.int32, device=DEV)
        fg.check(fg.fg_sssp_batch(h, s_d, len(srcs), dist))
        fg.check(fg.fg_sync())
        bc = torch.empty(g.n, dtype=torch.float64, device=DEV)
        st, info = fg.fg_bc_accumulate(h, s_d, len(srcs), dist, True, bc)
        fg.check(st)
        ref, sigma_max, exact = oracle.bc(g, srcs, True)
        assert exact and info.inexact == 0 and info.sigma_max == sigma_max
        assert np.array_equal(bc.cpu().numpy(), ref)
    finally:
        fg.fg_graph_destroy(h)
