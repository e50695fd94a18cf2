"""fg_opts.yield_edges bounds a visit by whole frontiers: with yield_edges = 1 a
visit expands the vertices that were queued when it began and leaves what they
reach to the next one, so a tree inside one partition takes one visit a level.
In both forms of a visit: arc records (out-degrees up to 8) and offsets."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_2103_14915_gb300 import fg, inputs

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def tree(widths):
    """Level sizes; the vertices of a level are spread evenly under the level above. Arcs point away from the root."""
    first = np.concatenate([[0], np.cumsum(widths)])
    edges = []
    for k in range(1, len(widths)):
        for i in range(widths[k]):
            edges.append((int(first[k - 1] + i % widths[k - 1]), int(first[k] + i), 1 + i % 3))
    return inputs.from_edges(int(first[-1]), edges, directed=True)


@pytest.mark.parametrize("widths", [(1, 8, 64, 512), (1, 300, 300)])
def test_one_visit_a_level(widths):
    g = tree(widths)
    assert (g.out_degree().max() <= 8) == (widths[1] == 8)
    st, h = fg.fg_graph_create_ex(g.n, g.m, g.row_ptr, g.col, g.w, 0,
                                  fg.fg_default_graph_opts(partition_method=fg.FG_PART_RANGE, partition_vertices=1024))
    fg.check(st)
    src = np.array([0], dtype=np.int32)
    s_d = torch.from_numpy(src).to(DEV)
    out = torch.empty((1, g.n), dtype=torch.int32, device=DEV)
    try:
        for call, ref in ((fg.fg_bfs_batch, oracle.bfs), (fg.fg_sssp_batch, oracle.sssp)):
            fg.check(call(h, s_d, 1, out, None, fg.fg_default_opts(group=1, yield_edges=1, watchdog_ms=20000)))
            fg.check(fg.fg_sync())
            assert np.array_equal(out.cpu().numpy().view(np.uint32), ref(g, src))
            st, stats = fg.fg_stats(h)
            fg.check(st)
            # the last level has no arcs: its visit ends with it
            assert stats.visits == len(widths) and stats.edges == g.m
    finally:
        fg.fg_graph_destroy(h)
