"""SSSP / BFS visits of the query-major engine where the arcs of a vertex stand
in records of fixed size (out-degrees up to 8) and just beyond, against the
oracle: degrees around a half and a whole record, loops and parallel arcs,
partitions from one bitmap word to the largest, wide and narrow frontiers, and
the options that leave work to later visits."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_2103_14915_gb300 import fg, inputs

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def wheel(n, deg, far):
    """n vertices of `deg` or fewer out-arcs: to near ones (a loop and a parallel arc among them), one to a far one."""
    r = np.random.RandomState(100 * n + deg)
    v = np.arange(n)
    cols = [(v + 1) % n, v, (v + 1) % n]
    cols += [(v + r.randint(2, 40)) % n for _ in range(deg - 4)]
    cols.append((v * 7 + far) % n)
    col = np.stack(cols[:deg], 1)
    keep = r.rand(n, deg) < 0.9
    keep[0] = True  # one vertex has them all
    rp = np.zeros(n + 1, np.int64)
    rp[1:] = np.cumsum(keep.sum(1))
    w = r.randint(0, 1000, (n, deg))
    return inputs.Graph(n, rp, col[keep].astype(np.int32), w[keep].astype(np.int32), True)


OPTS = [dict(), dict(sched=fg.FG_SCHED_PRIORITY, sched_window=700, delta=300), dict(bucket=90, delta=400),
        dict(emit_capacity=1), dict(yield_edges=3)]


@pytest.mark.parametrize("deg", [4, 5, 8, 9])
@pytest.mark.parametrize("S", [32, 1024, 4096])
def test_records(deg, S):
    g = wheel(5 * S // 2 + 7 if S < 4096 else 9001, deg, 11)
    assert g.out_degree().max() == deg
    srcs = np.array([0, 1, g.n - 1, 0] + list(range(5, g.n, g.n // 30)), dtype=np.int32)
    sssp, bfs = oracle.sssp(g, srcs), oracle.bfs(g, srcs)
    st, h = fg.fg_graph_create_ex(g.n, g.m, g.row_ptr, g.col, g.w, 0,
                                  fg.fg_default_graph_opts(partition_method=fg.FG_PART_RANGE, partition_vertices=S))
    fg.check(st)
    s_d = torch.from_numpy(srcs).to(DEV)
    out = torch.empty((len(srcs), g.n), dtype=torch.int32, device=DEV)
    try:
        for opts in OPTS:
            for nq in (1, len(srcs)):
                o = fg.fg_default_opts(group=1, watchdog_ms=20000, **opts)
                fg.check(fg.fg_sssp_batch(h, s_d, nq, out, None, o))
                fg.check(fg.fg_sync())
                assert np.array_equal(out[:nq].cpu().numpy().view(np.uint32), sssp[:nq]), opts
                fg.check(fg.fg_bfs_batch(h, s_d, nq, out, None, o))
                fg.check(fg.fg_sync())
                assert np.array_equal(out[:nq].cpu().numpy().view(np.uint32), bfs[:nq]), opts
    finally:
        fg.fg_graph_destroy(h)
