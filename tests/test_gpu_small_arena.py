"""An operation arena that holds a round's operations must not slow the round
down, however few slots it has: 64 queries run along a directed path, each
visit sends one operation into the next partition, 64 a round, so an arena of
128 slots (visits stop at 96) takes exactly the rounds of an unlimited one."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_2103_14915_gb300 import fg, inputs

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("kind", ["bfs", "sssp"])
def test_every_slot_is_used(kind):
    n = 2048
    g = inputs.from_edges(n, [(i, i + 1, 1 + i % 5) for i in range(n - 1)], directed=True)
    st, h = fg.fg_graph_create_ex(g.n, g.m, g.row_ptr, g.col, g.w, 0,
                                  fg.fg_default_graph_opts(partition_method=fg.FG_PART_RANGE, partition_vertices=32))
    fg.check(st)
    srcs = np.arange(64, dtype=np.int32) % 32  # all in the first partition
    call, ref = (fg.fg_bfs_batch, oracle.bfs(g, srcs)) if kind == "bfs" else (fg.fg_sssp_batch, oracle.sssp(g, srcs))
    s_d = torch.from_numpy(srcs).to(DEV)
    out = torch.empty((len(srcs), g.n), dtype=torch.int32, device=DEV)
    rounds = []
    try:
        for slots in (0, 128):
            fg.check(call(h, s_d, len(srcs), out, None, fg.fg_default_opts(group=1, emit_capacity=slots,
                                                                          watchdog_ms=20000)))
            fg.check(fg.fg_sync())
            assert np.array_equal(out.cpu().numpy().view(np.uint32), ref)
            st, stats = fg.fg_stats(h)
            fg.check(st)
            assert stats.spills == 0
            rounds.append(stats.rounds)
        assert rounds[0] == n // 32 and rounds[1] == rounds[0]
    finally:
        fg.fg_graph_destroy(h)
