"""Graph creation is synchronous: when it returns, the graph is on the device
for every stream, those that do not order after the default stream included."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_2103_14915_gb300 import fg, inputs

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("weighted", [False, True])
def test_nothing_is_left_on_the_default_stream(weighted):
    g = inputs.grid(2000, 2000, seed=3, weights=(100, 10000))
    srcs = np.array([0, g.n // 2 + 17], dtype=np.int32)
    ref = oracle.bfs(g, srcs)
    s_d = torch.from_numpy(srcs).to(DEV)
    out = torch.empty((len(srcs), g.n), dtype=torch.int32, device=DEV)
    side = torch.cuda.Stream()  # non-blocking
    torch.cuda.synchronize()
    opts = fg.fg_default_opts(sched=fg.FG_SCHED_PRIORITY, sched_window=24, watchdog_ms=20000)
    for _ in range(2):  # the first graph of a process also sets up the device
        st, h = fg.fg_graph_create(g.n, g.m, g.row_ptr, g.col, g.w if weighted else None, 0)
        idle = torch.cuda.default_stream().query()
        fg.check(st)
        try:
            assert idle
            fg.check(fg.fg_bfs_batch(h, s_d, len(srcs), out, side, opts))
            fg.check(fg.fg_sync(side))
            assert np.array_equal(out.cpu().numpy().view(np.uint32), ref)
        finally:
            fg.fg_graph_destroy(h)
