"""SSSP beyond one heavy arc: every value there is near enough to 2^32 for the
overflow test of the arcs that were left out, which must not cost more than the
batch (a look at every arc of a hub by one thread takes a hundred times that)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_2103_14915_gb300 import fg, inputs

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def batch_ms(h, srcs, out):
    s_d = torch.from_numpy(srcs).to(DEV)
    best = None
    for _ in range(4):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        a.record()
        fg.check(fg.fg_sssp_batch(h, s_d, len(srcs), out))
        b.record()
        fg.check(fg.fg_sync())
        b.synchronize()
        best = a.elapsed_time(b) if best is None else min(best, a.elapsed_time(b))
    return best


def test_sources_behind_a_heavy_arc():
    g0 = inputs.rmat(16, 16, seed=5, weights=(1, 255))
    r = np.random.RandomState(3)
    arcs, hub, far = 1 << 19, int(np.argmax(g0.out_degree())), g0.n
    u = np.concatenate([np.repeat(np.arange(g0.n), g0.out_degree()), [far], np.full(arcs, hub)])
    v = np.concatenate([g0.col, [hub], r.randint(0, g0.n, arcs)])
    w = np.concatenate([g0.w, [2**31 - 1], r.randint(1, 256, arcs)])
    order = np.argsort(u, kind="stable")
    rp = np.zeros(g0.n + 2, np.int64)
    rp[1:] = np.cumsum(np.bincount(u, minlength=g0.n + 1))
    g = inputs.Graph(g0.n + 1, rp, v[order].astype(np.int32), w[order].astype(np.int32), True)
    st, h = fg.fg_graph_create_ex(g.n, g.m, g.row_ptr, g.col, g.w, 0,
                                  fg.fg_default_graph_opts(partition_method=fg.FG_PART_RANGE))
    fg.check(st)
    out = torch.empty((64, g.n), dtype=torch.int32, device=DEV)
    try:
        near = batch_ms(h, inputs.sources_uniform(g, 64, 2).astype(np.int32), out)
        behind = batch_ms(h, np.full(64, far, dtype=np.int32), out)
        assert np.array_equal(out[63].cpu().numpy().view(np.uint32), oracle.sssp(g, [far])[0])
        assert behind < 5 * near, (behind, near)
    finally:
        fg.fg_graph_destroy(h)
