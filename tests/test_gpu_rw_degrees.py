"""Random walks from vertices whose degree lies around the line between the two
ways to the remainder, against the oracle, bit for bit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_2103_14915_gb300 import fg, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("degree", [1, 2, 3, 255, 32767, 32768, 50001])
def test_hub_and_leaves(degree):
    n = degree + 1  # every leaf goes back to the hub: each second step draws from `degree` arcs
    row_ptr, col = inputs.csr_from_edges(n, np.zeros(degree, np.int64), np.arange(1, n), True)
    g = inputs.Graph(n, row_ptr, col, None, False)
    srcs = np.zeros(3000, np.int32)
    st, h = fg.fg_graph_create_ex(g.n, g.m, g.row_ptr, g.col, None, 0, fg.fg_default_graph_opts())
    fg.check(st)
    try:
        paths = torch.empty((srcs.size, 41), dtype=torch.int32, device="cuda:0")
        fg.check(fg.fg_rw_batch(h, torch.from_numpy(srcs).to("cuda:0"), srcs.size, 40, 11, paths))
        fg.check(fg.fg_sync())
        assert np.array_equal(paths.cpu().numpy(), oracle.rw(g, srcs, 40, 11))
    finally:
        fg.fg_graph_destroy(h)
