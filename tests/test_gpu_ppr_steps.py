"""PPR pushes from vertices whose arcs end inside, at or just beyond the steps of
32 and 128 arcs that a visit takes together, and from vertices without arcs."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2103_14915_gb300 import fg, inputs

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
ALPHA, EPS = 0.15, 1e-7


def exact(g, s):
    """Power iteration in FP64; a vertex without arcs sends everything back to the source."""
    deg = np.diff(g.row_ptr)
    u = np.repeat(np.arange(g.n), deg)
    x = np.zeros(g.n)
    x[s] = 1.0
    p = np.zeros(g.n)
    for _ in range(400):  # 0.85^400 < 1e-28
        p += ALPHA * x
        y = np.zeros(g.n)
        np.add.at(y, g.col, (1 - ALPHA) * (x / np.maximum(deg, 1))[u])
        y[s] += (1 - ALPHA) * x[deg == 0].sum()
        x = y
    return p


@pytest.mark.parametrize("degree", [1, 31, 32, 33, 127, 128, 129, 1500])
@pytest.mark.parametrize("directed", [False, True])
def test_hub(degree, directed):
    """A hub (0) with `degree` leaves, the last of which leads on to vertex degree + 1 (and back, undirected)."""
    n = degree + 2
    u, v = np.append(np.zeros(degree, np.int64), degree), np.append(np.arange(1, degree + 1), degree + 1)
    row_ptr, col = inputs.csr_from_edges(n, u, v, not directed)
    g = inputs.Graph(n, row_ptr, col, None, directed)
    src = np.array([0, 1, degree + 1], np.int32)
    opts = fg.fg_default_graph_opts()
    st, h = fg.fg_graph_create_ex(g.n, g.m, g.row_ptr, g.col, None, 0, opts)
    fg.check(st)
    try:
        p = torch.empty((3, n), dtype=torch.float32, device=DEV)
        r = torch.empty((3, n), dtype=torch.float32, device=DEV)
        mass = torch.empty(3, dtype=torch.float64, device=DEV)
        fg.check(fg.fg_ppr_batch(h, torch.from_numpy(src).to(DEV), 3, ALPHA, EPS, p, r, mass))
        fg.check(fg.fg_sync())
        p, r = p.cpu().numpy().astype(np.float64), r.cpu().numpy().astype(np.float64)
        deg = np.maximum(np.diff(g.row_ptr), 1)
        for i, s in enumerate(src):
            assert (r[i] >= 0).all() and (r[i] < EPS * deg * (1 + 1e-5)).all()
            # what is left is at most all residuals; FP32 sums of up to `degree` terms of at most 1
            d = exact(g, s) - p[i]
            slack = (n + 64) * 2.0 ** -24
            assert d.min() >= -slack and d.max() <= r[i].sum() + slack
    finally:
        fg.fg_graph_destroy(h)
