"""Sweep cuts where the way to the kept vertices changes, against the oracle:
rows listed whole and rows sampled, sizes around the lines between them, lists
that come out too long (ties) or too short (mass where the sample does not
look), more rows than one launch takes, and hubs whose arcs are cut into pieces."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_2103_14915_gb300 import fg, inputs

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def graph(n, seed=1):
    """Sparse, with two hubs."""
    r = np.random.RandomState(seed)
    k = 3 * n
    u, v = r.randint(0, n, k), r.randint(0, n, k)
    u[: n // 2] = 7 % n
    u[n // 2: n // 2 + n // 9] = n - 1
    row_ptr, col = inputs.csr_from_edges(n, u, v, True)
    return inputs.Graph(n, row_ptr, col, None, False)


def rows(n, kind, nq, seed=3):
    r = np.random.RandomState(seed)
    p = np.exp(1.5 * r.randn(nq, n)).astype(np.float32) * np.float32(1e-6)
    if kind == "sparse":
        p *= r.rand(nq, n) < 0.1
    elif kind == "ties":  # one value for all, and a few above it
        p[:] = 1e-6
        p[:, ::997] = 2e-6
    elif kind == "clustered":  # the largest keys side by side, in a few places
        p *= np.float32(1e-3)
        for a in (0, n // 3, n - 2600):
            a = max(0, a)
            p[:, a:a + 2600] *= np.float32(1e6)
    return p


@pytest.mark.parametrize("n", [300, 2049, 16384, 16385, 24577, 65536, 65540, 200001])
@pytest.mark.parametrize("kind", ["spread", "sparse", "ties", "clustered"])
def test_kept_set(n, kind):
    g = graph(n)
    st, h = fg.fg_graph_create_ex(g.n, g.m, g.row_ptr, g.col, None, 0, fg.fg_default_graph_opts())
    fg.check(st)
    try:
        p = rows(n, kind, 2)
        p_d = torch.from_numpy(p).to(DEV)
        for top in (1, 300, 4096):
            order = torch.empty((2, top), dtype=torch.int32, device=DEV)
            phi = torch.empty((2, top), dtype=torch.float64, device=DEV)
            count = torch.empty(2, dtype=torch.int32, device=DEV)
            ncp = torch.empty(top, dtype=torch.float64, device=DEV)
            fg.check(fg.fg_ncp_sweep(h, p_d, 2, top, order, phi, count, ncp))
            fg.check(fg.fg_sync())
            ref = oracle.ncp_sweep(g, p, top)
            assert np.array_equal(count.cpu().numpy(), ref[2])
            assert np.array_equal(order.cpu().numpy(), ref[0])
            assert np.array_equal(phi.cpu().numpy(), ref[1], equal_nan=True)
            best = np.where(np.isnan(ref[1]), np.inf, ref[1]).min(0)
            assert np.array_equal(ncp.cpu().numpy(), best)
    finally:
        fg.fg_graph_destroy(h)


@pytest.mark.parametrize("n", [300, 24580])
def test_more_rows_than_a_launch_takes_and_a_profile_over_two_calls(n):
    g = graph(n)
    st, h = fg.fg_graph_create_ex(g.n, g.m, g.row_ptr, g.col, None, 0, fg.fg_default_graph_opts())
    fg.check(st)
    try:
        p = rows(n, "sparse", 1030)
        p_d = torch.from_numpy(p).to(DEV)
        order = torch.empty((1030, 50), dtype=torch.int32, device=DEV)
        phi = torch.empty((1030, 50), dtype=torch.float64, device=DEV)
        ncp = torch.empty(50, dtype=torch.float64, device=DEV)
        fg.check(fg.fg_ncp_sweep(h, p_d[1020:], 10, 50, None, None, None, ncp))
        fg.check(fg.fg_ncp_sweep(h, p_d[:1029], 1029, 50, order, phi, None, ncp, True))
        fg.check(fg.fg_sync())
        ref = oracle.ncp_sweep(g, p, 50)
        assert np.array_equal(order[:1029].cpu().numpy(), ref[0][:1029])
        assert np.array_equal(phi[:1029].cpu().numpy(), ref[1][:1029], equal_nan=True)
        assert np.array_equal(ncp.cpu().numpy(), np.where(np.isnan(ref[1]), np.inf, ref[1]).min(0))
    finally:
        fg.fg_graph_destroy(h)
