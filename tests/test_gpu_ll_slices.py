"""Landmark queries of many pairs, where the labels are taken in slices of
columns: every width and both kinds of load, the sums around 2^32, pairs without
a common landmark, ids outside the graph, and more pairs than one round takes."""
import pytest

torch = pytest.importorskip("torch")

from paper_2103_14915_gb300 import fg

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
INF = 0xFFFFFFFF


def estimates(labels, pairs):
    """min over k of the finite sums, in 64 bits; all ones where there is none."""
    n = labels.shape[0]
    out = torch.full((pairs.shape[0],), -1, dtype=torch.int64, device=DEV)
    big = 1 << 40
    wide = torch.where(labels < 0, labels.long() + (1 << 32), labels.long())
    wide = torch.where(wide == INF, big, wide)
    for i in range(0, pairs.shape[0], 1 << 15):
        p = pairs[i:i + (1 << 15)].long()
        ok = ((p >= 0) & (p < n)).all(1)
        u, v = torch.where(ok, p[:, 0], 0), torch.where(ok, p[:, 1], 0)
        s = (wide[u] + wide[v]).amin(1)
        out[i:i + (1 << 15)] = torch.where(ok & (s < big), s, -1)
    return out


def check(K, Q, n=700, shift=0, seed=1):
    r = torch.Generator(device=DEV).manual_seed(seed)
    values = torch.randint(0, 1000, (n, K), device=DEV, generator=r)
    kind = torch.arange(n, device=DEV) % 7
    values = torch.where((kind == 1)[:, None], values + 0x7FFFFF00, values)  # sums on both sides of 2^32
    values = torch.where((kind == 2)[:, None], INF - 1 - values % 3, values)  # 2^32 - 1 with a one, and beyond
    values = torch.where((kind == 3)[:, None], values % 2, values)
    values = torch.where((kind == 4)[:, None] | (torch.rand((n, K), device=DEV, generator=r) < 0.2), INF, values)
    flat = torch.zeros(n * K + 8, dtype=torch.int32, device=DEV)
    labels = flat[shift:shift + n * K].view(n, K)
    labels.copy_(torch.where(values > 0x7FFFFFFF, values - (1 << 32), values).int())
    pairs = torch.randint(-1, n + 1, (Q, 2), device=DEV, generator=r, dtype=torch.int32)
    est = torch.zeros(Q, dtype=torch.int64, device=DEV)
    fg.check(fg.fg_ll_query(labels, n, K, pairs, Q, est))
    fg.check(fg.fg_sync())
    assert torch.equal(est, estimates(labels, pairs))


@pytest.mark.parametrize("K", [1, 4, 15, 16, 17, 20, 32, 33, 64, 65, 68, 128, 129, 1023, 1024])
@pytest.mark.parametrize("Q", [32767, 32768, 40001])
def test_widths(K, Q):
    check(K, Q)


def test_unaligned_labels():
    check(64, 33000, shift=1)


def test_two_rounds():
    check(3, 152 * 4 * 8 * 256 + 1)
