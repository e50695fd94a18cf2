"""Landmark queries around the lines between a warp per pair and slices of
columns (width, kind of load, number of pairs, size of the labels), and the
cost of pairs that no landmark reaches: in slices they must not take much
longer than reached ones."""
import pytest

torch = pytest.importorskip("torch")

from paper_2103_14915_gb300 import fg
from test_gpu_ll_slices import DEV, check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K", [255, 256, 257, 260, 512, 513, 516, 2048])
@pytest.mark.parametrize("Q", [32768, 65535, 65536])
def test_lines_of_the_rule(K, Q):
    check(K, Q)


def test_labels_beyond_l2():
    check(1024, 65536, n=25_700)  # 105 MB


def query_ms(labels, pairs, est):
    times = []
    for _ in range(7):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        a.record()
        fg.check(fg.fg_ll_query(labels, labels.shape[0], labels.shape[1], pairs, pairs.shape[0], est))
        b.record()
        b.synchronize()
        times.append(a.elapsed_time(b))
    return min(times)


@pytest.mark.parametrize("K", [64, 256, 512])
def test_pairs_that_are_not_reached(K):
    n, Q = 4096, 1 << 20
    labels = torch.randint(0, 20000, (n, K), dtype=torch.int32, device=DEV)
    pairs = torch.randint(0, n, (Q, 2), dtype=torch.int32, device=DEV)
    est = torch.empty(Q, dtype=torch.int64, device=DEV)
    reached = query_ms(labels, pairs, est)
    labels.fill_(-1)
    unreached = query_ms(labels, pairs, est)
    assert bool((est == -1).all())
    assert unreached < 1.4 * reached, (unreached, reached)
