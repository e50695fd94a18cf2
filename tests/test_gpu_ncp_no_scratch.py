"""The NCP sweep without device memory for its scratch: the stream-ordered
allocator is made to refuse (a memory pool of the smallest size, used up), and
the call has to give the same sweep without it."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_2103_14915_gb300 import fg, inputs

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


class PoolProps(ctypes.Structure):
    _fields_ = [("alloc_type", ctypes.c_int), ("handle_types", ctypes.c_int), ("location_type", ctypes.c_int),
                ("location_id", ctypes.c_int), ("security", ctypes.c_void_p), ("max_size", ctypes.c_size_t),
                ("usage", ctypes.c_ushort), ("reserved", ctypes.c_ubyte * 54)]


class NoPoolMemory:
    """The device's current memory pool is one of at most `limit` bytes, all of them taken."""

    def __init__(self, limit=1 << 21):
        self.cu = ctypes.CDLL("libcuda.so.1")
        self.limit = limit

    def call(self, name, *args):
        st = getattr(self.cu, name)(*args)
        assert st == 0, (name, st)

    def __enter__(self):
        torch.cuda.synchronize()
        self.before, self.pool = ctypes.c_void_p(), ctypes.c_void_p()
        self.call("cuDeviceGetMemPool", ctypes.byref(self.before), 0)
        props = PoolProps(alloc_type=1, location_type=1, location_id=0, max_size=self.limit)  # pinned, on device 0
        self.call("cuMemPoolCreate", ctypes.byref(self.pool), ctypes.byref(props))
        self.held = []
        self.call("cuDeviceSetMemPool", 0, self.pool)
        for size in (1 << 21, 1 << 18, 1 << 14, 1 << 9):
            for _ in range(64):
                p = ctypes.c_void_p()
                if self.cu.cuMemAllocAsync(ctypes.byref(p), ctypes.c_size_t(size), None) != 0:
                    break
                self.held.append(p)
            else:
                self.__exit__()
                pytest.skip("the driver does not hold the pool to its size")
        return self

    def __exit__(self, *_):
        self.call("cuDeviceSetMemPool", 0, self.before)
        for p in self.held:
            self.call("cuMemFreeAsync", p, None)
        torch.cuda.synchronize()
        self.call("cuMemPoolDestroy", self.pool)


@pytest.mark.parametrize("accumulate", [False, True])
def test_same_sweep_without_scratch(accumulate):
    g = inputs.rmat(17, 8, seed=21)
    top, nq = 1000, 3
    r = np.random.RandomState(4)
    rows = (r.rand(nq, g.n) * (r.rand(nq, g.n) < 0.05)).astype(np.float32)
    order_ref, phi_ref, count_ref = oracle.ncp_sweep(g, rows, top)
    assert (count_ref == top).all()
    ncp_ref = phi_ref.min(axis=0)
    st, h = fg.fg_graph_create(g.n, g.m, g.row_ptr, g.col, None, 0)
    fg.check(st)
    try:
        p = torch.from_numpy(rows).to(DEV)
        order = torch.empty((nq, top), dtype=torch.int32, device=DEV)
        phi = torch.empty((nq, top), dtype=torch.float64, device=DEV)
        count = torch.empty(nq, dtype=torch.int32, device=DEV)
        ncp = torch.full((top,), 0.25 if accumulate else -1.0, dtype=torch.float64, device=DEV)
        fg.check(fg.fg_ncp_sweep(h, p, 1, top, order))  # the graph's degree table
        with NoPoolMemory():
            st = fg.fg_ncp_sweep(h, p, nq, top, order, phi, count, ncp, accumulate)
            torch.cuda.synchronize()
        fg.check(st)
        assert np.array_equal(count.cpu().numpy(), count_ref)
        assert np.array_equal(order.cpu().numpy(), order_ref)
        assert np.array_equal(phi.cpu().numpy(), phi_ref, equal_nan=True)
        assert np.array_equal(ncp.cpu().numpy(), np.minimum(ncp_ref, 0.25) if accumulate else ncp_ref)
    finally:
        fg.fg_graph_destroy(h)
