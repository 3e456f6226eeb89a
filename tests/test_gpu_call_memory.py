"""Device memory of calls that keep no handle: what they took is free for any
other allocator when they return, but for a bounded rest."""
import ctypes

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

KEPT = 64 << 20


@pytest.fixture(scope="module")
def fz():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2407_20474_gb300 as m
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    torch.cuda.set_device(0)
    return m


def _free():
    """cuMemGetInfo: no synchronisation, unlike the allocators' own calls."""
    drv = ctypes.CDLL("libcuda.so.1")
    a, b = ctypes.c_size_t(), ctypes.c_size_t()
    assert drv.cuMemGetInfo_v2(ctypes.byref(a), ctypes.byref(b)) == 0
    return a.value


def test_calls_give_their_memory_back(fz):
    g, n = (50, 60, 71, 77), 30000000  # a count table of 1.2 GB, rolling rows of 480 MB
    tail, top = (7, 10, 11, 19, 39), 1100
    rows = fz.fz_memo_rows(tail, top)
    off = torch.zeros(top + 1, dtype=torch.int64, device="cuda")
    out = torch.zeros((rows, len(tail)), dtype=torch.int32, device="cuda")
    few = torch.zeros((1000, 4), dtype=torch.int32, device="cuda")
    host = torch.zeros((1000, 4), dtype=torch.int32).pin_memory()
    calls = [lambda: fz.fz_count(g, n), lambda: fz.fz_count_upto(g, n), lambda: fz.fz_memo_rows((2, 3), n),
             lambda: fz.fz_build_memo_into(tail, top, off, out, rows),
             lambda: fz.fz_enumerate(g, n, few, 0, 1000), lambda: fz.fz_enumerate_host(g, n, host, 0, 1000)]
    fz.fz_count((3, 5), 100)
    for call in calls:  # kernels and streams of each made once
        call()
    torch.cuda.synchronize()
    start = _free()
    for i, call in enumerate(calls):
        call()
        assert _free() >= start - KEPT, i


def test_a_failed_allocation_is_reported_once(fz):
    """Tables larger than the device: the call says so, and the next one works."""
    g = tuple(range(1, 17))
    for make in (lambda: fz.Plan(g, 2**31 - 2, k=0), lambda: fz.Batch([(g, 2**31 - 2)]),
                 lambda: fz.Batch([((5, 8, 11, 14), 500), (g, 2**31 - 2)]),
                 lambda: fz.Server(memory_bytes=1 << 42)):
        with pytest.raises(fz.FzError, match="ENOMEM"):
            make()
        assert fz.fz_count((5, 8, 11, 14), 500) == 3783
        with fz.Plan((5, 8, 11, 14), 500) as plan:
            assert plan.count == 3783
