"""Memos and run-order tables built by levels against the oracle, and plans
that read them (enumeration and random access)."""
import numpy as np
import pytest

import oracle
from paper_2407_20474_gb300 import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CANARY = -7


@pytest.fixture(scope="module")
def fz():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2407_20474_gb300 as m
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    torch.cuda.set_device(0)
    return m


# depths 1..9 (9: past the levels), every order, repeats, common factors, a 1,
# generators above the last element, one element, ring and warp-window
# remainders
TAILS = [((5,), 40), ((11, 14), 501), ((14, 11), 501), ((4, 9, 10), 300), ((10, 4, 9), 301), ((2, 2, 3), 130),
         ((6, 10, 15), 400), ((5, 1, 4), 200), ((900, 3, 4, 5), 310), ((3, 900, 4, 5), 310), ((3, 5, 7, 8), 260),
         ((7, 5, 6, 4, 9), 150), ((4, 6, 8, 10, 12, 14), 170), ((3, 4, 5, 6, 7, 8, 9), 75),
         ((3, 4, 5, 6, 7, 8, 9, 10), 60), ((3, 4, 5, 6, 7, 8, 9, 10, 11), 45), ((4, 9, 10), 1), ((7, 3, 5, 2), 2),
         ((33, 2, 3, 5), 700)]


@pytest.mark.parametrize("tail,top", TAILS)
@pytest.mark.parametrize("shift", [0, 1])
def test_memo_by_levels(fz, tail, top, shift):
    """shift: rows at an address that is 4-byte aligned only."""
    ref_off, ref_rows = oracle.memo_csr(tail, top)
    rows, k = int(ref_off[-1]), len(tail)
    off = torch.zeros(top + 1, dtype=torch.int64, device="cuda")
    buf = torch.full((shift + (rows + 4) * k,), CANARY, dtype=torch.int32, device="cuda")
    assert fz.fz_build_memo_into(tail, top, off, buf[shift:], rows) == rows
    torch.cuda.synchronize()
    host = buf.cpu().numpy()
    assert (host[:shift] == CANARY).all() and (host[shift + rows * k:] == CANARY).all()
    assert np.array_equal(off.cpu().numpy().view(np.uint64), ref_off)
    assert np.array_equal(host[shift:shift + rows * k].reshape(rows, k), ref_rows)


@pytest.mark.parametrize("g,target", [((5, 8, 11, 14), 4000), ((14, 5, 11, 8, 9), 9000), ((2, 2, 3, 3), 5000),
                                      ((9, 6, 12, 15, 21, 10), 20000), ((400, 7, 3, 5), 3000),
                                      ((3, 5, 7, 9, 11, 13, 4), 30000), ((13, 37, 38, 40, 41, 42, 43, 44, 45), 20000)])
def test_plans_on_levels(fz, g, target):
    """Every memo depth: enumeration after two rebuilds, and the tuple of every
    rank by random access."""
    n = workloads.find_n(oracle.count_upto, g, target, 64)
    ref = oracle.enumerate_desc(g, n)
    total, d = ref.shape
    ranks = torch.randperm(total, device="cuda")
    for k in range(1, d):
        with fz.Plan(g, n, k=k) as plan:
            for _ in range(2):
                plan.rebuild()
            out = torch.full((total + 3, d), CANARY, dtype=torch.int32, device="cuda")
            assert plan.enumerate(out[:total]) == total
            pick = torch.full((total + 3, d), CANARY, dtype=torch.int32, device="cuda")
            plan.unrank(ranks, pick[:total])
            plan.sync()
            assert np.array_equal(out[:total].cpu().numpy(), ref), k
            assert np.array_equal(pick[:total].cpu().numpy(), ref[ranks.cpu().numpy()]), k
            assert bool((out[total:] == CANARY).all()) and bool((pick[total:] == CANARY).all())


def _window(fz, g, n, k, begin, end, slice_rows, shift):
    d = len(g)
    out = torch.full((shift + (end - begin + 3) * d,), CANARY, dtype=torch.int32, device="cuda")
    with fz.Plan(g, n, k=k, slice_rows=slice_rows) as plan:
        assert plan.enumerate(out[shift:], begin, end) == end - begin
        plan.sync()
    host = out.cpu().numpy()
    last = shift + (end - begin) * d
    assert (host[:shift] == CANARY).all() and (host[last:] == CANARY).all()
    return host[shift:last].reshape(-1, d)


@pytest.mark.parametrize("d", [3, 4, 5, 6, 7, 8, 9])
@pytest.mark.parametrize("lo,hi", [(2, 9), (20, 60)])
def test_flat_walk(fz, d, lo, hi):
    """Leaves of one to three prefix words over run-order tables and of d - 2
    over the pair's closed form (k = 0): dense leaves (small generators) and
    mostly empty ones (large generators), items that start inside a leaf,
    ring remainders, rank windows, outputs aligned to 4 bytes only."""
    rng = np.random.Generator(np.random.PCG64(1000 * d + lo))
    g = tuple(int(x) for x in rng.integers(lo, hi, size=d))
    n = workloads.find_n(oracle.count_upto, g, 12000)
    ref = oracle.enumerate_desc(g, n)
    total = ref.shape[0]
    for k in {0, d - 2, max(0, d - 3), max(0, d - 4), -1}:
        for slice_rows in (4, 100, 0):
            assert np.array_equal(_window(fz, g, n, k, 0, total, slice_rows, 0), ref), (g, n, k)
        for shift in (0, 1, 2):
            a, b = sorted(int(x) for x in rng.integers(0, total, size=2))
            got = _window(fz, g, n, k, a, b + 1, 40, shift)
            assert np.array_equal(got, ref[a:b + 1]), (g, n, k, a, b, shift)


def test_batch_flat_shapes(fz):
    """Every shape of the batch kernel's flat walk in one batch, and each depth
    on its own."""
    rng = np.random.Generator(np.random.PCG64(77))
    inst = []
    for d in range(3, 9):
        for lo, hi, target in ((2, 12, 6000), (15, 70, 3000), (40, 200, 300)):
            g = tuple(int(x) for x in rng.integers(lo, hi, size=d))
            inst.append((g, workloads.find_n(oracle.count_upto, g, target)))
    refs = [oracle.enumerate_desc(g, n) for g, n in inst]
    for k in (-1, 0, 1, 2, 3, 4, 5, 6):
        sub = [i for i, (g, _) in enumerate(inst) if k <= len(g) - 1]
        with fz.Batch([inst[i] for i in sub], k=k) as b:
            out = torch.full((b.total_words + 8,), CANARY, dtype=torch.int32, device="cuda")
            b.rebuild()
            b.enumerate(out)
            b.sync()
            host = out.cpu().numpy()
            assert (host[b.total_words:] == CANARY).all()
            for j, i in enumerate(sub):
                at, ref = int(b.word_offsets[j]), refs[i]
                assert np.array_equal(host[at:at + ref.size].reshape(ref.shape), ref), (inst[i], k)


def test_batch_in_a_graph(fz):
    """Rebuild and enumeration captured in a CUDA graph (the overlapped launches
    of the shapes included) and replayed: the same bytes, twice."""
    rng = np.random.Generator(np.random.PCG64(78))
    inst = []
    for d in (3, 4, 5, 6, 7, 8, 2, 9):
        g = tuple(int(x) for x in rng.integers(5, 40, size=d))
        inst.append((g, workloads.find_n(oracle.count_upto, g, 20000)))
    with fz.Batch(inst) as b:
        out = torch.full((b.total_words + 8,), CANARY, dtype=torch.int32, device="cuda")
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.stream(side):
            b.rebuild(stream=side)
            b.enumerate(out, stream=side)
            side.synchronize()
            with torch.cuda.graph(graph, stream=side):
                b.rebuild(stream=side)
                b.enumerate(out, stream=side)
        for _ in range(2):
            out.fill_(CANARY)
            graph.replay()
            # the end of the graph is the end of every launch in it
            host = out.cpu().numpy()
            for j, (g, n) in enumerate(inst):
                ref = oracle.enumerate_desc(g, n)
                at = int(b.word_offsets[j])
                assert np.array_equal(host[at:at + ref.size].reshape(ref.shape), ref), (g, n)
        b.sync()
