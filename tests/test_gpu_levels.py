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


SPARSE = [((401, 397, 389, 383), 300), ((83, 97, 89, 101, 103), 900), ((59, 61, 60, 67, 71, 73), 2000),
          ((41, 43, 44, 47, 53, 51, 59), 6000)]


@pytest.mark.parametrize("g,target", SPARSE)
def test_rank_walk_windows(fz, g, target):
    """Sets with far more prefixes than rows: windows of the rank walk at every
    remainder of a round, outputs aligned to 4 bytes only."""
    n = workloads.find_n(oracle.count_upto, g, target)
    ref = oracle.enumerate_desc(g, n)
    total = ref.shape[0]
    for slice_rows in (4, 33, 0):
        for shift, a, b in ((0, 0, total), (1, 0, total), (3, 1, total - 1), (2, total - 1, total),
                            (1, total // 3, total // 3 + 33)):
            got = _window(fz, g, n, 0, a, b, slice_rows, shift)
            assert np.array_equal(got, ref[a:b]), (slice_rows, shift, a, b)


def test_rank_walk_in_batches(fz):
    """The same sets in one batch without memos, beside dense ones and sets of
    no row and of one."""
    inst = [(g, workloads.find_n(oracle.count_upto, g, t // c)) for g, t in SPARSE for c in (1, 3)]
    inst += [((5, 7, 9, 11), 300), (SPARSE[0][0], 382), (SPARSE[0][0], 383), (SPARSE[1][0], inst[1][1] + 1)]
    with fz.Batch(inst, k=0) as b:
        out = torch.full((b.total_words + 8,), CANARY, dtype=torch.int32, device="cuda")
        b.enumerate(out)
        b.sync()
        host = out.cpu().numpy()
        assert (host[b.total_words:] == CANARY).all()
        for j, (g, n) in enumerate(inst):
            at, ref = int(b.word_offsets[j]), oracle.enumerate_desc(g, n)
            assert np.array_equal(host[at:at + ref.size].reshape(ref.shape), ref), (g, n)


def test_serve_resident_shapes(fz):
    """Requests far below and at a resident set's largest element: tables of
    every depth, and (large generators up to 3e6) none, served by rank."""
    sets = [((997, 1009, 1013, 1019), 3000000, 200000), ((5, 8, 11, 14, 17), 900, 300), ((9, 6, 12, 15, 21, 10), 220, 90),
            ((13, 4, 7, 30, 22, 9, 17), 160, 161), ((3, 5, 7), 3000, 1)]
    with fz.Server(memory_bytes=64 << 20) as srv:
        ids = [srv.register(g, max(top, n)) for g, top, n in sets]
        asked = [(i, s[0], n) for i, s in zip(ids, sets) for n in (s[2], s[2] // 2, 0)]
        tickets = [srv.submit(i, n) for i, _, n in asked]
        for t, (_, g, n) in zip(tickets, asked):
            r = srv.wait(t)
            ref = oracle.enumerate_desc(g, n)
            assert int(r.count) == ref.shape[0], (g, n)
            out = torch.full((ref.size + 4,), CANARY, dtype=torch.int32, device="cuda")
            srv.copy(t, out[:ref.size])
            srv.release(t)
            host = out.cpu().numpy()
            assert (host[ref.size:] == CANARY).all()
            assert np.array_equal(host[:ref.size].reshape(ref.shape), ref), (g, n)


@pytest.mark.parametrize("n", [0, 1, 2, 255, 256, 4095, 11999, 12000, 12001])
def test_short_count_tables(fz, n):
    """Count tables up to the one-launch range and past it: generators of 1,
    above n, at n, repeated, and counts that saturate (width 16)."""
    for g in ((3, 5, 7, 11), (n + 1, 4, 9), (max(n, 1), 2, 2), (1, 6), (7,), tuple(range(1, 17))):
        d = len(g)
        out = torch.zeros((d + 1, n + 1), dtype=torch.int64, device="cuda")
        fz.fz_count_table(g, n, out)
        torch.cuda.synchronize()
        got = out.cpu().numpy().view(np.uint64)
        for j in range(d):
            ref = np.array([min(int(x), 2**64 - 1) for x in oracle.count_upto(g[j:], n)], dtype=np.uint64)
            assert np.array_equal(got[j], ref), (g, j)


@pytest.mark.parametrize("n", [2999, 3000, 3001])
def test_one_launch_count_tables(fz, n):
    """Both sides of the longest single table built in one launch."""
    test_short_count_tables(fz, n)


@pytest.mark.parametrize("g,n", [((70001, 65537), 150000), ((131071, 3, 65536), 150000), ((6, 4), 13000),
                                 ((4, 2, 2, 9), 20000), ((9,), 12500), ((1, 1), 12001), ((200000, 300000), 100000)])
def test_closed_count_rows(fz, g, n):
    """The last rows of longer count tables from their closed forms (moduli on
    both sides of 2^16, common factors, generators above n) and the rolling
    counts that start from them."""
    d = len(g)
    out = torch.full((d + 1, n + 1), CANARY, dtype=torch.int64, device="cuda")
    fz.fz_count_table(g, n, out)
    torch.cuda.synchronize()
    got = out.cpu().numpy()
    assert got[d, 0] == 1 and (got[d, 1:] == 0).all()
    for j in range(d):
        assert np.array_equal(got[j].astype(np.uint64), oracle.count_upto(g[j:], n)), j
    assert np.array_equal(fz.fz_count_upto(g, n), oracle.count_upto(g, n))


# (generators, n): rows scanned by tiles and by lanes: 256 and 257 entries a
# chain, 7, 8, 31 and 32 chains, one long chain, wrapping lengths around 16384
CHAINS = [((7, 50), 7 * 256 - 1), ((7, 50), 7 * 256), ((8, 31), 8 * 300), ((31, 8), 31 * 256 + 5), ((32, 31), 32 * 257),
          ((1, 2, 3), 16383), ((1, 2, 3), 16384), ((2, 1), 40001), ((64, 1), 64 * 255 + 63)]


@pytest.mark.parametrize("g,n", CHAINS)
def test_batch_chain_scans(fz, g, n):
    """Batch counts of the chains above: the rows of d = 2 and 3 sets, alone and
    among many small ones, against the oracle's counts."""
    many = [((5, 8, 11), 90 + i) for i in range(40)]
    for inst in ([(g, n)], [(g, n)] + many):
        _, rows = fz.fz_plan_batch(inst)
        assert [int(r) for r in rows] == [oracle.count(x, m) for x, m in inst]


def test_calls_after_a_context_reset(fz):
    """Counts and a host enumeration before and after the process resets its own
    device context (in a child process): function attributes and the memory
    pool are those of the new context."""
    import subprocess
    import sys
    code = """
import ctypes, numpy as np, oracle
import paper_2407_20474_gb300 as fz
drv = ctypes.CDLL('libcuda.so.1')
g, n = (5, 8, 11, 14), 9000
ref, rows = oracle.count_upto(g, n), oracle.enumerate_desc(g, 500)
for k in range(3):
    assert np.array_equal(fz.fz_count_upto(g, n, stream=0), ref), k
    out = np.full(rows.shape, -7, dtype=np.int32)
    fz.fz_enumerate_host(g, 500, out, stream=0)
    assert np.array_equal(out, rows), k
    if k < 2:
        dev = ctypes.c_int()
        assert drv.cuDeviceGet(ctypes.byref(dev), 0) == 0
        assert drv.cuDevicePrimaryCtxReset_v2(dev) == 0
print('same')
"""
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=300,
                       cwd=__import__("os").path.dirname(__import__("os").path.dirname(__file__)))
    assert r.returncode == 0 and r.stdout.strip().endswith("same"), r.stderr[-2000:]
