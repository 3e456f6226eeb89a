"""Batches whose instances of some enumeration kernel hold no rows at all,
beside instances of other kernels that do: every launch of a batch is made for
the kernels that have work, in order behind the counters' reset."""
import numpy as np
import pytest

import oracle
from paper_2407_20474_gb300 import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CANARY = -7
ROWS = [((5, 8, 11, 14), 500), ((3, 5, 7), 200), ((4, 9, 10, 13, 21), 240)]
# no rows: widths 1, 2 and 9 and, as partial memos, 4 are the general kernel's
EMPTY = {"width 2": [((4, 6), 7)], "width 1": [((7,), 50)],
         "width 9": [((4, 6, 8, 10, 12, 14, 16, 18, 20), 71)],
         "together": [((4, 6), 7), ((7,), 50), ((4, 6, 8, 10, 12, 14, 16, 18, 20), 71), ((6, 4), 1)]}


@pytest.fixture(scope="module")
def fz():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2407_20474_gb300 as m
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    torch.cuda.set_device(0)
    return m


def _check(out, offsets, inst):
    host = out.cpu().numpy()
    assert (host[int(offsets[len(inst)]):] == CANARY).all()
    for j, (g, n) in enumerate(inst):
        if oracle.count(g, n) == 0:
            continue
        ref, at = oracle.enumerate_desc(g, n), int(offsets[j])
        assert np.array_equal(host[at:at + ref.size].reshape(ref.shape), ref), (g, n)


def _run(fz, inst, **kw):
    """Enumeration, rebuild and enumeration, and both captured in a graph."""
    with fz.Batch(inst, **kw) as b:
        assert [int(r) for r in b.rows] == [oracle.count(g, n) for g, n in inst]
        out = torch.full((b.total_words + 8,), CANARY, dtype=torch.int32, device="cuda")
        b.enumerate(out)
        b.sync()
        _check(out, b.word_offsets, inst)
        side, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            b.rebuild(stream=side)
            b.enumerate(out, stream=side)
            side.synchronize()
            with torch.cuda.graph(graph, stream=side):
                b.rebuild(stream=side)
                b.enumerate(out, stream=side)
        for _ in range(3):
            out.fill_(CANARY)
            graph.replay()
            _check(out, b.word_offsets, inst)
        b.sync()


@pytest.mark.parametrize("name", sorted(EMPTY))
def test_general_kernel_without_rows(fz, name):
    inst = EMPTY[name] + ROWS
    _run(fz, inst)
    _run(fz, inst[::-1])
    words = sum(oracle.enumerate_desc(g, n).size + 32 for g, n in inst)
    out = torch.full((words,), CANARY, dtype=torch.int32, device="cuda")
    _check(out, fz.fz_enumerate_batch(inst, out), inst)


def test_autotune_of_general_sets_without_rows(fz):
    try:
        fz.fz_batch_autotune(EMPTY["together"] + ROWS)
        _run(fz, EMPTY["together"] + ROWS)
    finally:
        fz.fz_batch_policy_reset()


def test_partial_memos_without_rows(fz):
    """A partial memo's instances are the general kernel's, those whose element
    lies below its top are not."""
    _run(fz, [((4, 6, 8, 10), 101), ((5, 8, 11, 14), 59), ((3, 5, 7), 50)], top=60)


def test_first_group_without_rows(fz):
    """The costliest kernel's instances hold no rows (even generators, odd
    element, a million prefixes): the next kernel is the first one launched."""
    even = ((2, 4, 6, 8, 10, 12, 14, 16), 4001)
    inst = [even, (even[0], 4003)] + ROWS + [((4, 6), 7)]
    _run(fz, inst)
    with fz.Batch(inst) as b:
        out = torch.empty(b.total_words + 8, dtype=torch.int32, device="cuda")
        for _ in range(20):
            out.fill_(CANARY)
            b.enumerate(out)
            _check(out, b.word_offsets, inst)
        b.sync()


def test_items_of_the_general_kernel(fz):
    """Partial memos of widths 4 to 8 in mixed order: at most eight work items
    for each of 16 warps an SM (an item starts with a dozen dependent loads), and the
    oracle's rows."""
    rng = np.random.Generator(np.random.PCG64(79))
    inst = []
    for i in range(30):
        g = tuple(int(x) for x in rng.integers(8, 60, size=4 + i % 5))
        inst.append((g, workloads.find_n(oracle.count_upto, g, 100000)))
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    with fz.Batch(inst, top=60) as b:
        assert b.work_items <= sms * 16 * 8 + 1 + len(inst)
        out = torch.full((b.total_words + 8,), CANARY, dtype=torch.int32, device="cuda")
        b.enumerate(out)
        b.sync()
        _check(out, b.word_offsets, inst)


@pytest.mark.parametrize("g", [(13, 17, 19, 23, 29, 31, 37, 41, 43), (13, 17, 19, 23, 29, 31, 37, 41, 43, 44)])
def test_cost_of_a_wide_walk(fz, g):
    """Widths above 8 without a memo are walked by the general kernel, where a
    prefix of d - 2 coordinates costs as much as 64 rows: the work items."""
    n = workloads.find_n(oracle.count_upto, g, 30000)
    prefixes = oracle.count(g[:-2] + (1,), n)
    cost = oracle.count(g, n) + 64 * prefixes
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    target = max(4096, cost // (sms * 16 * 8 + 1))
    with fz.Batch([(g, n)], k=0) as b:
        assert b.work_items == -(-cost // target)
        out = torch.full((b.total_words + 8,), CANARY, dtype=torch.int32, device="cuda")
        b.enumerate(out)
        b.sync()
        _check(out, b.word_offsets, [(g, n)])
