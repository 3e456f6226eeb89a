"""The occupancy cap of the enumeration leaves room for another plan's (or
batch's) rebuild: with both capped, the rebuild ends long before the enumeration
that was already running when it began."""
import pytest

import oracle
from paper_2407_20474_gb300 import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

WIDE = (53, 71, 91, 115, 176, 195)


@pytest.fixture(scope="module")
def fz():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2407_20474_gb300 as m
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    torch.cuda.set_device(0)
    return m


def _ends(long, other, out):
    """Milliseconds from a common start to the end of `long`'s enumeration and of
    `other`'s rebuild, enqueued behind it on a stream of its own."""
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(3)]
    enum, side = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    ev[0].record(enum)
    long.enumerate(out, stream=enum)
    long.enumerate(out, stream=enum)
    ev[1].record(enum)
    side.wait_event(ev[0])
    other.rebuild(stream=side)
    ev[2].record(side)
    torch.cuda.synchronize()
    long.sync()
    other.sync()
    return ev[0].elapsed_time(ev[1]), ev[0].elapsed_time(ev[2])


@pytest.mark.parametrize("cap", [1, 2, 3])
@pytest.mark.parametrize("g,target,depths", [(WIDE, 200000000, (2, 3)), (WIDE, 400000, (2, 3)),
                                             ((5, 7, 11, 14), 20000000, (2,)), ((5, 8, 11, 14), 4000, (2, 3)),
                                             ((7, 10, 11, 19, 39), 2000000, (2, 3))])
def test_plan_rebuild_beside_a_capped_enumeration(fz, cap, g, target, depths):
    """Rebuilds of long and short count tables and of tables of depth 1 to 3
    (memo depths 2 and 3; each a tenth of the enumerations' time or less on its
    own, 0.02 to 0.15 of it beside them)."""
    n = workloads.find_n(fz.fz_count_upto, WIDE, 200000000)
    m = workloads.find_n(fz.fz_count_upto, g, target)
    with fz.Plan(WIDE, n, k=3) as long:
        out = torch.empty((long.count, 6), dtype=torch.int32, device="cuda")
        long.set_enum_ctas_per_sm(cap)
        for k in depths:
            with fz.Plan(g, m, k=k) as other:
                other.set_enum_ctas_per_sm(cap)
                _ends(long, other, out)
                enum, rebuild = min((_ends(long, other, out) for _ in range(3)), key=lambda x: x[1] / x[0])
                assert rebuild < 0.7 * enum, (k, enum, rebuild)


@pytest.mark.parametrize("cap", [1, 2, 3])
def test_batch_rebuild_beside_a_capped_enumeration(fz, cap):
    big = [(WIDE, workloads.find_n(fz.fz_count_upto, WIDE, 20000000))] * 10
    small = [((5, 8, 11, 14), 500), ((7, 10, 11, 19, 39), 700), ((9, 6, 12, 15, 21, 10), 300)] * 8
    with fz.Batch(big) as long, fz.Batch(small) as other:
        out = torch.empty(long.total_words, dtype=torch.int32, device="cuda")
        long.set_enum_ctas_per_sm(cap)
        other.set_enum_ctas_per_sm(cap)
        _ends(long, other, out)
        enum, rebuild = min((_ends(long, other, out) for _ in range(3)), key=lambda x: x[1] / x[0])
        assert rebuild < 0.7 * enum, (enum, rebuild)
