"""Random access by a warp a rank (few ranks) and by a thread a rank: both
sides of the line between them, with tables in run order, none, partial memos
and memos in element order, against the enumeration."""
import pytest

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


# (generators, target rows, k, top)
PLANS = [((53, 71, 91, 115, 176, 195), 20000, -1, -1), ((53, 71, 91, 115, 176, 195), 20000, 3, -1),
         ((53, 71, 91, 115, 176, 195), 20000, 0, -1), ((53, 71, 91, 115, 176, 195), 20000, 3, 300),
         ((5, 8, 11, 14), 9000, 2, -1), ((5, 8, 11, 14), 9000, 1, -1), ((5, 8, 11, 14), 9000, 3, 40),
         ((3, 7), 9000, 0, -1), ((7, 3), 9000, 1, -1), ((500, 3, 7), 9000, -1, -1),
         ((13, 17, 19, 23, 29, 31, 37, 41, 43, 44), 20000, 4, -1), ((13, 17, 19, 23, 29, 31, 37, 41, 43, 44), 20000, 5, 60),
         (tuple(range(20, 36)), 20000, -1, -1), (tuple(range(20, 36)), 20000, 0, -1)]


@pytest.mark.parametrize("g,target,k,top", PLANS)
def test_numbers_of_ranks(fz, g, target, k, top):
    n = workloads.find_n(fz.fz_count_upto, g, target, 256)
    d = len(g)
    with fz.Plan(g, n, k=k, top=top) as plan:
        rows = torch.empty((plan.count, d), dtype=torch.int32, device="cuda")
        plan.enumerate(rows)
        gen = torch.Generator(device="cuda").manual_seed(5)
        ends = torch.tensor([0, plan.count - 1], device="cuda")
        for m in (1, 2, 3, 31, 33, 1000, 6144, 6145, 8192, 8193, 20001):
            ranks = torch.cat([ends, torch.randint(0, plan.count, (m,), generator=gen, device="cuda")])[:m]
            out = torch.full((m + 3, d), CANARY, dtype=torch.int32, device="cuda")
            plan.unrank(ranks, out[:m])
            plan.sync()
            assert torch.equal(out[:m], rows[ranks]), m
            assert bool((out[m:] == CANARY).all()), m


@pytest.mark.parametrize("m", [5, 9000])
def test_rank_past_the_last(fz, m):
    """A rank past the last: its row is -1, the others' are right, and the
    plan's next synchronisation says so, once."""
    g, n = (5, 8, 11, 14), 700
    for k in (0, 2, 3):
        with fz.Plan(g, n, k=k) as plan:
            rows = torch.empty((plan.count, 4), dtype=torch.int32, device="cuda")
            plan.enumerate(rows)
            ranks = torch.arange(m, device="cuda") % plan.count
            ranks[3] = plan.count
            out = torch.full((m, 4), CANARY, dtype=torch.int32, device="cuda")
            plan.unrank(ranks, out)
            with pytest.raises(fz.FzError):
                plan.sync()
            plan.sync()
            ok = torch.arange(m, device="cuda") != 3
            assert bool((out[3] == -1).all()) and torch.equal(out[ok], rows[ranks[ok]])
