"""Enumeration and random access of elements next to 2^31, where a coordinate's
next multiple of its generator no longer fits 32 bits: the flat walk over the
closed form of the last two generators (windows of a dense set), and the rank
walk and searches of a sparse one."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N = 2**31 - 2
CANARY = -7


@pytest.fixture(scope="module")
def fz():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2407_20474_gb300 as m
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    torch.cuda.set_device(0)
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    if free < 200 << 30:
        pytest.skip("needs 200 GB of device memory")
    return m


def test_windows_of_a_dense_set(fz):
    g = (500000009, 700000001, 3, 2)
    first, blocks = 0, []  # (first rank, a_1, a_2, remainder) of every prefix
    for a in range(N // g[0], -1, -1):
        for b in range((N - a * g[0]) // g[1], -1, -1):
            p = N - a * g[0] - b * g[1]
            top = p // 3 - (p // 3 - p) % 2  # the greatest a_3 of p's parity
            blocks.append((first, a, b, p, top))
            first += top // 2 + 1
    with fz.Plan(g, N, k=0) as plan:
        assert plan.count == first
        for f, a, b, p, top in blocks + [(first, 0, 0, 0, 0)]:
            lo, hi = max(0, f - 40000), min(first, f + 40000)
            out = torch.full((hi - lo + 2, 4), CANARY, dtype=torch.int32, device="cuda")
            assert plan.enumerate(out, lo, hi) == hi - lo
            plan.sync()
            got = out.cpu().numpy()
            assert (got[hi - lo:] == CANARY).all()
            ref = []
            for f2, a2, b2, p2, top2 in blocks:
                r = np.arange(max(lo, f2), min(hi, f2 + top2 // 2 + 1), dtype=np.int64) - f2
                c = top2 - 2 * r
                ref.append(np.stack([np.full_like(c, a2), np.full_like(c, b2), c, (p2 - 3 * c) // 2], axis=1))
            assert np.array_equal(got[:hi - lo], np.concatenate(ref).astype(np.int32)), (a, b)


def test_sparse_set(fz):
    g = (500000009, 300000007, 200000003, 3)
    ref = oracle.enumerate_desc(g, N)
    with fz.Plan(g, N, k=0) as plan:
        assert plan.count == len(ref) > 20
        out = torch.full((len(ref) + 2, 4), CANARY, dtype=torch.int32, device="cuda")
        plan.enumerate(out)
        ranks = torch.arange(len(ref), device="cuda").repeat(1 + 9000 // len(ref))
        for m in (len(ref), len(ranks)):
            pick = torch.full((m, 4), CANARY, dtype=torch.int32, device="cuda")
            plan.unrank(ranks[:m], pick)
            assert np.array_equal(pick.cpu().numpy(), ref[ranks[:m].cpu().numpy()]), m
        plan.sync()
        assert np.array_equal(out.cpu().numpy()[:len(ref)], ref)
        assert bool((out[len(ref):] == CANARY).all())
