"""Plans, memos and batches made by several threads at once, each on its own
stream beside a busy one: the descriptions of every table's levels reach the
device as they were written (each thread's stack and heap are reused at once)."""
import threading

import numpy as np
import pytest

import oracle
from paper_2407_20474_gb300 import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SETS = [((5, 8, 11, 14), 3000, (1, 2, 3)), ((9, 6, 12, 15, 21, 10), 9000, (2, 3, 4)), ((7, 10, 11, 19, 39), 6000, (3, 2, -1)),
        ((13, 4, 7, 30, 22, 9, 17), 9000, (5, 4, 3)), ((3, 5, 7, 9, 11, 13, 4, 6), 9000, (6, 5, 4)),
        ((400, 7, 3, 5), 2000, (2, 3, -1))]


@pytest.fixture(scope="module")
def fz():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2407_20474_gb300 as m
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    torch.cuda.set_device(0)
    return m


def test_many_threads(fz):
    busy = torch.cuda.Stream()
    big = torch.empty(1 << 28, dtype=torch.int32, device="cuda")
    sets = [(g, workloads.find_n(oracle.count_upto, g, t), ks) for g, t, ks in SETS]
    refs = [oracle.enumerate_desc(g, n) for g, n, _ in sets]
    memos = [oracle.memo_csr(g[1:], 60) for g, _, _ in sets]
    errors = []

    def work(i):
        try:
            g, n, ks = sets[i]
            ref, (off, rows) = refs[i], memos[i]
            stream = torch.cuda.Stream()
            out = torch.empty(ref.shape, dtype=torch.int32, device="cuda")
            o = torch.empty(61, dtype=torch.int64, device="cuda")
            r = torch.empty(rows.shape, dtype=torch.int32, device="cuda")
            stream.wait_stream(torch.cuda.default_stream())
            for rep in range(12):
                with fz.Plan(g, n, k=ks[rep % 3], stream=stream) as plan:
                    plan.enumerate(out, stream=stream)
                    plan.sync(stream=stream)
                    stream.synchronize()
                    assert np.array_equal(out.cpu().numpy(), ref), (g, n, rep)
                fz.fz_build_memo_into(g[1:], 60, o, r, len(rows), stream=stream)
                stream.synchronize()
                assert np.array_equal(o.cpu().numpy().view(np.uint64), off), (g, rep)
                assert np.array_equal(r.cpu().numpy(), rows), (g, rep)
                with fz.Batch([(g, n), (g, n // 2)], stream=stream) as b:
                    assert int(b.rows[0]) == len(ref)
        except Exception as e:  # reported by the main thread
            errors.append(e)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(sets))]
    for t in threads:
        t.start()
    with torch.cuda.stream(busy):
        while any(t.is_alive() for t in threads):
            for _ in range(20):
                big.add_(1)
            busy.synchronize()
    for t in threads:
        t.join()
    assert not errors, errors[0]
