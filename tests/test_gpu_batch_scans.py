"""The batched scans' shapes at their limits: rows of 7, 8, 31 and 32 residue
chains of 127 to 129 and 255 to 257 entries, read from memory and computed
(width 3), against the oracle's counts and rows."""
import numpy as np
import pytest

import oracle

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


@pytest.mark.parametrize("chains", [7, 8, 31, 32])
@pytest.mark.parametrize("length", [127, 128, 129, 255, 256, 257])
def test_short_chains(fz, chains, length):
    inst = [(g, n) for n in (chains * length - 1, chains * length)
            for g in ((5, chains, 41, 60), (chains, 45, 58), (9, chains, chains, 77, 80))]
    _, rows = fz.fz_plan_batch(inst)
    assert [int(r) for r in rows] == [oracle.count(g, n) for g, n in inst]


@pytest.mark.parametrize("chains", [7, 31, 32])
def test_rows_of_short_chains(fz, chains):
    """Every row, partial memos included (their tables are scanned for the walk)."""
    inst = [(g, chains * 128) for g in ((90, chains, 151, 260), (chains, 145, 158), (79, 200, chains, 277, 180))]
    for top in (-1, 40):
        with fz.Batch(inst, top=top) as b:
            out = torch.full((b.total_words + 8,), CANARY, dtype=torch.int32, device="cuda")
            b.rebuild()
            b.enumerate(out)
            b.sync()
            host = out.cpu().numpy()
            assert (host[b.total_words:] == CANARY).all()
            for j, (g, n) in enumerate(inst):
                ref, at = oracle.enumerate_desc(g, n), int(b.word_offsets[j])
                assert np.array_equal(host[at:at + ref.size].reshape(ref.shape), ref), (g, n, top)
