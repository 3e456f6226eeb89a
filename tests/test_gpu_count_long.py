"""Count tables of the longest elements: every residue chain of a scanned row
is written, also where a row has more than 2^20 - 16 tiles of 8 chains."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fz():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2407_20474_gb300 as m
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    torch.cuda.set_device(0)
    return m


def test_every_chain_of_the_longest_rows(fz):
    """n = 2^31 - 2, g_1 = 8388600: the last chains of row 0 against sums of
    row 1 (closed form), every entry written."""
    g, n = (8388600, 5, 3), 2**31 - 2
    need = 4 * 8 * (n + 1) + (4 << 30)
    free, _ = torch.cuda.mem_get_info()
    if free < need:
        pytest.skip("needs %d GB of device memory" % (need >> 30))
    T = torch.full((4, n + 1), -7, dtype=torch.int64, device="cuda")
    fz.fz_count_table(g, n, T)
    torch.cuda.synchronize()
    assert int(T.min()) >= 0
    c = g[0]
    for lo in (0, c - 200):  # the first and the last classes
        acc = torch.zeros(200, dtype=torch.int64, device="cuda")
        for a in range(lo, n + 1, c):
            b = min(a + 200, n + 1)
            acc[:b - a] += T[1, a:b]
            assert torch.equal(T[0, a:b], acc[:b - a]), a
    del T
    torch.cuda.empty_cache()
