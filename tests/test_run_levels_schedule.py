"""The memo built by run-order levels, restated on the CPU with the index
formulas of the kernels (fz_runs.cu, fz_walk.cuh) and compared with the
oracle's memo: class starts, flat element index -> (class, step), the leaf of
a row (the last start at or before it), one contiguous range per element, and
the closed form of the last two generators.  Generator orders, repeats,
common factors, generators above the last element."""
import math

import numpy as np
import pytest

import oracle


def _pair(g, h):
    e = math.gcd(g, h)
    h1, g1 = h // e, g // e
    inv = pow(g1, -1, h1) if h1 > 1 else 0
    return e, h1, g1, inv


def _element_at(f, n, g):
    """Flat index of the class order -> (class, step)."""
    qn, rr = divmod(n, g)
    lim = (rr + 1) * (qn + 1)
    if f < lim:
        return f // (qn + 1), f % (qn + 1)
    return rr + 1 + (f - lim) // qn, (f - lim) % qn


def _levels(t, top, rows_a_warp=7):
    """Offsets and rows of Z(m, t), m < top, by the chain; every table row is
    written through its warp's window and leaf search."""
    k, n = len(t), top - 1
    C = oracle.count_table(t, n)          # C[j][r] = |Z(r, (t_j..))|
    C = [[int(x) for x in row] for row in C]
    table = cls_src = None
    for j in range(k - 3, -1, -1):
        K, g = k - 1 - j, t[j]
        G = min(g, n + 1)
        cls = [0]
        for c in range(G):
            cls.append(cls[-1] + C[j][c + (n - c) // g * g])
        rows = cls[-1]
        assert rows == sum(C[j + 1])
        leaves = []                        # (end, p, step)
        for f in range(n + 1):
            c, s = _element_at(f, n, g)
            p = c + s * g
            assert 0 <= p <= n
            leaves.append((cls[c] + C[j][p], p, s))
        assert sorted(p for _, p, _ in leaves) == list(range(n + 1))
        out = [None] * rows
        ends = [e for e, _, _ in leaves]
        assert ends == sorted(ends)
        for row0 in range(0, rows, rows_a_warp):
            for row in range(row0, min(rows, row0 + rows_a_warp)):
                leaf = int(np.searchsorted(ends, row, side="right"))
                end, p, s = leaves[leaf]
                start = leaves[leaf - 1][0] if leaf else 0
                o = row - start
                if K == 2:
                    e, h1, g1, inv = _pair(t[j + 1], t[j + 2])
                    q = p // t[j + 1]
                    at = q - (q - (p // e) % h1 * inv % h1) % h1
                    b0 = (p - at * t[j + 1]) // t[j + 2]
                    body = [at - o * h1, b0 + o * g1]
                else:
                    gl = t[j + 1]
                    r = table[cls_src[p % gl] + o]
                    body = [p // gl - r[0]] + r[1:]
                out[row] = [s] + body
        table, cls_src = out, cls
    off, res = [0], []
    for m in range(top):
        cnt = C[0][m]
        src = cls_src[m % t[0]]
        for o in range(cnt):
            r = table[src + o]
            res.append([m // t[0] - r[0]] + r[1:])
        off.append(off[-1] + cnt)
    return off, res


@pytest.mark.parametrize("t,top", [((4, 9, 10), 90), ((10, 4, 9), 77), ((3, 5, 7, 8), 60), ((2, 2, 3), 40),
                                   ((6, 10, 15), 130), ((1, 2, 3), 25), ((5, 1, 4), 33),
                                   ((50, 3, 4, 5), 45), ((3, 90, 4, 5), 45), ((4, 6, 8), 61),
                                   ((7, 5, 6, 4, 9), 48), ((3, 4, 4, 4, 5, 6), 30), ((4, 9, 10), 1),
                                   ((7, 3, 5), 2)])
def test_levels_match_the_oracle(t, top):
    off, rows = _levels(t, top)
    ref_off, ref_rows = oracle.memo_csr(t, top)
    assert off == [int(x) for x in ref_off]
    assert rows == ref_rows.tolist()
