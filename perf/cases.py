"""The work that a user of this library has it do, as cases that can be timed.

Each case is one kind of call with its sizes.  ``prepare`` draws the inputs
from a seed (generator sets and elements whose output has about the asked
number of rows) and makes what a user's program holds before the call: output
tensors, plans, batches, servers.  ``run`` is one pass through the public
calls.  All outputs are whole numbers (int32 tuples, 64-bit counts).
"""
import math
import random

import numpy as np
import torch

import paper_2407_20474_gb300 as fz


def listed():
    return [
        # Counting before anything else: |Z(r)| for every r <= n on the host, as
        # a program does that looks for the element with a wanted number of
        # rows, or admits queries by their exact size.
        {"name": "counts", "kind": "counts", "d": 6, "lo": 50, "hi": 200, "n": 39064},
        # The whole counting table in device memory for a long range of elements
        # (the widest tables a batch of d = 3 instances needs have millions of
        # entries a row).
        {"name": "count_table", "kind": "table", "d": 4, "lo": 2, "hi": 300, "n": 2000003},
        # The smallest call: one element with a few thousand factorizations,
        # one-shot, memo depth 2 (generators of the size of (5, 8, 11, 14)).
        {"name": "oneshot_small", "kind": "oneshot", "d": 4, "lo": 5, "hi": 14, "rows": 3800, "k": 2},
        # One element delivered into page-locked host memory, plan and all.
        {"name": "host_mid", "kind": "host", "d": 5, "lo": 10, "hi": 60, "rows": 1000000},
        # The large element: count table, memo and 5e8 rows (12 GB) a pass with a
        # resident plan.
        {"name": "plan_large", "kind": "plan", "d": 6, "lo": 50, "hi": 200, "rows": 500000000, "k": -1},
        # Wide tuples of close generators (the paper's own runtime table goes to
        # d = 9 with generators 13..45 and memo depth 4).
        {"name": "plan_wide", "kind": "plan", "d": 9, "lo": 13, "hi": 45, "rows": 14000000, "k": -1},
        # The plain walk without a memo, the paper's baseline method.
        {"name": "plan_plain", "kind": "plan", "d": 6, "lo": 50, "hi": 200, "rows": 10000001, "k": 0},
        # The tabulation on its own: every Z(r), r < top, as one CSR.
        {"name": "memo", "kind": "memo", "d": 5, "lo": 3, "hi": 40, "rows": 36000000},
        # Thousands of uneven instances in one batch, rebuilt and enumerated.
        {"name": "batch", "kind": "batch", "count": 4096, "d_lo": 3, "d_hi": 8, "lo": 2, "hi": 300,
         "t_lo": 100, "t_hi": 1000000},
        # A batch of few and small instances, where launches count.
        {"name": "batch_small", "kind": "batch", "count": 96, "d_lo": 3, "d_hi": 8, "lo": 2, "hi": 300,
         "t_lo": 100, "t_hi": 10000},
        # A burst of queries to a server with resident sets; every result is
        # copied out and released.
        {"name": "serve", "kind": "serve", "sets": 16, "requests": 64, "d_lo": 4, "d_hi": 7, "lo": 5,
         "hi": 500, "t_lo": 1000, "t_hi": 10000000},
        # Random access: the tuples of given ranks (sampling without enumerating).
        {"name": "unrank", "kind": "unrank", "d": 6, "lo": 50, "hi": 200, "rows": 100000000,
         "ranks": 1000003, "k": -1},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["counts", "table", "oneshot", "host", "plan", "plan", "plain", "memo", "batch",
                       "batch", "serve", "unrank"])
    if kind == "counts":
        return {"kind": kind, "d": rng.randint(3, 6), "lo": 20, "hi": 300, "n": _log(rng, 500, 200000)}
    if kind == "table":
        return {"kind": kind, "d": rng.randint(3, 5), "lo": 20, "hi": 300, "n": _log(rng, 2000, 1000000)}
    if kind == "oneshot":
        return {"kind": kind, "d": rng.randint(3, 8), "lo": 5, "hi": 60, "rows": _log(rng, 500, 2000000),
                "k": rng.choice([-1, -1, 2])}
    if kind == "host":
        return {"kind": kind, "d": rng.randint(4, 8), "lo": 10, "hi": 60, "rows": _log(rng, 10000, 4000000)}
    if kind == "plan":
        return {"kind": kind, "d": rng.randint(3, 9), "lo": 13, "hi": rng.choice([45, 100, 200]),
                "rows": _log(rng, 50000, 200000000), "k": -1}
    if kind == "plain":
        return {"kind": "plan", "d": rng.randint(4, 7), "lo": 13, "hi": 200, "rows": _log(rng, 50000, 10000000),
                "k": 0}
    if kind == "memo":
        return {"kind": kind, "d": rng.randint(3, 6), "lo": 3, "hi": rng.choice([40, 100]),
                "rows": _log(rng, 100000, 36000000)}
    if kind == "batch":
        return {"kind": kind, "count": _log(rng, 16, 3000), "d_lo": 3, "d_hi": rng.randint(4, 8), "lo": 2,
                "hi": 300, "t_lo": 100, "t_hi": _log(rng, 5000, 1000000)}
    if kind == "serve":
        return {"kind": kind, "sets": rng.randint(4, 24), "requests": rng.randint(8, 96), "d_lo": 4, "d_hi": 7,
                "lo": 5, "hi": 500, "t_lo": 1000, "t_hi": _log(rng, 10000, 5000000)}
    return {"kind": kind, "d": rng.randint(4, 8), "lo": 13, "hi": 200, "rows": _log(rng, 100000, 100000000),
            "ranks": _log(rng, 1000, 1000000), "k": -1}


def _gens(rng, d, lo, hi):
    """d distinct generators of [lo, hi], ascending, with gcd 1."""
    while True:
        g = sorted(rng.sample(range(lo, hi + 1), d))
        if math.gcd(*g) == 1:
            return tuple(g)


def _element(g, rows):
    """An n with about `rows` factorizations: |Z(n)| is about
    (n + sum(g) / 2)^(d-1) / ((d-1)! prod(g))."""
    d = len(g)
    x = rows * math.factorial(d - 1) * math.prod(g)
    return max(g[-1], int(round(x ** (1.0 / (d - 1)) - sum(g) / 2)))


def _memo_top(g, rows):
    """A top with about `rows` rows in all Z(r), r < top."""
    d = len(g)
    x = rows * math.factorial(d) * math.prod(g)
    return max(g[-1], int(round(x ** (1.0 / d) - sum(g) / 2)))


def _shapes(case):
    """The widths and wanted sizes of a batch's instances or a burst's
    requests: the same for every seed, which draws the generators."""
    rng = random.Random(12)
    count = case["count"] if case["kind"] == "batch" else case["sets"]
    d = [rng.randint(case["d_lo"], case["d_hi"]) for _ in range(count)]
    if case["kind"] == "batch":
        return [(i, d[i], _log(rng, case["t_lo"], case["t_hi"])) for i in range(count)]
    asked = [rng.randrange(count) for _ in range(case["requests"])]
    return [(i, d[i], _log(rng, case["t_lo"], case["t_hi"])) for i in asked]


def _room(shapes):
    """Words that hold the rows of all shapes (sizes come out near the wanted
    ones; the buffer's unused end stays zero)."""
    return sum(d * (t + t // 4 + 256) for _, d, t in shapes)


def _fitting(g, rows):
    """The element next below the estimate with at most `rows` factorizations."""
    n = _element(g, rows)
    while n > 0 and fz.fz_count(g, n) > rows:
        n -= max(1, n // 1000)
    return n


def prepare(case, seed):
    """Output buffers have the size the case names, whatever the seed draws:
    a program's own buffers, of which a call fills as much as it needs."""
    rng = random.Random(int(seed))
    kind = case["kind"]
    st = {"kind": kind}
    if kind in ("batch", "serve"):
        shapes = _shapes(case)
        sets = {i: _gens(rng, d, case["lo"], case["hi"]) for i, d in sorted({(i, d) for i, d, _ in shapes})}
        asked = [(i, _element(sets[i], t)) for i, _, t in shapes]
        st["out"] = torch.zeros(_room(shapes), dtype=torch.int32, device="cuda")
        if kind == "batch":
            st["batch"] = fz.Batch([(sets[i], n) for i, n in asked])
            return st
        words, off = [], 0
        for i, n in asked:
            w = fz.fz_count(sets[i], n) * len(sets[i])
            words.append((off, w))
            off += w
        srv = fz.Server(memory_bytes=4 * off + (64 << 20))
        ids = {i: srv.register(g, max(n for j, n in asked if j == i)) for i, g in sets.items()}
        st.update(server=srv, asked=[(ids[i], n) for i, n in asked], words=words)
        return st
    d = case["d"]
    g = _gens(rng, d, case["lo"], case["hi"])
    st.update(g=g, k=case.get("k", fz.FZ_AUTO))
    if kind in ("counts", "table"):
        st["n"] = case["n"]
        if kind == "table":
            st["out"] = torch.zeros((d + 1, case["n"] + 1), dtype=torch.int64, device="cuda")
    elif kind == "memo":
        top = _memo_top(g, case["rows"])
        while fz.fz_memo_rows(g, top) > case["rows"]:
            top -= max(1, top // 1000)
        widest = _memo_top(range(case["hi"] - d + 1, case["hi"] + 1), case["rows"])
        st.update(top=top, offsets=torch.zeros(widest + 1, dtype=torch.int64, device="cuda"),
                  out=torch.zeros((case["rows"], d), dtype=torch.int32, device="cuda"))
    elif kind == "unrank":
        st["plan"] = fz.Plan(g, _element(g, case["rows"]), k=st["k"])
        gen = torch.Generator(device="cuda").manual_seed(int(seed))
        st["ranks"] = torch.randint(0, st["plan"].count, (case["ranks"],), generator=gen, device="cuda")
        st["out"] = torch.zeros((case["ranks"], d), dtype=torch.int32, device="cuda")
    else:
        st["n"] = _fitting(g, case["rows"])
        st["out"] = torch.zeros((case["rows"], d), dtype=torch.int32, pin_memory=kind == "host",
                                device="cpu" if kind == "host" else "cuda")
        if kind == "plan":
            st["plan"] = fz.Plan(g, st["n"], k=st["k"])
    return st


def run(st):
    kind = st["kind"]
    if kind == "counts":
        return fz.fz_count_upto(st["g"], st["n"]).view(np.int64)
    if kind == "table":
        fz.fz_count_table(st["g"], st["n"], st["out"])
    elif kind == "memo":
        fz.fz_build_memo_into(st["g"], st["top"], st["offsets"], st["out"], len(st["out"]))
        return st["offsets"], st["out"]
    elif kind == "batch":
        st["batch"].rebuild()
        st["batch"].enumerate(st["out"])
    elif kind == "serve":
        srv, out = st["server"], st["out"]
        tickets = [srv.submit(s, n) for s, n in st["asked"]]
        for t, (off, w) in zip(tickets, st["words"]):
            srv.wait(t)
            srv.copy(t, out[off:off + w])
            srv.release(t)
    elif kind == "oneshot":
        fz.fz_enumerate(st["g"], st["n"], st["out"], k=st["k"])
    elif kind == "host":
        fz.fz_enumerate_host(st["g"], st["n"], st["out"], k=st["k"])
    elif kind == "plan":
        st["plan"].rebuild()
        st["plan"].enumerate(st["out"])
    else:
        st["plan"].unrank(st["ranks"], st["out"])
    return st["out"]


def work(case):
    """Bytes: every output written once (the inputs are a few generators; the
    ranks of random access are read once).  flops: integer additions of the
    counting recurrence where the counts are the result, one per entry."""
    kind = case["kind"]
    if kind == "counts":
        return {"bytes": 8.0 * (case["n"] + 1), "flops": float(case["d"]) * (case["n"] + 1)}
    if kind == "table":
        e = float(case["d"] + 1) * (case["n"] + 1)
        return {"bytes": 8.0 * e, "flops": e}
    if kind in ("batch", "serve"):
        return {"bytes": 4.0 * sum(d * t for _, d, t in _shapes(case)), "flops": 0.0}
    if kind == "unrank":
        return {"bytes": case["ranks"] * (8.0 + 4.0 * case["d"]), "flops": 0.0}
    return {"bytes": 4.0 * case["rows"] * case["d"], "flops": 0.0}


def _table(g, n):
    """Rows 0..d of |Z(r, (g_{j+1}, ..., g_d))|, r = 0..n, in 64-bit integers."""
    rows = [np.zeros(n + 1, dtype=np.int64)]
    rows[0][0] = 1
    for v in reversed(g):
        pad = -(n + 1) % v
        x = np.concatenate([rows[-1], np.zeros(pad, dtype=np.int64)]).reshape(-1, v)
        rows.append(np.cumsum(x, axis=0).reshape(-1)[:n + 1])
    return rows[::-1]


def _walk(g, n):
    """All factorizations of n in descending lexicographic order."""
    d, C = len(g), _table(g, n)
    cols, rem = [], np.array([n], dtype=np.int64)
    for j in range(d - 1):
        top = rem // g[j]
        first = np.cumsum(top + 1) - (top + 1)
        src = np.repeat(np.arange(len(rem)), top + 1)
        a = top[src] - (np.arange(len(src)) - first[src])
        left = rem[src] - a * g[j]
        live = C[j + 1][left] > 0
        src, a, rem = src[live], a[live], left[live]
        cols = [c[src] for c in cols] + [a]
    return np.stack(cols + [rem // g[-1]], axis=1).astype(np.int32)


def exact(case, seed):
    """The counts (64-bit recurrence) and the sets small enough to be walked
    here; the larger lists have no other plain form that is quick enough."""
    kind = case["kind"]
    if kind not in ("counts", "table", "oneshot", "host") or case.get("rows", 0) > 100000:
        return None
    g = _gens(random.Random(int(seed)), case["d"], case["lo"], case["hi"])
    if kind == "counts":
        return _table(g, case["n"])[0]
    if kind == "table":
        return np.stack(_table(g, case["n"]))
    n = _element(g, case["rows"])
    while n > 0 and _table(g, n)[0][n] > case["rows"]:
        n -= max(1, n // 1000)
    rows = _walk(g, n)
    return np.concatenate([rows, np.zeros((case["rows"] - len(rows), len(g)), dtype=np.int32)])
