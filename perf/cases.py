"""The work that users of the hash table have it do, as cases that can be timed.

Every case runs public calls of the package only.  Keys are distinct 64-bit
words of a SplitMix64-like stream of the seed; values are key * 3, and counts
are sums of ones.  All outputs are whole numbers with exactly one right answer:
where the library leaves a choice open (which of several equal keys of a batch
reports "inserted", the order of an export) the case does not ask for it, and
so no floating-point reference exists for any output.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_1601_04017_gb300 as cht

ADD, OVERWRITE = cht.ADD, cht.OVERWRITE
CELL = 16  # bytes of a cell

# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------


def _s64(x):
    x &= (1 << 64) - 1
    return x - (1 << 64) if x >> 63 else x


def _mix(x):
    """A bijection of 64-bit words (Stafford's variant 13 of the SplitMix64 finalizer)."""
    x = x ^ ((x >> 30) & ((1 << 34) - 1))
    x = x * _s64(0xBF58476D1CE4E5B9)
    x = x ^ ((x >> 27) & ((1 << 37) - 1))
    x = x * _s64(0x94D049BB133111EB)
    return x ^ ((x >> 31) & ((1 << 33) - 1))


def _keys(seed, first, count):
    """Words first + 1 ... first + count of the seed's stream: distinct, and neither 0 nor ~0 in any range used here."""
    i = torch.arange(first + 1, first + count + 1, dtype=torch.int64, device="cuda")
    k = _mix(i * _s64(0x9E3779B97F4A7C15) + _s64((seed * 2 + 1) * 0xD1342543DE82EF95))
    return torch.where((k == 0) | (k == -1), torch.full_like(k, 0x1234567), k)


def _uniform(seed, count):
    """Doubles in [0, 1)."""
    return ((_keys(seed ^ 0x5EED, 1 << 40, count) >> 11) & ((1 << 53) - 1)).to(torch.float64) * 2.0 ** -53


def _below(seed, count, n):
    """Whole numbers drawn uniformly from 0 ... n - 1."""
    return (_uniform(seed, count) * n).to(torch.int64).clamp_(0, n - 1)


def _zipf(seed, count, s, n):
    """Ranks 0 ... n - 1 of about Zipf(s) frequencies (inverse of the continuous distribution function)."""
    u = _uniform(seed, count)
    if abs(s - 1.0) < 1e-6:
        x = torch.exp(u * math.log(n + 1.0))
    else:
        x = (u * ((n + 1.0) ** (1.0 - s) - 1.0) + 1.0) ** (1.0 / (1.0 - s))
    return x.to(torch.int64).sub_(1).clamp_(0, n - 1)


def _probes(seed, keys_seed, live, count, hit):
    """`count` keys to look up: a share `hit` of them drawn from the first `live` keys of the stream, the others absent, mixed."""
    present = _keys(keys_seed, 0, live)[_below(seed + 1, count, live)]
    absent = _keys(keys_seed, 1 << 34, count)
    return torch.where(_uniform(seed + 2, count) < hit, present, absent)


def _codes(n, **kw):
    return torch.empty(n, dtype=torch.uint8, **(kw or {"device": "cuda"}))


def _words(n, **kw):
    return torch.empty(n, dtype=torch.int64, **(kw or {"device": "cuda"}))


def _cap(n, load=0.5):
    return max(64, 1 << math.ceil(math.log2(max(n, 1) / load)))


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------


def listed():
    return [
        # a hash join or a per-frame table: the table is cleared, the build
        # side inserted and the probe side looked up.  A request's worth of
        # rows (three launches: latency) ...
        {"name": "join_small", "kind": "join", "n": 1000, "probes": 1000, "cap": 1 << 11},
        # ... the paper's small table, which stays in the L2 cache ...
        {"name": "join_l2", "kind": "join", "n": 1 << 19, "probes": (1 << 19) - 3, "cap": 1 << 20},
        # ... and a table far larger than it.
        {"name": "join_large", "kind": "join", "n": (1 << 26) - 12345, "probes": (1 << 26) + 777, "cap": 1 << 27},
        # lookups in a resident table (an index, a cache directory), half of
        # them present, at the load a growable table keeps ...
        {"name": "lookup_half", "kind": "lookup", "cap": 1 << 26, "load": 0.5, "n": (1 << 25) + 77, "hit": 0.5},
        # ... and in a bounded table filled to 0.9, where probes are long.
        {"name": "lookup_dense", "kind": "lookup", "cap": 1 << 25, "load": 0.9, "n": (1 << 24) - 5, "hit": 0.5},
        # lookups of a program whose keys and results are in pinned host memory
        {"name": "lookup_host", "kind": "host", "cap": 1 << 24, "load": 0.4, "n": (1 << 24) + (1 << 22) + 9, "hit": 0.7},
        # counting words or events of a log: mildly skewed keys (mostly
        # distinct cells) and heavily skewed ones (few hot cells)
        {"name": "count_flat", "kind": "count", "n": 1 << 26, "vocab": 1 << 24, "s": 0.5, "cap": 1 << 25},
        {"name": "count_skewed", "kind": "count", "n": (1 << 26) + 1001, "vocab": 1 << 24, "s": 1.25, "cap": 1 << 25},
        # loading a table in bulk (an index build, with some rows repeated),
        # then merging a day's changes into it; the finished cells are what
        # such a program writes out
        {"name": "bulk", "kind": "bulk", "n": (1 << 25) - 31, "repeat": 0.125, "delta": (1 << 22) + 5, "cap": 1 << 26},
        # a stream with a sliding window: a growable table begins small,
        # grows, and then takes a batch in and drops the oldest one each
        # round, purging tombstones as they pile up
        {"name": "stream", "kind": "stream", "live": 1 << 22, "batch": (1 << 18) - 7, "rounds": 32, "cap": 1 << 12},
        # many small to middling tables and many uneven batches in one launch
        {"name": "plan", "kind": "plan", "tables": 256, "log2_min": 10, "log2_max": 20, "rounds": 24},
        # requests against resident tables through the serving loop
        {"name": "serve", "kind": "serve", "tables": 64, "log2_min": 10, "log2_max": 20, "requests": 4000, "size_log2": 14},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    kind = rng.choice(["join", "join", "lookup", "lookup", "host", "count", "count", "bulk", "stream", "plan", "serve"])
    if kind == "join":
        n = _log(rng, 700, (1 << 26) - 12345)
        return {"kind": kind, "n": n, "probes": max(1, int(n * rng.uniform(0.5, 1.0))), "cap": _cap(n)}
    if kind == "lookup":
        cap = 1 << rng.randint(14, 26)
        return {"kind": kind, "cap": cap, "load": round(rng.uniform(0.2, 0.9 if cap <= 1 << 25 else 0.6), 3),
                "n": _log(rng, 1000, min((1 << 25) + 77, cap)), "hit": round(rng.uniform(0.2, 1.0), 2)}
    if kind == "host":
        cap = 1 << rng.randint(18, 24)
        return {"kind": kind, "cap": cap, "load": round(rng.uniform(0.2, 0.5), 3),
                "n": _log(rng, 1 << 16, (1 << 24) + (1 << 22)), "hit": round(rng.uniform(0.3, 1.0), 2)}
    if kind == "count":
        n = _log(rng, 1 << 16, 1 << 26)
        vocab = max(64, n // rng.choice([4, 8, 16]))
        return {"kind": kind, "n": n, "vocab": vocab, "s": round(rng.uniform(0.5, 1.5), 2), "cap": _cap(vocab)}
    if kind == "bulk":
        n = _log(rng, 1 << 14, (1 << 25) - 31)
        delta = max(1, int(n * rng.uniform(0.01, 0.12)))
        return {"kind": kind, "n": n, "repeat": round(rng.uniform(0.0, 0.5), 3), "delta": delta, "cap": _cap(n + delta, 0.75)}
    if kind == "stream":
        live = _log(rng, 1 << 14, 1 << 22)
        return {"kind": kind, "live": live, "batch": max(64, live // rng.choice([16, 24, 40])), "rounds": rng.randint(16, 32), "cap": 1 << 12}
    if kind == "plan":
        lo = rng.randint(8, 12)
        return {"kind": kind, "tables": rng.randint(16, 256), "log2_min": lo, "log2_max": rng.randint(lo + 2, 20), "rounds": rng.randint(6, 24)}
    lo = rng.randint(9, 12)
    return {"kind": kind, "tables": rng.randint(8, 64), "log2_min": lo, "log2_max": rng.randint(lo + 2, 20),
            "requests": _log(rng, 200, 4000), "size_log2": rng.randint(9, 14)}


# ---------------------------------------------------------------------------
# what a program has in hand, and one pass
# ---------------------------------------------------------------------------


def _filled(seed, cap, load):
    live = int(cap * load)
    k = _keys(seed, 0, live)
    t = cht.Table(cap)
    t.insert(k, k * 3)
    return t, live


def _prepare_join(c, seed):
    k = _keys(seed, 0, c["n"])
    return {"table": cht.Table(c["cap"]), "keys": k, "vals": k * 3, "codes": _codes(c["n"]),
            "probes": _probes(seed, seed, c["n"], c["probes"], 0.5), "out": _words(c["probes"]), "found": _codes(c["probes"])}


def _run_join(c, s):
    t = s["table"]
    t.clear()
    t.insert(s["keys"], s["vals"], s["codes"])
    t.find(s["probes"], s["out"], s["found"])
    return [s["codes"], s["out"], s["found"]]


def _work_join(c):
    return CELL * c["cap"] + 17 * c["n"] + c["probes"] * (8 + 9) + CELL * min(c["probes"], c["cap"])


def _prepare_lookup(c, seed):
    t, live = _filled(seed, c["cap"], c["load"])
    return {"table": t, "probes": _probes(seed, seed, live, c["n"], c["hit"]), "out": _words(c["n"]), "found": _codes(c["n"])}


def _run_lookup(c, s):
    s["table"].find(s["probes"], s["out"], s["found"])
    return [s["out"], s["found"]]


def _work_lookup(c):
    return c["n"] * (8 + 9) + CELL * min(c["n"], c["cap"])


def _prepare_host(c, seed):
    t, live = _filled(seed, c["cap"], c["load"])
    p = _probes(seed, seed, live, c["n"], c["hit"]).cpu().pin_memory()
    pin = {"pin_memory": True}
    return {"table": t, "probes": p, "out": _words(c["n"], **pin), "found": _codes(c["n"], **pin)}


def _run_host(c, s):
    s["table"].find(s["probes"], s["out"], s["found"])
    torch.cuda.current_stream().synchronize()  # results in host memory are valid once the stream is done
    return [s["out"], s["found"]]


def _prepare_count(c, seed):
    words = _keys(seed, 0, c["vocab"])
    order = _below(seed + 5, 1, 1 << 20)  # which words are the frequent ones
    ranks = (_zipf(seed + 3, c["n"], c["s"], c["vocab"]) + order) % c["vocab"]
    return {"table": cht.Table(c["cap"]), "log": words[ranks], "ones": torch.ones(c["n"], dtype=torch.int64, device="cuda"),
            "words": words, "counts": _words(c["vocab"]), "seen": _codes(c["vocab"])}


def _run_count(c, s):
    t = s["table"]
    t.clear()
    t.insert_or_update(s["log"], s["ones"], ADD)
    t.find(s["words"], s["counts"], s["seen"])
    return [s["counts"], s["seen"]]


def _work_count(c):
    return CELL * c["cap"] + 16 * c["n"] + c["vocab"] * (8 + 9 + CELL)


def _prepare_bulk(c, seed):
    distinct = max(1, int(c["n"] * (1.0 - c["repeat"])))
    k = _keys(seed, 0, c["n"])
    again = _uniform(seed + 1, c["n"]) < c["repeat"]
    k = torch.where(again, _keys(seed, 0, distinct)[_below(seed + 2, c["n"], distinct)], k)
    d = _keys(seed, 0, c["n"])[_below(seed + 3, c["delta"], c["n"])]  # half of the changes are to rows that exist
    d = torch.where(_uniform(seed + 4, c["delta"]) < 0.5, d, _keys(seed, 1 << 34, c["delta"]))
    return {"table": cht.Table(c["cap"]), "keys": k, "vals": _keys(seed + 9, 0, c["n"]), "dkeys": d, "dvals": _keys(seed + 10, 0, c["delta"])}


def _run_bulk(c, s):
    t = s["table"]
    t.clear()
    t.build(s["keys"], s["vals"])
    t.merge(s["dkeys"], s["dvals"])
    return t.cells()


def _work_bulk(c):
    # the rows in, the built cells out; the cells and the changes in, the merged cells out; their copy
    return 16 * c["n"] + CELL * c["cap"] + 16 * c["delta"] + 2 * CELL * c["cap"] + 2 * CELL * c["cap"]


def _prepare_stream(c, seed):
    total = c["live"] + c["batch"] * c["rounds"]
    k = _keys(seed, 0, total)
    return {"keys": k, "vals": k * 3, "ins": _codes(total), "era": _codes(c["batch"] * c["rounds"]),
            "probes": _probes(seed, seed, total, c["live"], 0.9), "out": _words(c["live"]), "found": _codes(c["live"])}


def _run_stream(c, s):
    live, b = c["live"], c["batch"]
    t = cht.Table(c["cap"], growable=True)
    t.insert(s["keys"][:live], s["vals"][:live], s["ins"][:live])
    for r in range(c["rounds"]):
        new = slice(live + r * b, live + (r + 1) * b)
        old = slice(r * b, (r + 1) * b)
        t.insert(s["keys"][new], s["vals"][new], s["ins"][new])
        t.erase(s["keys"][old], s["era"][old])
    t.find(s["probes"], s["out"], s["found"])
    t.destroy()
    return [s["ins"], s["era"], s["out"], s["found"]]


def _work_stream(c):
    total = c["live"] + c["batch"] * c["rounds"]
    # each key in and its code out, its cell written; each erased key's cell changed; the final lookups
    return total * (17 + CELL) + c["batch"] * c["rounds"] * (9 + CELL) + c["live"] * (17 + CELL)


def _sizes(rng, lo, hi, n):
    return [int(2.0 ** rng.uniform(lo, hi)) for _ in range(n)]


def _resident(seed, tables, universe, config=None, growable=False):
    """Tables that hold the first half of their universe of keys each; the universes are parts of one stream."""
    starts, made, at = [], [], 0
    for n in universe:
        starts.append(at)
        at += n
    every = _keys(seed, 0, at)
    for a, n in zip(starts, universe):
        t = cht.Table(_cap(n), growable=growable, config=config)
        half = every[a:a + n // 2]
        t.insert(half, half * 3)
        made.append(t)
    return made, every, starts


def _batch_of(rng, n, most):
    """(first, size) of a run of distinct keys in a universe of n, the size spread over its logarithm."""
    size = max(1, min(n, int(math.exp(rng.uniform(0.0, math.log(most + 1.0))))))
    return rng.randrange(n - size + 1), size


# shares of find, insert, insert-or-add, insert-or-overwrite, update-add
_PLAN_MIX = [(cht.OP_FIND, 0.5), (cht.OP_INSERT, 0.1), (cht.OP_IOU_ADD, 0.2), (cht.OP_IOU_OVERWRITE, 0.1), (cht.OP_UPDATE_ADD, 0.1)]
# of find, insert, insert-or-add, erase
_SERVE_MIX = [(cht.OP_FIND, 0.5), (cht.OP_INSERT, 0.3), (cht.OP_IOU_ADD, 0.15), (cht.OP_ERASE, 0.05)]


def _pick(rng, mix):
    u = rng.random()
    for op, share in mix:
        u -= share
        if u < 0:
            return op
    return mix[0][0]


def _plan_batches(c):
    """[(table, op, first, size)], round by round; the same for every seed, so that work() needs none."""
    rng = random.Random(c["tables"] * 1009 + c["log2_max"] * 31 + c["rounds"])
    universe = _sizes(rng, c["log2_min"], c["log2_max"], c["tables"])
    return universe, [(t, _pick(rng, _PLAN_MIX)) + _batch_of(rng, n, n // 4) for _ in range(c["rounds"]) for t, n in enumerate(universe)]


def _arrays(seed, every, starts, batches):
    """Flat keys, values, found values and codes of the batches, and each one's place in them."""
    sizes = torch.tensor([b[3] for b in batches], dtype=torch.int64, device="cuda")
    first = torch.tensor([starts[b[0]] + b[2] for b in batches], dtype=torch.int64, device="cuda")
    ends = torch.cumsum(sizes, 0)
    total = int(ends[-1])
    at = torch.arange(total, dtype=torch.int64, device="cuda") - torch.repeat_interleave(ends - sizes, sizes)
    keys = every[torch.repeat_interleave(first, sizes) + at]
    return {"keys": keys, "vals": _keys(seed + 7, 0, total), "out": torch.zeros(total, dtype=torch.int64, device="cuda"),
            "codes": torch.zeros(total, dtype=torch.uint8, device="cuda")}, np.concatenate([[0], ends.cpu().numpy()]).tolist()


def _prepare_plan(c, seed):
    universe, batches = _plan_batches(c)
    tables, every, starts = _resident(seed, c["tables"], universe)
    a, ends = _arrays(seed, every, starts, batches)
    ops = []
    for i, (t, op, _, _) in enumerate(batches):
        lo, hi = ends[i], ends[i + 1]
        vals = None if op == cht.OP_FIND else a["vals"][lo:hi]
        ops.append((tables[t], op, a["keys"][lo:hi], vals, a["out"][lo:hi] if op == cht.OP_FIND else None, a["codes"][lo:hi]))
    return {"plan": cht.Plan(ops), "tables": tables, **a}


def _run_plan(c, s):
    s["plan"].launch()
    return [s["out"], s["codes"]]


def _work_ops(batches):
    """Keys, values in or found values out, codes, and a cell read (and written, where it changes) for each operation."""
    total = 0
    for _, op, _, n in batches:
        total += n * (8 + 1 + CELL) + (0 if op == cht.OP_ERASE else 8 * n) + (0 if op == cht.OP_FIND else CELL * n)
    return total


def _work_plan(c):
    return _work_ops(_plan_batches(c)[1])


def _serve_batches(c):
    rng = random.Random(c["tables"] * 2003 + c["log2_max"] * 37 + c["requests"])
    universe = _sizes(rng, c["log2_min"], c["log2_max"], c["tables"])
    weights = [1.0 / (r + 1) for r in range(c["tables"])]  # some tables are asked more often than others
    got = []
    for t in rng.choices(range(c["tables"]), weights, k=c["requests"]):
        got.append((t, _pick(rng, _SERVE_MIX)) + _batch_of(rng, universe[t], 1 << c["size_log2"]))
    return universe, got


def _prepare_serve(c, seed):
    universe, batches = _serve_batches(c)
    tables, every, starts = _resident(seed, c["tables"], universe, {"reuse_tombstones": 1}, growable=True)
    a, ends = _arrays(seed, every, starts, batches)
    server = cht.Server(tables, arena_bytes=1 << 24, max_inflight_steps=2, max_step_requests=1024, max_step_ops=1 << 22)
    reqs = []
    for i, (t, op, _, _) in enumerate(batches):
        lo, hi = ends[i], ends[i + 1]
        vals = a["vals"][lo:hi] if op in (cht.OP_INSERT, cht.OP_IOU_ADD) else None
        reqs.append(cht.Server.request(t, op, a["keys"][lo:hi], vals, a["out"][lo:hi] if op == cht.OP_FIND else None, a["codes"][lo:hi]))
    return {"server": server, "tables": tables, "requests": reqs, "arrivals": np.zeros(len(reqs)), **a}


def _run_serve(c, s):
    s["server"].replay(s["requests"], s["arrivals"])
    return [s["out"], s["codes"]]


def _work_serve(c):
    return _work_ops(_serve_batches(c)[1])


_PREPARE = {"join": _prepare_join, "lookup": _prepare_lookup, "host": _prepare_host, "count": _prepare_count, "bulk": _prepare_bulk,
            "stream": _prepare_stream, "plan": _prepare_plan, "serve": _prepare_serve}
_RUN = {"join": _run_join, "lookup": _run_lookup, "host": _run_host, "count": _run_count, "bulk": _run_bulk,
        "stream": _run_stream, "plan": _run_plan, "serve": _run_serve}
_WORK = {"join": _work_join, "lookup": _work_lookup, "host": _work_lookup, "count": _work_count, "bulk": _work_bulk,
         "stream": _work_stream, "plan": _work_plan, "serve": _work_serve}


def prepare(case, seed):
    s = _PREPARE[case["kind"]](case, seed)
    s["case"] = case
    torch.cuda.synchronize()
    return s


def run(state):
    return _RUN[state["case"]["kind"]](state["case"], state)


def work(case):
    return {"bytes": _WORK[case["kind"]](case), "flops": 0}
