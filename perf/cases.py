"""The work that is timed when the library's speed is looked at: its operators, plans, batches and shared scans
over the sizes a user of it has, each through its public entry point.

* ``listed()``          the named cases; ``draw(rng)`` one more case of the same ranges;
* ``prepare(case, s)``  tables, queries, plans and output buffers on the GPU, made from the seed ``s``;
* ``run(state)``        one pass through the entry point; returns the output buffers (zero where nothing is written);
* ``work(case)``        the bytes a pass cannot do without: each input read once, each output written once;
* ``exact(case, s)``    what ``run`` returns, from plain torch in 64 bits.

Columns follow the repository's synthetic tables: fact rows (date i32 over 2557 days, discount i64 0..10, quantity
i32 1..50, price i64 100..10^7, flag u8 0..2, status u8 0..1), dimension rows (unique keys, an int32 payload), probe
rows (Zipf(0.5) foreign keys over the build keys, an int64 value) and string columns (one to three words of a
32-word vocabulary, 0-padded).
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_2203_01877_gb300 as tqp

DEV = "cuda:0"
DAYS = 2557
Q1_AGGS = [("sum", [("col", 3)]), ("sum", [("col", 4)]),
           ("sum", [("col", 4), ("const", 100), ("col", 5), "sub", "mul"]), ("count", None), ("avg", [("col", 4)])]
MINMAX_AGGS = [("min", [("col", 4)]), ("max", [("col", 4)]), ("count", None)]
REVENUE = [("col", 3), ("col", 1), "mul"]   # price * discount of (date, discount, quantity, price)
TOPK = 100


def listed():
    return [
        # an interactive query on a small table: one launch-bound call
        {"name": "filter_100K", "kind": "filter", "rows": 100_003, "wide": False, "ids": True},
        # the scan benchmark: a 365-day window, a discount band, a quantity cutoff (1.8% pass), row ids and a sum
        {"name": "filter_60M", "kind": "filter", "rows": 60_000_000, "wide": False, "ids": True},
        # the same columns under a predicate that nearly every row passes: the compaction writes as much as it reads
        {"name": "filter_wide_20M", "kind": "filter", "rows": 20_000_003, "wide": True, "ids": True},
        # the scan-aggregate report (six groups) on a small table
        {"name": "groupby_few_1M", "kind": "few", "rows": 1_000_000, "shape": "q1"},
        # the same report over a large resident table
        {"name": "groupby_few_200M", "kind": "few", "rows": 200_000_000, "shape": "q1"},
        # totals per customer: as many groups as a large key column has values
        {"name": "groupby_many_60M", "kind": "many", "rows": 60_000_000, "groups": 1_500_000},
        # a join materialised as index pairs, on keys scattered over the int32 range (a hashed build side)
        {"name": "join_pairs_60M", "kind": "pairs", "rows": 60_000_000, "build": 1_500_000, "dup": 1, "sparse": True,
         "join": "inner"},
        # the star-schema report: fact joined to a dimension with surrogate keys, 150K groups, the top 100
        {"name": "join_topk_60M", "kind": "topk", "rows": 60_000_000, "build": 1_500_000, "sparse": False},
        # a nightly batch: 512 queries of the three shapes over tables of uneven sizes, captured once and replayed
        {"name": "batch_512", "kind": "batch", "plans": 512, "low": 10_000, "high": 5_000_000, "mix": 3},
        # what a serving loop hands over at a time: 64 queries of the three shapes over ranges of a resident table
        {"name": "plans_64", "kind": "plans", "plans": 64, "rows": 60_000_000, "low": 10_000, "high": 5_000_000,
         "dim": 15_000_000, "mix": 4},
        # a dashboard: 32 filter queries over one table in shared passes
        {"name": "shared_32q_60M", "kind": "shared", "rows": 60_000_000, "queries": 32},
        # a text search: LIKE on a string column and a price bound, count and sum
        {"name": "strings_like_20M", "kind": "strings", "rows": 20_000_000, "width": 24, "pattern": "contains"},
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(math.exp(rng.uniform(math.log(lo), math.log(hi))))))


def draw(rng):
    kind = rng.choice(["filter", "few", "many", "pairs", "topk", "batch", "plans", "shared", "strings"])
    if kind == "filter":
        return {"kind": kind, "rows": _log_int(rng, 10_000, 60_000_000), "wide": rng.random() < 0.4,
                "ids": rng.random() < 0.75}
    if kind == "few":
        return {"kind": kind, "rows": _log_int(rng, 10_000, 200_000_000),
                "shape": rng.choice(["q1", "q1", "minmax", "ungrouped"])}
    if kind == "many":
        rows = _log_int(rng, 100_000, 60_000_000)
        return {"kind": kind, "rows": rows, "groups": _log_int(rng, 1_000, max(1_000, min(1_500_000, rows // 8)))}
    if kind == "pairs":
        rows = _log_int(rng, 100_000, 60_000_000)
        join = rng.choice(["inner", "inner", "inner", "semi", "anti", "left_outer"])
        dup = rng.choice([1, 1, 10]) if rows <= 6_000_000 else 1
        return {"kind": kind, "rows": rows, "build": _log_int(rng, 1_000, max(1_000, rows // 20)), "dup": dup,
                "sparse": rng.random() < 0.5, "join": join}
    if kind == "topk":
        rows = _log_int(rng, 100_000, 60_000_000)
        return {"kind": kind, "rows": rows, "build": _log_int(rng, 1_000, max(1_000, rows // 20)),
                "sparse": rng.random() < 0.4}
    if kind == "batch":
        return {"kind": kind, "plans": _log_int(rng, 8, 400), "low": 10_000,
                "high": _log_int(rng, 500_000, 5_000_000), "mix": rng.randrange(1 << 20)}
    if kind == "plans":
        return {"kind": kind, "plans": _log_int(rng, 4, 64), "rows": _log_int(rng, 6_000_000, 60_000_000),
                "low": 10_000, "high": _log_int(rng, 500_000, 5_000_000), "dim": _log_int(rng, 200_000, 15_000_000),
                "mix": rng.randrange(1 << 20)}
    if kind == "shared":
        return {"kind": kind, "rows": _log_int(rng, 1_000_000, 60_000_000), "queries": rng.randint(3, 48)}
    return {"kind": kind, "rows": _log_int(rng, 100_000, 20_000_000), "width": rng.choice([24, 24, 32, 27]),
            "pattern": rng.choice(["contains", "prefix", "suffix", "two", "in"])}


# ---- inputs --------------------------------------------------------------------------------------------------

def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed) * 1_000_003 + 20220301)


def _ints(g, n, lo, hi, dtype):
    """Uniform on [lo, hi]."""
    return torch.randint(lo, hi + 1, (n,), dtype=dtype, device=DEV, generator=g)


def _fact(g, n):
    return {"date": _ints(g, n, 0, DAYS - 1, torch.int32), "flag": _ints(g, n, 0, 2, torch.uint8),
            "status": _ints(g, n, 0, 1, torch.uint8), "quantity": _ints(g, n, 1, 50, torch.int32),
            "price": _ints(g, n, 100, 10_000_000, torch.int64), "discount": _ints(g, n, 0, 10, torch.int64)}


def _zipf(g, n, m):
    """n key indices of [0, m): Zipf(0.5) ranks, each rank's index drawn by a random permutation."""
    cdf = np.cumsum(np.arange(1, m + 1, dtype=np.float64) ** -0.5)
    cdf = torch.from_numpy(cdf / cdf[-1]).to(DEV)
    perm = torch.randperm(m, device=DEV, generator=g)
    out = torch.empty(n, dtype=torch.int64, device=DEV)
    for i in range(0, n, 1 << 25):
        u = torch.rand(min(1 << 25, n - i), dtype=torch.float64, device=DEV, generator=g)
        out[i:i + u.numel()] = perm[torch.searchsorted(cdf, u, right=True).clamp_(max=m - 1)]
    return out


def _keys(idx, sparse):
    """The int32 join key of a key index: itself, or scattered over [0, 2^31) (an odd multiplier: distinct)."""
    return ((idx * 1_000_003) & ((1 << 31) - 1) if sparse else idx).to(torch.int32)


def _dim(g, rows, groups, sparse=False, dup=1):
    key = _keys(torch.arange(rows, dtype=torch.int64, device=DEV) // dup, sparse)
    return key, (torch.randperm(rows, device=DEV, generator=g) % groups).to(torch.int32)


def _words(seed, width):
    """Every string of one to three vocabulary words, and the vocabulary."""
    rng = random.Random(seed)
    vocab = ["".join(rng.choice("abcdefghijklmnopqrstuvwxyz") for _ in range(rng.randint(3, 7))) for _ in range(32)]
    texts = list(vocab)
    texts += [a + " " + b for a in vocab for b in vocab]
    texts += [a + " " + b + " " + c for a in vocab for b in vocab for c in vocab]
    table = np.zeros((len(texts), width), np.uint8)
    for i, t in enumerate(texts):
        table[i, :len(t)] = np.frombuffer(t.encode(), np.uint8)
    return vocab, texts, torch.from_numpy(table).to(DEV)


def _like(pattern, vocab):
    """The string predicate of a case as (operator, operand) and as a function of one text."""
    w, v = vocab[0], vocab[1]
    if pattern == "prefix":
        return ("like", w[:2] + "%"), lambda t: t.startswith(w[:2])
    if pattern == "suffix":
        return ("like", "%" + w[-2:]), lambda t: t.endswith(w[-2:])
    if pattern == "two":
        def two(t):
            i = t.find(w[:2])
            return i >= 0 and t.find(v[:2], i + 2) >= 0
        return ("like", "%" + w[:2] + "%" + v[:2] + "%"), two
    if pattern == "in":
        some = set(vocab[:8])
        return ("in", sorted(some)), lambda t: t in some
    return ("like", "%" + w[:2] + "%"), lambda t: w[:2] in t


def _window(rng):
    """A filter query of the headline's form: (first day, lowest discount, quantity bound)."""
    return rng.randrange(0, DAYS - 365), rng.randint(0, 8), rng.randint(2, 50)


def _window_preds(w):
    return [(0, "ge", w[0]), (0, "lt", w[0] + 365), (1, "between", w[1], w[1] + 2), (2, "lt", w[2])]


Q6 = (731, 5, 24)


def _mix(case):
    """The shapes of a mix of plans: (kind, rows, first row) per plan; the same for every seed."""
    rng = random.Random(case["mix"])
    out = []
    for i in range(case["plans"]):
        n = _log_int(rng, case["low"], case["high"])
        first = rng.randrange(0, max(1, (case.get("rows", n) - n) // 16 + 1)) * 16
        out.append((("q1", "q6", "join")[i % 3], n, first))
    return out


# ---- state ---------------------------------------------------------------------------------------------------

_CTX = []


def _context():
    """The one context of the program: its scratch serves every call."""
    if not _CTX:
        _CTX.append(tqp.Context(0, 4 << 30))
    return _CTX[0]


def _z(n, dtype=torch.int64):
    return torch.zeros(max(int(n), 1), dtype=dtype, device=DEV)


def _q1_outputs():
    return {"keys": _z(128), "ivals": _z(320), "fvals": _z(320, torch.float64), "groups": _z(1)}


class _Slab:
    """Output slices of many plans out of a few tensors."""

    def __init__(self, ids, ints, floats):
        self.ids, self.ints, self.floats = _z(ids, torch.int32), _z(ints), _z(floats, torch.float64)
        self.at = {"ids": 0, "ints": 0, "floats": 0}

    def take(self, which, n):
        a = self.at[which]
        self.at[which] = a + n
        return getattr(self, which)[a:a + n]

    def out(self):
        return {"ids": self.ids, "ints": self.ints, "floats": self.floats}


Q1_INTS, Q6_INTS, JOIN_INTS = 128 + 320 + 3, 2, 3 * TOPK + 3


def _slab_for(mix):
    kinds = [k for k, _, _ in mix]
    return _Slab(sum(n for k, n, _ in mix if k == "q6"),
                 kinds.count("q1") * Q1_INTS + kinds.count("q6") * Q6_INTS + kinds.count("join") * JOIN_INTS,
                 kinds.count("q1") * 320)


def _plan(kind, fact, slab, dim=None, prepared=None):
    """A plan of one of the three shapes over `fact` and its result slices."""
    t = slab.take
    if kind == "q1":
        p = tqp.make_plan(fact, [(0, "le", 2450)], None, 0, 0, [1, 2], Q1_AGGS)
        r = tqp.make_result(None, 0, t("ints", 1), None, t("ints", 128), t("ints", 320), t("floats", 320), 64,
                            t("ints", 1), t("ints", 1), None)
    elif kind == "q6":
        p = tqp.make_plan(fact, _window_preds(Q6), sum_expr=REVENUE, emit_row_ids=True)
        n = fact.num_rows
        r = tqp.make_result(t("ids", n), n, t("ints", 1), t("ints", 1))
    else:
        p = tqp.make_plan(fact, (), dim, 0, 0, [3], [("sum", [("col", 1)]), ("count", None)], None, TOPK, 0,
                          prepared=prepared)
        r = tqp.make_result(None, 0, None, None, t("ints", TOPK), t("ints", 2 * TOPK), None, TOPK, t("ints", 1),
                            t("ints", 1), t("ints", 1))
    return p, r


def _mix_inputs(case, seed):
    """Per plan of a mix: its fact columns and, for a join of a batch, its dimension's columns."""
    g, mix = _gen(seed), _mix(case)
    if case["kind"] == "plans":   # ranges of one resident table; the joins share a prepared dimension
        f = _fact(g, case["rows"])
        f["key"] = _ints(g, case["rows"], 0, 99_999, torch.int32)
        dim = _dim(g, case["dim"], min(150_000, case["dim"]))
        cols = {"q1": ("date", "flag", "status", "quantity", "price", "discount"),
                "q6": ("date", "discount", "quantity", "price"), "join": ("key", "price")}
        return mix, [([f[c][r0:r0 + n] for c in cols[k]], dim if k == "join" else None) for k, n, r0 in mix]
    # every plan its own table, as slices that start on 16-row boundaries
    pad = lambda n: (n + 15) // 16 * 16  # noqa: E731
    f, at, out = _fact(g, sum(pad(n) for k, n, _ in mix if k != "join")), 0, []
    for k, n, _ in mix:
        if k == "join":
            nb = max(1000, n // 40)
            out.append(([_keys(_zipf(g, n, nb), False), _ints(g, n, 100, 10_000_000, torch.int64)],
                        _dim(g, nb, max(1, nb // 10))))
            continue
        names = ("date", "flag", "status", "quantity", "price", "discount") if k == "q1" else (
            "date", "discount", "quantity", "price")
        out.append(([f[c][at:at + n] for c in names], None))
        at += pad(n)
    return mix, out


def _few_columns(case, seed):
    f = _fact(_gen(seed), case["rows"])
    return [f[c] for c in ("date", "flag", "status", "quantity", "price", "discount")]


def _few_query(case):
    if case["shape"] == "minmax":
        return [1, 2], MINMAX_AGGS
    return ([1, 2] if case["shape"] == "q1" else []), Q1_AGGS


def _filter_columns(case, seed):
    f = _fact(_gen(seed), case["rows"])
    return [f[c] for c in ("date", "discount", "quantity", "price")]


def _filter_preds(case):
    return [(0, "le", 2450), (2, "ge", 1)] if case["wide"] else _window_preds(Q6)


def _many_columns(case, seed):
    g = _gen(seed)
    return [_zipf(g, case["rows"], case["groups"]).to(torch.int32), _ints(g, case["rows"], 100, 10_000_000, torch.int64)]


def _join_columns(case, seed):
    """Probe (key, value) and build (key, payload) columns."""
    g, dup = _gen(seed), case.get("dup", 1)
    m = (case["build"] + dup - 1) // dup
    probe = _zipf(g, case["rows"], m if case.get("join", "inner") == "inner" else m + m // 4)
    return ([_keys(probe, case["sparse"]), _ints(g, case["rows"], 100, 10_000_000, torch.int64)],
            _dim(g, case["build"], max(1, case["build"] // 10), case["sparse"], dup))


def _pairs_capacity(case):
    return case["rows"] * (case["dup"] if case["join"] in ("inner", "left_outer") else 1)


def _string_columns(case, seed):
    g = _gen(seed)
    vocab, texts, table = _words(seed, case["width"])
    n = case["rows"]
    k = _ints(g, n, 1, 3, torch.int64)
    a, b, c = (_ints(g, n, 0, 31, torch.int64) for _ in range(3))
    idx = torch.where(k == 1, a, torch.where(k == 2, 32 + a * 32 + b, 32 + 1024 + (a * 32 + b) * 32 + c))
    return vocab, texts, idx, table[idx], _ints(g, n, 100, 10_000_000, torch.int64)


def _windows(case, seed):
    rng = random.Random(seed)
    return [_window(rng) for _ in range(case["queries"])]


def prepare(case, seed):
    kind = case["kind"]
    s = {"kind": kind}
    if kind == "filter":
        cols = _filter_columns(case, seed)
        s.update(ctx=_context(), table=tqp.TableRef(cols), preds=_filter_preds(case), count=_z(1), sum=_z(1),
                 ids=_z(case["rows"], torch.int32) if case["ids"] else None)
    elif kind == "few":
        gc, aggs = _few_query(case)
        s.update(ctx=_context(), table=tqp.TableRef(_few_columns(case, seed)), group_cols=gc, aggs=aggs,
                 **_q1_outputs())
    elif kind == "many":
        m = case["groups"]
        s.update(ctx=_context(), table=tqp.TableRef(_many_columns(case, seed)), capacity=m, keys=_z(m),
                 ivals=_z(2 * m), groups=_z(1))
    elif kind == "pairs":
        probe, build = _join_columns(case, seed)
        cap = _pairs_capacity(case)
        s.update(ctx=_context(), probe=tqp.TableRef(probe), build=tqp.TableRef(build), join=case["join"],
                 capacity=cap, build_idx=_z(cap, torch.int32), probe_idx=_z(cap, torch.int32), count=_z(1))
    elif kind == "topk":
        probe, build = _join_columns(case, seed)
        fact, dim = tqp.TableRef(probe), tqp.TableRef(build)
        slab = _Slab(1, JOIN_INTS, 1)
        p, r = _plan("join", fact, slab, dim)
        s.update(ctx=_context(), plan=p, result=r, slab=slab)
    elif kind in ("batch", "plans"):
        mix, inputs = _mix_inputs(case, seed)
        slab = _slab_for(mix)
        ctx = tqp.Context(0, 4 << 30)
        dims = {}
        prepared = None
        plans, results = [], []
        for (k, _, _), (fact, dim) in zip(mix, inputs):
            D = None
            if dim is not None:
                D = dims.setdefault(id(dim), tqp.TableRef(list(dim)))
                if kind == "plans" and prepared is None:
                    prepared = tqp.tqp_dim_prepare(ctx, D, 0, [1], max_groups=min(150_000, case["dim"]))
            p, r = _plan(k, tqp.TableRef(fact), slab, D, prepared)
            plans.append(p)
            results.append(r)
        s.update(ctx=ctx, plans=plans, results=results, slab=slab, dims=dims, prepared=prepared)
        if kind == "batch":
            s["batch"] = tqp.tqp_batch_create(ctx, plans, results)
    elif kind == "shared":
        table = tqp.TableRef(_filter_columns(case, seed))
        m = case["queries"]
        counts, sums = _z(m), _z(m)
        queries = [(_window_preds(w), REVENUE, counts[i:i + 1], sums[i:i + 1])
                   for i, w in enumerate(_windows(case, seed))]
        s.update(ctx=_context(), table=table, queries=tqp.ScanQueries(queries, table), counts=counts, sums=sums)
    else:
        vocab, _, _, col, price = _string_columns(case, seed)
        (op, arg), _ = _like(case["pattern"], vocab)
        s.update(ctx=_context(), table=tqp.TableRef([col, price]), preds=[(0, op, arg), (1, "lt", 5_000_000)],
                 count=_z(1), sum=_z(1))
    return s


def run(s):
    kind = s["kind"]
    if kind == "filter":
        tqp.tqp_filter(s["ctx"], s["table"], s["preds"], REVENUE, s["sum"], s["ids"],
                       s["table"].num_rows if s["ids"] is not None else 0, s["count"])
        out = {"count": s["count"], "sum": s["sum"]}
        if s["ids"] is not None:
            out["ids"] = s["ids"]
        return out
    if kind == "few":
        tqp.tqp_groupby_agg(s["ctx"], s["table"], [(0, "le", 2450)], s["group_cols"], s["aggs"], s["keys"],
                            s["ivals"], s["fvals"], 64, s["groups"])
        return {k: s[k] for k in ("keys", "ivals", "fvals", "groups")}
    if kind == "many":
        tqp.tqp_groupby_agg(s["ctx"], s["table"], [], [0], [("sum", [("col", 1)]), ("count", None)], s["keys"],
                            s["ivals"], None, s["capacity"], s["groups"])
        return {k: s[k] for k in ("keys", "ivals", "groups")}
    if kind == "pairs":
        tqp.tqp_hash_join_kind(s["ctx"], s["build"], 0, s["probe"], 0, s["join"], s["build_idx"], s["probe_idx"],
                               s["capacity"], s["count"])
        return {k: s[k] for k in ("build_idx", "probe_idx", "count")}
    if kind == "topk":
        tqp.tqp_run_plan(s["ctx"], s["plan"], s["result"])
        return {"ints": s["slab"].ints}
    if kind == "batch":
        tqp.tqp_batch_run(s["batch"])
        return s["slab"].out()
    if kind == "plans":
        tqp.tqp_run_plans(s["ctx"], s["plans"], s["results"])
        return s["slab"].out()
    if kind == "shared":
        tqp.tqp_filter_shared(s["ctx"], s["table"], s["queries"])
        return {"counts": s["counts"], "sums": s["sums"]}
    tqp.tqp_filter(s["ctx"], s["table"], s["preds"], [("col", 1)], s["sum"], None, 0, s["count"])
    return {"count": s["count"], "sum": s["sum"]}


# ---- work ----------------------------------------------------------------------------------------------------

def _q6_bytes(n, ids=True):
    # the predicate columns of every row; per passing row (365 of 2557 days, 3 of 11 discounts, 23 of 50 quantities)
    # its price and its row id
    return 16 * n + n * (365 / DAYS) * (3 / 11) * (23 / 50) * (8 + (4 if ids else 0))


def work(case):
    kind, n = case["kind"], case.get("rows", 0)
    if kind == "filter":
        if case["wide"]:
            b = 24 * n + (n * (2451 / DAYS) * 4 if case["ids"] else 0)
        else:
            b = _q6_bytes(n, case["ids"])
    elif kind == "few":
        b = n * {"q1": 26, "minmax": 14, "ungrouped": 24}[case["shape"]]
    elif kind == "many":
        b = 12 * n + 24 * case["groups"]
    elif kind == "pairs":
        pairs = n * (case["dup"] if case["join"] == "inner" else 1)   # (the other kinds: about one per row at most)
        b = 4 * n + 4 * case["build"] + 8 * pairs
    elif kind == "topk":
        b = 12 * n + 8 * case["build"] + 8 * JOIN_INTS
    elif kind in ("batch", "plans"):
        b = 0
        for k, m, _ in _mix(case):
            b += 26 * m if k == "q1" else _q6_bytes(m) if k == "q6" else 12 * m
            if kind == "batch" and k == "join":
                b += 8 * max(1000, m // 40)
    elif kind == "shared":
        b = 24 * n
    else:
        b = n * (case["width"] + 8)
    return {"bytes": int(b), "flops": 0}


# ---- the same in plain torch ---------------------------------------------------------------------------------

def _padded(x, n):
    out = torch.zeros(n, dtype=x.dtype, device=x.device)
    out[:x.numel()] = x
    return out


def _exact_window(cols, w, price_disc=True):
    date, disc, qty, price = cols
    m = (date >= w[0]) & (date < w[0] + 365) & (disc >= w[1]) & (disc <= w[1] + 2) & (qty < w[2])
    ids = m.nonzero().flatten()
    return ids, (price[ids] * disc[ids]).sum()


def _exact_q1(cols, shape="q1"):
    """keys, ivals, fvals (64 groups, zero-padded) and the number of groups."""
    date, flag, status, qty, price, disc = cols
    m = date <= 2450
    gid = flag.to(torch.int64) * 2 + status if shape != "ungrouped" else torch.zeros_like(price)
    gid = gid[m]
    q, p, d = qty[m].to(torch.int64), price[m], disc[m]
    cnt = torch.bincount(gid, minlength=6)
    used = cnt.nonzero().flatten()
    add = lambda x: torch.zeros(6, dtype=torch.int64, device=DEV).scatter_add_(0, gid, x)[used]  # noqa: E731
    cnt = cnt[used]
    if shape == "minmax":
        red = lambda how: torch.zeros(6, dtype=torch.int64, device=DEV).scatter_reduce_(  # noqa: E731
            0, gid, p, how, include_self=False)[used]
        iv = torch.stack([red("amin"), red("amax"), cnt], 1)
        fv = torch.zeros_like(iv, dtype=torch.float64)
    else:
        sp = add(p)
        iv = torch.stack([add(q), sp, add(p * (100 - d)), cnt, sp], 1)
        fv = torch.zeros_like(iv, dtype=torch.float64)
        fv[:, 4] = sp.to(torch.float64) / cnt.to(torch.float64)
    keys = torch.stack([used // 2, used % 2], 1).flatten() if shape != "ungrouped" else used[:0]
    return _padded(keys, 128), _padded(iv.flatten(), 320), _padded(fv.flatten(), 320), used.numel()


def _exact_topk(fact, dim):
    """The integer outputs of a join plan: keys, ivals, groups, all groups, joined rows (dimension keys unique)."""
    (fk, val), (key, payload) = fact, dim
    order = torch.argsort(key)
    at = torch.searchsorted(key[order], fk).clamp_(max=key.numel() - 1)
    hit = key[order][at] == fk
    g = payload[order][at[hit]].to(torch.int64)
    m = int(payload.max()) + 1
    tot = torch.zeros(m, dtype=torch.int64, device=DEV).scatter_add_(0, g, val[hit])
    cnt = torch.bincount(g, minlength=m)
    used = cnt.nonzero().flatten()
    best = used[torch.argsort(-tot[used], stable=True)[:TOPK]]
    one = lambda v: torch.tensor([int(v)], dtype=torch.int64, device=DEV)  # noqa: E731
    return [_padded(best, TOPK), _padded(torch.stack([tot[best], cnt[best]], 1).flatten(), 2 * TOPK),
            one(best.numel()), one(used.numel()), one(hit.sum())]


def exact(case, seed):
    kind = case["kind"]
    one = lambda v: torch.tensor([int(v)], dtype=torch.int64, device=DEV)  # noqa: E731
    if kind == "filter":
        cols = _filter_columns(case, seed)
        if case["wide"]:
            ids = ((cols[0] <= 2450) & (cols[2] >= 1)).nonzero().flatten()
            total = (cols[3][ids] * cols[1][ids]).sum()
        else:
            ids, total = _exact_window(cols, Q6)
        out = {"count": one(ids.numel()), "sum": one(total)}
        if case["ids"]:
            out["ids"] = _padded(ids.to(torch.int32), case["rows"])
        return out
    if kind == "few":
        keys, iv, fv, m = _exact_q1(_few_columns(case, seed), case["shape"])
        return {"keys": keys, "ivals": iv, "fvals": fv, "groups": one(m)}
    if kind == "many":
        key, val = _many_columns(case, seed)
        m = case["groups"]
        cnt = torch.bincount(key, minlength=m)
        tot = torch.zeros(m, dtype=torch.int64, device=DEV).scatter_add_(0, key.to(torch.int64), val)
        used = cnt.nonzero().flatten()
        return {"keys": _padded(used, m), "ivals": _padded(torch.stack([tot[used], cnt[used]], 1).flatten(), 2 * m),
                "groups": one(used.numel())}
    if kind == "pairs":
        (fk, _), (key, _) = _join_columns(case, seed)
        order = torch.argsort(key, stable=True)
        ks = key[order]
        lo, hi = torch.searchsorted(ks, fk), torch.searchsorted(ks, fk, right=True)
        cnt, join = hi - lo, case["join"]
        if join in ("semi", "anti"):
            rows = ((cnt > 0) if join == "semi" else (cnt == 0)).nonzero().flatten()
            b = torch.full_like(rows, -1)
        else:
            n = cnt.clamp(min=1) if join == "left_outer" else cnt
            rows = torch.repeat_interleave(torch.arange(fk.numel(), device=DEV), n)
            k = torch.arange(rows.numel(), device=DEV) - (torch.cumsum(n, 0) - n)[rows]
            b = torch.where(cnt[rows] > 0, order[(lo[rows] + k).clamp_(max=key.numel() - 1)], -1)
        cap = _pairs_capacity(case)
        return {"build_idx": _padded(b.to(torch.int32), cap), "probe_idx": _padded(rows.to(torch.int32), cap),
                "count": one(rows.numel())}
    if kind == "topk":
        return {"ints": torch.cat(_exact_topk(*_join_columns(case, seed)))}
    if kind in ("batch", "plans"):
        mix, inputs = _mix_inputs(case, seed)
        ids, ints, floats = [torch.zeros(0, dtype=torch.int32, device=DEV)], [], []
        for (k, n, _), (cols, dim) in zip(mix, inputs):
            if k == "q1":
                keys, iv, fv, m = _exact_q1(cols)
                ints += [one((cols[0] <= 2450).sum()), keys, iv, one(m), one(m)]
                floats.append(fv)
            elif k == "q6":
                rows, total = _exact_window(cols, Q6)
                ids.append(_padded(rows.to(torch.int32), n))
                ints += [one(rows.numel()), one(total)]
            else:
                ints += _exact_topk(cols, dim)
        return {"ids": torch.cat(ids), "ints": torch.cat(ints), "floats": torch.cat(floats)}
    if kind == "shared":
        cols = _filter_columns(case, seed)
        found = [_exact_window(cols, w) for w in _windows(case, seed)]
        return {"counts": torch.cat([one(r.numel()) for r, _ in found]), "sums": torch.cat([one(t) for _, t in found])}
    vocab, texts, idx, _, price = _string_columns(case, seed)
    _, match = _like(case["pattern"], vocab)
    hit = torch.tensor([match(t) for t in texts], device=DEV)[idx] & (price < 5_000_000)
    return {"count": one(hit.sum()), "sum": one(price[hit].sum())}
