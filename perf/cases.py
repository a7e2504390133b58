"""Timed cases of the query path, through the public binding (tid.h's calls).

One case is one call (or one short run of calls) that a program using the
library makes, with the inputs it has in hand: a resident triple store, index
lists, bound tuple sets, prepared patterns and plans.  Stores are the
university recipe of ``synth`` (20 predicates, typed subjects, entity- and
literal-valued objects) drawn on the device; operator inputs are tuple sets of
the sizes those stores give.  A seed gives the entities other IDs (within their
class) and the triples another order, and leaves the graph's shape, so a case's
results have the same number of rows for every seed.  Every input is int32 and
so is every result: ``exact`` has nothing to add to whole numbers.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1807_01409_gb300 import binding as tb
from paper_1807_01409_gb300 import synth

X, Y, Z, V = 0, 1, 2, 3
FULL = 200_000_000  # triples of the full university store


def listed():
    return [
        # the smallest request: one subject's triples from a 1M-triple store, rows on the host
        {"name": "lookup_1m", "call": "lookup", "n": 1_000_000, "shape": "s"},
        # eight single-pattern searches (two of each of (s,?,?), (?,p,?), (?,?,o), (?,p,o)) of the
        # full store, their index lists left on the device
        {"name": "scan_200m", "call": "scan", "n": FULL, "patterns": 8},
        # the subqueries of one star query searched in one pass: (?x type C), (?x p ?v), (?x p ?y)
        {"name": "multi_200m", "call": "multi", "n": FULL, "patterns": 3},
        # a subquery's result vector with its FILTER: 24M triples of a literal-valued predicate,
        # half of them in the value range
        {"name": "bind_filter_200m", "call": "bind", "n": FULL, "keep": 0.5},
        # operators on a large result vector (x, v): FILTER, and SELECT DISTINCT ?v ?x (a sort)
        {"name": "filter_project_24m", "call": "rows", "rows": 24_000_000, "digits": 4},
        # star join (x) with (x, y): the typed subjects against an entity-valued predicate
        {"name": "join_star_8m", "call": "join", "left": 500_000, "right": 8_200_000, "how": "star"},
        # chain join (x, y) with (y, z): the shared term is an object on one side and a subject on the other
        {"name": "join_chain_8m", "call": "join", "left": 8_000_000, "right": 8_000_000, "how": "chain"},
        # union of two branches with different variables, (x, v) and (x, y)
        {"name": "union_32m", "call": "union", "left": 23_600_000, "right": 8_200_000},
        # whole queries (two star joins, two chains, two unions, two filters) on a small store,
        # rows on the host: latency
        {"name": "plans_1m", "call": "plans", "n": 1_000_000, "host": True},
        # the same query classes on the full store, rows left on the device
        {"name": "plans_200m", "call": "plans", "n": FULL, "host": False},
        # the six RDFS rules over the full store and its schema
        {"name": "entail_200m", "call": "entail", "n": FULL},
        # many single-pattern queries of all seven shapes answered together
        {"name": "batch_200m", "call": "batch", "n": FULL, "queries": 512, "most": 100_000},
    ]


def _size(rng, lo, hi):
    """Log-uniform on [lo, hi], any remainder."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["lookup", "scan", "multi", "bind", "rows", "join", "join", "union", "plans", "entail", "batch"])
    if call == "lookup":
        return {"call": call, "n": _size(rng, 20_000, 20_000_000), "shape": rng.choice(["s", "sp", "po", "o"])}
    if call == "scan":
        return {"call": call, "n": _size(rng, 1_000_000, FULL), "patterns": rng.choice([1, 4, 8])}
    if call == "multi":
        return {"call": call, "n": _size(rng, 1_000_000, FULL), "patterns": rng.randint(2, 16)}
    if call == "bind":
        return {"call": call, "n": _size(rng, 200_000, FULL), "keep": round(rng.uniform(0.02, 1.0), 2)}
    if call == "rows":
        return {"call": call, "rows": _size(rng, 2_000, 24_000_000), "digits": rng.randint(2, 7)}
    if call == "join":
        how = rng.choice(["star", "chain", "inner2", "optional", "full"])
        return {"call": call, "left": _size(rng, 2_000, 8_000_000), "right": _size(rng, 2_000, 8_200_000), "how": how}
    if call == "union":
        return {"call": call, "left": _size(rng, 2_000, 24_000_000), "right": _size(rng, 2_000, 8_200_000)}
    if call == "plans":
        n = _size(rng, 200_000, FULL)
        return {"call": call, "n": n, "host": n < 10_000_000}
    if call == "entail":
        return {"call": call, "n": _size(rng, 200_000, FULL)}
    return {"call": call, "n": _size(rng, 1_000_000, FULL), "queries": _size(rng, 17, 1024), "most": _size(rng, 1_000, 100_000)}


# ---------------------------------------------------------------------------
# handles
# ---------------------------------------------------------------------------

class _Ctx:
    """The program's one context, on a torch stream."""
    handle = None

    @classmethod
    def get(cls):
        if cls.handle is None:
            torch.cuda.init()
            cls.stream = torch.cuda.Stream()
            cls.handle = tb.tid_ctx_create(0, cls.stream.cuda_stream)
        return cls.handle


class _Set:
    """A tuple set, freed with the last reference; its columns as CUDA tensors."""

    def __init__(self, h):
        self.h = h

    def __del__(self):
        tb.tid_set_free(self.h)

    def columns(self):
        rows = tb.tid_set_rows(self.h)
        info = tb.tid_set_info(self.h)
        return [_Column(self, p, rows).tensor() for p in info["dev_cols"]]


class _Column:
    def __init__(self, owner, ptr, rows):
        self.owner, self.rows = owner, rows
        self.__cuda_array_interface__ = {"shape": (rows,), "typestr": "<i4", "data": (ptr, False), "version": 2}

    def tensor(self):
        if self.rows == 0:
            return torch.empty(0, dtype=torch.int32, device="cuda")
        return torch.as_tensor(self, device="cuda")


class _Store:
    """A store borrowing three device columns."""

    def __init__(self, s, p, o):
        self.cols = (s, p, o)
        torch.cuda.synchronize()
        self.h = tb.tid_load(_Ctx.get(), s, p, o, copy=0)

    def __del__(self):
        torch.cuda.synchronize()
        tb.tid_store_free(self.h)


def _host(h):
    s = _Set(h)
    return tb.tid_set_to_host(s.h)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

SHAPE_SEED = 1807  # of what a seed leaves alone


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _layout(n):
    return synth.uni_layout(synth.uni_subjects(n))


def _renaming(sizes, seed):
    """New IDs of the entities 1..sum(sizes), each within its block: table[id]."""
    g = _gen(SHAPE_SEED + 1 + seed)
    parts, at = [torch.zeros(1, dtype=torch.int64, device="cuda")], 1
    for k in sizes:
        parts.append(torch.randperm(int(k), generator=g, device="cuda") + at)
        at += int(k)
    return torch.cat(parts).int()


def _renamed(c, table):
    return torch.where(c < table.shape[0], table[c.clamp(max=table.shape[0] - 1)], c)


def _shuffled(cols, seed):
    order = torch.randperm(cols[0].shape[0], generator=_gen(SHAPE_SEED - 1 - seed), device="cuda")
    return [c[order] for c in cols]


def _pairs(rows, subjects, g, values):
    """`rows` distinct (subject, value) pairs in random order: subjects uniform, values(m) drawn."""
    def some(m):
        s = torch.randint(1, subjects + 1, (m,), generator=g, device="cuda")
        return (s << 31) | values(m)
    keys = torch.unique(some(int(rows * 1.1) + 1024))
    while keys.shape[0] < rows:
        keys = torch.unique(torch.cat([keys, some(rows)]))
    keys = keys[torch.randperm(keys.shape[0], generator=g, device="cuda")[:rows]]
    return (keys >> 31).int(), (keys & 0x7FFFFFFF).int()


def _entities(subjects, g):
    cdf = torch.as_tensor(synth.zipf_cdf(1.1, subjects), device="cuda")
    perm = torch.randperm(subjects, generator=g, device="cuda") + 1

    def values(m):
        u = torch.rand(m, generator=g, device="cuda", dtype=torch.float64)
        return perm[torch.searchsorted(cdf, u, right=True).clamp_(max=subjects - 1)]
    return values


def _literals(digits, g):
    return lambda m: synth.LIT_BASE + torch.randint(0, 10 ** digits, (m,), generator=g, device="cuda")


def _result_vector(s, o, var, table, seed):
    """The result vector of (?, p, ?) over the triples (s, p, o), renamed and shuffled: variables var of
    the s and o slots (-1: anonymous)."""
    ctx = _Ctx.get()
    s, o = _shuffled([_renamed(s, table), _renamed(o, table)], seed)
    st = _Store(s, torch.full_like(s, 1), o)
    idx = _Set(tb.tid_match(ctx, st.h, (0, 1, 0)))
    out = _Set(tb.tid_bind(ctx, st.h, synth.Pattern(0, 1, 0, var=(var[0], -1, var[1])), idx.h))
    tb.tid_ctx_sync(ctx)
    return out


def _subjects_of(rows):
    return max(64, rows * 5 // 8)


def _scan_patterns(cols, n, m, table, hrng):
    """m patterns cycling through (s,?,?), (?,p,?), (?,p,o), (?,?,o), keyed from stored triples but for
    the predicates, which run through the store's frequencies."""
    s, p, o = cols
    pid = _layout(n)["pred_ids"]
    out = []
    for i in range(m):
        r = int(hrng.integers(0, n))
        t = [int(s[r]), int(p[r]), int(o[r])]
        t[0], t[2] = (int(_renamed(torch.tensor([x], device="cuda"), table)) for x in (t[0], t[2]))
        kind = i % 4
        if kind == 0:
            out.append(synth.Pattern(t[0], 0, 0, var=(-1, Y, Z)))
        elif kind == 1:
            out.append(synth.Pattern(0, int(pid[(1, 9, 4, 14)[i // 4 % 4]]), 0, var=(X, -1, Y)))
        elif kind == 2:
            out.append(synth.Pattern(0, t[1], t[2], var=(X, -1, -1)))
        else:
            out.append(synth.Pattern(0, 0, t[2], var=(X, Y, -1)))
    return out


def _plans(cols, n, table, hrng):
    """Two plans of each class of the multi-pattern workload: star joins on a typed subject, chains
    through object-subject joins, unions over one subject, and literal-range filters."""
    s, p, o = cols
    lay = _layout(n)
    pid = [int(x) for x in lay["pred_ids"]]
    P = synth.Pattern

    def typed(k):  # (?x type C), C one of the frequent (sub)classes of top class k
        return {"op": "match", "pattern": P(0, pid[0], int(lay["class_base"]) + k * synth.SUBCLASSES + int(hrng.integers(0, 6)),
                                            var=(X, -1, -1))}

    def prop(j, a, b):
        return {"op": "match", "pattern": P(0, pid[j], 0, var=(a, -1, b))}
    plans = []
    for k, js in ((0, (7, 11)), (1, (6, 2, 19))):  # star: property patterns on the same subject
        nodes = [typed(k)] + [prop(j, X, 4 + t) for t, j in enumerate(js)]
        cur = 0
        for r in range(1, len(js) + 1):
            nodes.append({"op": "join", "inputs": [cur, r], "algo": "auto"})
            cur = len(nodes) - 1
        if k:
            nodes.append({"op": "project", "input": cur, "vars": [X, 4]})
        plans.append(nodes)
    for k, a, b in ((0, 4, 8), (2, 12, 13)):  # chain: (?x type C), (?x pa ?y), (?y pb ?z)
        plans.append([typed(k), prop(a, X, Y), prop(b, Y, Z), {"op": "join", "inputs": [0, 1], "algo": "auto"},
                      {"op": "join", "inputs": [3, 2], "algo": "auto"}, {"op": "project", "input": 4, "vars": [X, Z]}])
    for _ in range(2):  # union: values of some predicates of one subject
        s0 = int(s[int(hrng.integers(0, n))])
        own = torch.unique(p[s == s0]).cpu().numpy()
        js = [int(x) for x in hrng.choice(own, size=min(3, len(own)), replace=False)] + [pid[1]]
        plans.append([{"op": "match", "pattern": P(int(table[s0]), j, 0, var=(-1, -1, Y))} for j in js]
                     + [{"op": "union", "inputs": list(range(len(js)))}])
    for i, (j, digits, k) in enumerate(((3, 7, 2), (5, 5, 1))):  # filter, the second joined with a type
        lo = int(hrng.integers(0, 10 ** digits // 2))
        nodes = [prop(j, X, Y), {"op": "filter", "input": 0, "var": Y, "cmp": "range", "a": synth.LIT_BASE + lo,
                                 "b": synth.LIT_BASE + lo + 10 ** digits // 10}]
        if i:
            nodes += [typed(k), {"op": "join", "inputs": [1, 2], "algo": "auto"}]
        plans.append(nodes)
    return [tb.plan_nodes(x) for x in plans]


def prepare(case, seed):
    call = case["call"]
    hrng = np.random.default_rng(synth.QUERY_SEED)
    g = _gen(SHAPE_SEED)
    st = {"call": call, "ctx": _Ctx.get()}
    if "n" in case:
        n = case["n"]
        lay = _layout(n)
        pid = [int(x) for x in lay["pred_ids"]]
        cols = synth.university_store_torch(n, seed=SHAPE_SEED)
        table = _renaming(lay["sizes"], seed)
        if call == "lookup":
            r = int(hrng.integers(0, n))
            t = [int(_renamed(c[r:r + 1], table)) for c in cols]
            st["pattern"] = tb.as_pattern(tuple(t[j] if "spo"[j] in case["shape"] else 0 for j in range(3)))
        elif call == "scan":
            st["patterns"] = [tb.as_pattern(q) for q in _scan_patterns(cols, n, case["patterns"], table, hrng)]
        elif call == "multi":
            js = (1, 7, 2, 3, 5, 6, 9, 10, 11, 12, 13, 14, 15, 16, 17)
            pats = [synth.Pattern(0, pid[0], int(lay["class_base"]), var=(X, -1, -1))]
            pats += [synth.Pattern(0, pid[j], 0, var=(X, -1, Y)) for j in js]
            st["patterns"] = [tb.as_pattern(q) for q in pats[:case["patterns"]]]
        elif call == "plans":
            st["plans"] = _plans(cols, n, table, hrng)
            st["host"] = case["host"]
        elif call == "batch":
            qs = synth.batch_queries(*cols, m=case["queries"], hi=case["most"])
            keys = torch.as_tensor(np.array([q.key() for q, _, _ in qs], np.int64), device="cuda")
            for c in (0, 2):
                keys[:, c] = _renamed(keys[:, c], table)
            st["patterns"] = tb.pattern_array(keys.cpu().numpy())
        elif call == "entail":
            schema = [torch.as_tensor(x, device="cuda") for x in synth.rdfs_schema(synth.uni_subjects(n))]
            cols = [torch.cat([c, x]) for c, x in zip(cols, schema)]
            st["vocab"] = synth.rdfs_vocab(synth.uni_subjects(n))
        st["store"] = _Store(*_shuffled([_renamed(cols[0], table), cols[1], _renamed(cols[2], table)], seed))
        if call == "bind":
            pat = synth.Pattern(0, pid[1], 0, var=(X, -1, V))
            st["pattern"] = tb.as_pattern(pat)
            lo = synth.LIT_BASE + 10
            st["preds"] = [(V, "range", lo, lo + int(round(case["keep"] * 100)) - 1)]
            st["idx"] = _Set(tb.tid_match(st["ctx"], st["store"].h, pat))
    elif call == "rows":
        rows = case["rows"]
        sub = max(64, rows // 4)
        st["set"] = _result_vector(*_pairs(rows, sub, g, _literals(case["digits"], g)), (X, V), _renaming([sub], seed), seed)
        lo = synth.LIT_BASE + 10 ** case["digits"] // 10
        st["preds"] = [(V, "range", lo, lo + 10 ** case["digits"] // 2 - 1)]
    else:
        l, r = case["left"], case["right"]
        sub = _subjects_of(max(l, r))
        ent = _entities(sub, g)
        table = _renaming([sub], seed)
        if call == "union":
            st["sets"] = [_result_vector(*_pairs(l, max(64, l // 4), g, _literals(4, g)), (X, V), table, seed),
                          _result_vector(*_pairs(r, sub, g, ent), (X, Y), table, seed)]
        else:
            how = case["how"]
            st["how"] = {"optional": "left", "full": "full"}.get(how, "auto")
            if how == "star":  # left: distinct subjects
                table = _renaming([max(sub, l)], seed)
                left = torch.randperm(max(sub, l), generator=g, device="cuda")[:l].int() + 1
                st["left"] = _result_vector(left, torch.full_like(left, 1 << 30), (X, -1), table, seed)
            elif how == "chain":
                st["left"] = _result_vector(*_pairs(l, sub, g, ent), (Z, X), table, seed)
            else:
                st["left"] = _result_vector(*_pairs(l, sub, g, _literals(4, g)), (X, V), table, seed)
            st["right"] = _result_vector(*_pairs(r, sub, g, ent), (X, Y), table, seed)
    tb.tid_ctx_sync(st["ctx"])
    return st


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def run(st):
    ctx, call = st["ctx"], st["call"]
    if call == "lookup":
        return _host(tb.tid_match(ctx, st["store"].h, st["pattern"]))
    if call == "scan":
        sets = [_Set(tb.tid_match(ctx, st["store"].h, q)) for q in st["patterns"]]
        return [s.columns() for s in sets]
    if call == "multi":
        sets = [_Set(h) for h in tb.tid_match_multi(ctx, st["store"].h, st["patterns"])]
        return [s.columns() for s in sets]
    if call == "bind":
        return _Set(tb.tid_bind(ctx, st["store"].h, st["pattern"], st["idx"].h, st["preds"])).columns()
    if call == "rows":
        f = _Set(tb.tid_filter(ctx, st["set"].h, st["preds"]))
        p = _Set(tb.tid_project(ctx, st["set"].h, (V, X)))
        return [f.columns(), p.columns()]
    if call == "join":
        return _Set(tb.tid_join(ctx, st["left"].h, st["right"].h, st["how"])).columns()
    if call == "union":
        return _Set(tb.tid_union(ctx, [s.h for s in st["sets"]])).columns()
    if call == "plans":
        if st["host"]:
            return [_host(tb.tid_exec(ctx, st["store"].h, x)) for x in st["plans"]]
        return [_Set(tb.tid_exec(ctx, st["store"].h, x)).columns() for x in st["plans"]]
    if call == "entail":
        out = []
        for rule in (2, 3, 5, 7, 9, 11):
            h, stats = tb.tid_entail(ctx, st["store"].h, rule, st["vocab"])
            out.append([_Set(h).columns(), [stats[f] for f in ("res1", "dist1", "res2", "dist2", "all")]])
        return out
    # a batch: the queries' lists one after another, and their lengths
    lists = [_Set(h).columns()[0] for h in tb.tid_match_batch(ctx, st["store"].h, st["patterns"])]
    lengths = np.array([x.shape[0] for x in lists], np.int64)
    with torch.cuda.stream(_Ctx.stream):
        return [torch.cat(lists), lengths]


def work(case):
    """Bytes a pass cannot do without: each input read once, each output written once (row counts from
    the recipe's frequencies)."""
    call = case["call"]
    f = synth.PRED_FREQ
    if call == "lookup":
        return {"bytes": 4 * len(case["shape"]) * case["n"] + 4 * 40, "flops": 0.0}
    if call == "scan":
        n, b = case["n"], 0.0
        for i in range(case["patterns"]):
            b += 4 * n * (2 if i % 4 == 2 else 1) + (4 * n * f[(1, 9, 4, 14)[i // 4 % 4]] if i % 4 == 1 else 0)
        return {"bytes": b, "flops": 0.0}
    if call == "multi":
        js = (1, 7, 2, 3, 5, 6, 9, 10, 11, 12, 13, 14, 15, 16, 17)
        return {"bytes": case["n"] * (8 + 4 * sum(f[j] for j in js[:case["patterns"] - 1])), "flops": 0.0}
    if call == "bind":
        h = case["n"] * f[1]
        return {"bytes": float(12 * h + 8 * h * min(0.9, case["keep"])), "flops": 0.0}
    if call == "rows":
        return {"bytes": case["rows"] * (8 + 4 + 8), "flops": 0.0}
    if call == "join":
        l, r, how = case["left"], case["right"], case["how"]
        sub = _subjects_of(max(l, r))
        if how == "star":
            return {"bytes": 4 * l + 8 * r + 8 * l * r / max(sub, l), "flops": 0.0}
        out = l * r / sub
        out += l * math.exp(-r / sub) if how in ("optional", "full") else 0
        out += r * math.exp(-l / sub) if how == "full" else 0
        return {"bytes": 8 * l + 8 * r + 12 * out, "flops": 0.0}
    if call == "union":
        return {"bytes": 20 * (case["left"] + case["right"]), "flops": 0.0}
    if call == "plans":
        # 20 patterns in 8 searches: the predicate column, in the stars, chains and one filter also the
        # object column (a type pattern), in the unions the subject column; then the property patterns' rows
        return {"bytes": case["n"] * (4 * 15 + 12 * (f[7] + f[11] + f[6] + f[2] + f[19] + f[4] + f[8] + f[12] + f[13] + f[3] + f[5])),
                "flops": 0.0}
    if call == "entail":
        # the store once, and the conclusions: about 0.75 rows of three terms per triple over the six rules
        return {"bytes": 12 * case["n"] * 1.75, "flops": 0.0}
    hits = (case["most"] - 1) / math.log(case["most"])
    return {"bytes": 12 * case["n"] + 2 * 4 * hits * case["queries"], "flops": 0.0}


def exact(case, seed):
    return None  # IDs, indices and counts: whole numbers, compared as they are
