"""Row selection and joins at the edges of their kernels, against the CPU oracle,
bit-exact: selections around the step, range and kernel-choice boundaries, with
every comparison at the ends of int32; joins whose right side leads with the key
(runs found through a table over the key range, dense or spread over int32, one
and two key columns, skewed, unbound keys) and joins with a set of keys only."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1807_01409_gb300 import binding as tb

pytestmark = pytest.mark.gpu
LOWEST, HIGHEST = -2**31, 2**31 - 1


@pytest.fixture(scope="module")
def ctx():
    from paper_1807_01409_gb300 import build
    build.build()
    c = tb.tid_ctx_create(0, None)
    yield c
    tb.tid_ctx_destroy(c)


def _rows(h):
    try:
        return tb.tid_set_to_host(h).copy()
    finally:
        tb.tid_set_free(h)


def _set(ctx, s):
    return tb.tid_set_from_host(ctx, s.rows, s.vars)


# k_sel_mark / k_sel_expand from 2^13 rows up (steps of 1024, ranges of 8 or 32 steps), k_compact below
SELECT_ROWS = [1, 2047, 2**13 - 1, 2**13, 2**13 + 1, 20_001, 2**18 - 1, 2**18, 2**18 + 1, 2**18 + 8 * 1024 + 1023, 1_300_003]
PREDS = [("lt", 500, 0), ("ge", 999, 0), ("ne", 7, 0), ("eq", 7, 0), ("lt", LOWEST, 0), ("gt", HIGHEST, 0),
         ("le", HIGHEST, 0), ("ge", LOWEST, 0), ("range", 10, 9), ("range", 990, HIGHEST)]


@pytest.mark.parametrize("n", SELECT_ROWS)
@pytest.mark.parametrize("k", [1, 2, 4])
def test_filter_edges(ctx, orc, n, k):
    rng = np.random.default_rng(n + k)
    cols = [np.arange(1, n + 1)] + [rng.integers(0, 1000, n) for _ in range(k - 1)]
    s = orc.TupleSet(tuple(range(k)), np.stack(cols, 1).astype(np.int32))
    h = _set(ctx, s)
    for cmp_, a, b in PREDS:
        want = orc.filter(s, k - 1, cmp_, a, b).rows
        got = _rows(tb.tid_filter(ctx, h, [(k - 1, cmp_, a, b)]))
        assert np.array_equal(got, want), (cmp_, a, b)
    if k > 1:  # two predicates, and a distinct prefix of a reordered set
        got = _rows(tb.tid_filter(ctx, h, [(k - 1, "gt", 100, 0), (0, "le", n // 2 + 1, 0)]))
        want = orc.filter(orc.filter(s, k - 1, "gt", 100, 0), 0, "le", n // 2 + 1, 0).rows
        assert np.array_equal(got, want)
        got = _rows(tb.tid_project(ctx, h, (k - 1,)))
        assert np.array_equal(got, orc.project(s, (k - 1,)).rows)
        got = _rows(tb.tid_project(ctx, h, tuple(range(k))[::-1]))
        assert np.array_equal(got, orc.project(s, tuple(range(k))[::-1]).rows)
    tb.tid_set_free(h)


@pytest.mark.parametrize("n", [5000, 40_000, 2**18 - 1, 2**18 + 5, 700_001])
@pytest.mark.parametrize("shift", [0, 1])
def test_bind_tests_edges(ctx, orc, n, shift):
    """One tested slot (its values stashed), two tested slots, a repeated variable; borrowed columns
    16-byte aligned or not."""
    rng = np.random.default_rng(n + shift)
    full = [rng.integers(1, 60_000, n + shift).astype(np.int32), rng.integers(1, 4, n + shift).astype(np.int32),
            rng.integers(1, 50, n + shift).astype(np.int32)]
    keep = np.unique(np.stack([c[shift:] for c in full], 1), axis=0, return_index=True)[1]
    keep = rng.permutation(keep)
    S, P, O = (np.ascontiguousarray(c[shift:][keep]) for c in full)
    dev = [torch.from_numpy(np.concatenate([np.zeros(shift, np.int32), c])).cuda()[shift:] for c in (S, P, O)]
    st = tb.tid_load(ctx, *dev, copy=0)
    for key, var, preds in [((0, 2, 0), (0, -1, 1), [(1, "range", 10, 20)]), ((0, 2, 0), (0, -1, 1), [(0, "lt", 90, 0)]),
                            ((0, 0, 0), (0, 1, 2), [(2, "ge", 10, 0), (0, "gt", 100, 0)]),
                            ((0, 0, 0), (0, 1, 0), []), ((0, 0, 0), (0, 1, 2), [(1, "eq", 3, 0)])]:
        idx = tb.tid_match(ctx, st, key)
        want = orc.bind(S, P, O, key, var, orc.match(S, P, O, key))
        for v, c, a, b in preds:
            want = orc.filter(want, v, c, a, b)
        got = _rows(tb.tid_bind(ctx, st, tb.make_pattern(*key, var=var), idx, preds))
        assert np.array_equal(got, want.rows), (key, var, preds)
        tb.tid_set_free(idx)
    tb.tid_store_free(st)


def _random_set(orc, rng, vars_, n, ids):
    r = np.stack([ids(rng, n) for _ in vars_], 1).astype(np.int32)
    return orc.TupleSet(vars_, orc.canonical(r))


IDS = {
    "dense": lambda rng, n: rng.integers(0, max(2, n // 2), n),           # 0: unbound rows among them
    "clusters": lambda rng, n: rng.integers(0, max(2, n // 3), n) + (rng.integers(0, 2, n) << 30),
    "wide": lambda rng, n: rng.integers(LOWEST, HIGHEST, n) // 7919 * 7919,
    "skew": lambda rng, n: np.where(rng.random(n) < 0.02, 5, rng.integers(1, 4 * n + 2, n)),
}
JOINS = [((0, 1), (0, 2)), ((1, 0), (0, 2)), ((0, 1, 2), (1, 3)), ((2, 0, 1), (0, 1, 3)), ((0,), (0, 2)), ((0, 1), (0,)),
         ((0,), (0,)), ((1, 0), (0,))]


@pytest.mark.parametrize("ids", sorted(IDS))
@pytest.mark.parametrize("shape", range(len(JOINS)))
@pytest.mark.parametrize("size", [(3, 1), (1, 1025), (4000, 4097), (50_000, 7000), (300, 30_000)])
def test_joins_on_a_leading_key(ctx, orc, ids, shape, size):
    lv, rv = JOINS[shape]
    rng = np.random.default_rng([shape, *size, len(ids)])
    L = _random_set(orc, rng, lv, size[0], IDS[ids])
    R = _random_set(orc, rng, rv, size[1], IDS[ids])
    hl, hr = _set(ctx, L), _set(ctx, R)
    want = orc.join(L, R, method="sortmerge")
    for algo in ("auto", "sort_merge"):
        got = _rows(tb.tid_join(ctx, hl, hr, algo))
        assert np.array_equal(got, want.rows), algo
    assert np.array_equal(_rows(tb.tid_join(ctx, hl, hr, "left")), orc.left_join(L, R).rows)
    tb.tid_set_free(hl)
    tb.tid_set_free(hr)


def test_member_join_large(ctx, orc):
    """Keys only against 2^18 rows and more: the selection's two-launch form."""
    rng = np.random.default_rng(5)
    R = _random_set(orc, rng, (0, 2), 400_000, IDS["dense"])
    L = orc.TupleSet((0,), orc.canonical(rng.integers(0, 200_000, (60_000, 1)).astype(np.int32)))
    hl, hr = _set(ctx, L), _set(ctx, R)
    want = orc.join(L, R, method="sortmerge")
    assert np.array_equal(_rows(tb.tid_join(ctx, hl, hr)), want.rows)
    assert np.array_equal(_rows(tb.tid_join(ctx, hr, hl)), orc.join(R, L, method="sortmerge").rows)
    tb.tid_set_free(hl)
    tb.tid_set_free(hr)


@pytest.mark.parametrize("n", [1, 1023, 1024, 1025, 8191, 8193, 300_001, 39_900_007])
@pytest.mark.parametrize("shift", [0, 1])
def test_search_edges(ctx, n, shift):
    """Single and multi-pattern searches around the step and range boundaries (a range is 8 steps, from
    39.8M triples on 32), columns 16-byte aligned or not, against torch.nonzero; ranges without a hit,
    with few and with all."""
    g = torch.Generator(device="cuda").manual_seed(n)
    cols = [torch.randint(1, hi, (n + shift,), generator=g, device="cuda", dtype=torch.int32)[shift:]
            for hi in (5, 400, 2_000_000)]
    cols[1][n // 3: n // 2] = 7                       # a stretch where every triple matches
    cols[2][n - 1] = 3_000_000                        # a single hit, the last triple
    torch.cuda.synchronize()
    st = tb.tid_load(ctx, *cols, copy=0)
    keys = [(1, 0, 0), (0, 7, 0), (0, 0, 3_000_000), (2, 7, 0), (0, 0, 0), (4_000, 0, 0), (0, 9, 3_000_000)]
    want = []
    for k in keys:
        hit = torch.ones(n, dtype=torch.bool, device="cuda")
        for c, v in zip(cols, k):
            if v:
                hit &= c == v
        want.append(torch.nonzero(hit)[:, 0].int().cpu().numpy())
    for k, w in zip(keys, want):
        assert np.array_equal(_rows(tb.tid_match(ctx, st, k))[:, 0], w), k
    for h, k, w in zip(tb.tid_match_multi(ctx, st, keys), keys, want):
        assert np.array_equal(_rows(h)[:, 0], w), k
    tb.tid_store_free(st)


X, Y, Z, W = 0, 1, 2, 3


def _plan_store(seed, n):
    rng = np.random.default_rng(seed)
    t = np.unique(np.stack([rng.integers(1, n // 6, n), rng.integers(1, 5, n) + (1 << 20), rng.integers(1, n // 6, n)], 1),
                  axis=0)
    t = t[rng.permutation(len(t))].astype(np.int32)
    return [np.ascontiguousarray(t[:, c]) for c in range(3)]


@pytest.mark.parametrize("algo", ["auto", "hash", "left", "right", "full"])
@pytest.mark.parametrize("n", [3_000, 60_000, 1_200_000])
def test_plan_extracts_what_a_join_needs(ctx, orc, algo, n):
    """A small side reduces the extraction of a large MATCH (below and above the row selection's sizes), on
    either input, through FILTERs, on one and two shared variables, with an empty small side; outer joins
    keep their unmatched rows."""
    from paper_1807_01409_gb300 import synth
    S, P, O = _plan_store(n, n)
    st = tb.tid_load(ctx, S, P, O)
    p = 1 << 20
    few = {"op": "match", "pattern": synth.Pattern(0, p + 1, int(O[P == p + 1][0]), var=(X, -1, -1))}
    some = [{"op": "match", "pattern": synth.Pattern(0, p + 2, 0, var=(X, -1, Y))},
            {"op": "filter", "input": 0, "var": X, "cmp": "le", "a": n // 600}]
    many = {"op": "match", "pattern": synth.Pattern(0, p + 3, 0, var=(X, -1, Y))}
    other = {"op": "match", "pattern": synth.Pattern(0, p + 4, 0, var=(Z, -1, X))}
    none = {"op": "match", "pattern": synth.Pattern(0, p + 1, 1 << 29, var=(X, -1, -1))}
    plans = []
    for small in (few, none):
        for big in (many, other):
            plans += [[small, big, {"op": "join", "inputs": [0, 1], "algo": algo}],
                      [small, big, {"op": "join", "inputs": [1, 0], "algo": algo}]]
    plans += [some + [many, {"op": "join", "inputs": [1, 2], "algo": algo}],       # two shared variables
              some + [many, {"op": "filter", "input": 2, "var": Y, "cmp": "ge", "a": 10},
                      {"op": "join", "inputs": [3, 1], "algo": algo}],
              [few, many, other, {"op": "join", "inputs": [0, 1], "algo": algo}, {"op": "join", "inputs": [3, 2], "algo": algo},
               {"op": "project", "input": 4, "vars": [X, Z]}],
              [few, many, {"op": "join", "inputs": [0, 1], "algo": algo}, {"op": "union", "inputs": [1, 2]}]]
    if algo == "hash":  # an outer join is not a hash join; a chain through both inputs is
        plans = plans[:-1]
    for plan in plans:
        got = _rows(tb.tid_exec(ctx, st, plan))
        want = orc.execute(S, P, O, plan)
        assert np.array_equal(got, want.rows), plan
    bad = [few, many, {"op": "filter", "input": 1, "var": W, "cmp": "ge", "a": 1}, {"op": "join", "inputs": [0, 2]}]
    with pytest.raises(tb.TidError) as e:  # a FILTER on a variable that its MATCH lacks is still refused
        tb.tid_exec(ctx, st, bad)
    assert e.value.code == tb.TID_ERR_ARG
    tb.tid_store_free(st)


UNIONS = [((0, 1), (0, 2)), ((0, 1), (0, 1)), ((0,), (0, 1, 2)), ((0, 1, 2), (0, 2)), ((0, 1), (0, 2), (0, 1, 3)), ((2,), (2,))]


@pytest.mark.parametrize("ids", ["dense", "clusters", "wide", "literals", "one"])
@pytest.mark.parametrize("shape", range(len(UNIONS)))
@pytest.mark.parametrize("n", [1, 2048, 4095, 4097, 30_000])
def test_union_merges(ctx, orc, ids, shape, n):
    """Branches merged without a sort: rows of up to 64 bits packed (a branch without a variable adds its 0
    to the other's values), wider ones by column; repeats across branches, tile boundaries, uneven sizes."""
    rng = np.random.default_rng([n, shape, len(ids)])
    fn = dict(IDS, literals=lambda r, m: (1 << 30) + r.integers(0, 5000, m), one=lambda r, m: np.full(m, 9))[ids]
    sets = [_random_set(orc, rng, v, max(1, n >> i), fn) for i, v in enumerate(UNIONS[shape])]
    if UNIONS[shape][0] == UNIONS[shape][1]:  # half of the second branch repeats the first
        sets[1] = orc.TupleSet(sets[1].vars, orc.canonical(np.concatenate([sets[1].rows, sets[0].rows[::2]])))
    hs = [_set(ctx, s) for s in sets]
    got = tb.tid_union(ctx, hs)
    want = orc.union(sets)
    assert tb.tid_set_info(got)["vars"] == tuple(want.vars)
    assert np.array_equal(_rows(got), want.rows)
    for h in hs:
        tb.tid_set_free(h)


@pytest.mark.parametrize("rule", [2, 3, 5, 7, 9, 11])
@pytest.mark.parametrize("schema", ["tree", "many"])      # one schema row per key, or several
@pytest.mark.parametrize("spread", [1, 70_001])            # IDs dense, or over most of int32
@pytest.mark.parametrize("n", [900, 45_000])
def test_entailment_forms(ctx, orc, rule, schema, spread, n):
    """The forms of a rule's last step (bit matrix, key map, hash join) and of its key set (a range of
    bits, a table): small and large ID ranges, functional and branching schemas."""
    rng = np.random.default_rng([rule, len(schema), spread, n])
    v = {"type": 1, "domain": 2, "range": 3, "subprop": 4, "subclass": 5}
    t = []
    for k in range(30):                                     # terms 10 .. 39: classes and predicates
        ups = [k // 2] if schema == "tree" else rng.integers(0, 30, 3)
        for u in ups:
            for p in (v["domain"], v["range"], v["subprop"], v["subclass"]):
                t.append((10 + k, p, 10 + int(u)))
    data = np.stack([rng.integers(10, 10 + n // 3, n), np.where(rng.random(n) < 0.3, 1, rng.integers(10, 60, n)),
                     rng.integers(10, 60, n)], 1)
    data[::7, 2] = rng.integers(10, n // 3 + 10, len(data[::7]))
    t = np.unique(np.concatenate([np.array(t), data]), axis=0)
    t = np.where(t < 10, t, (t - 9) * spread % (2**31 - 1) + 9)
    t = t[rng.permutation(len(t))].astype(np.int32)
    S, P, O = (np.ascontiguousarray(t[:, c]) for c in range(3))
    st = tb.tid_load(ctx, S, P, O)
    h, stats = tb.tid_entail(ctx, st, rule, v)
    want, wstats = orc.entail(S, P, O, rule, v)
    assert stats == wstats
    assert np.array_equal(_rows(h), want.rows)
    tb.tid_store_free(st)
