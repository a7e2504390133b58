"""What a context keeps between calls, against the CPU oracle, bit-exact: searches
captured in a CUDA graph before and beside the context's other work, and two
threads on one context."""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1807_01409_gb300 import binding as tb

pytestmark = pytest.mark.gpu


class _Dev:
    def __init__(self, ptr, n, typestr):
        self.__cuda_array_interface__ = {"shape": (n,), "typestr": typestr, "data": (ptr, False), "version": 2}


def _read(h):
    """A set's rows by its device pointers (a captured set's row count is the graph's to write)."""
    info = tb.tid_set_info(h)
    n = int(torch.as_tensor(_Dev(info["dev_rows"], 1, "<i8"), device="cuda").item())
    if n == 0:
        return np.zeros((0, info["cols"]), np.int32)
    return np.stack([torch.as_tensor(_Dev(p, n, "<i4"), device="cuda").cpu().numpy() for p in info["dev_cols"]], 1)


def _rows(h):
    try:
        return tb.tid_set_to_host(h).copy()
    finally:
        tb.tid_set_free(h)


class _Program:
    """A context on a torch stream, with a store."""

    def __init__(self, n=300_000, seed=3):
        from paper_1807_01409_gb300 import build
        build.build()
        rng = np.random.default_rng(seed)
        t = np.unique(np.stack([rng.integers(1, hi, n) for hi in (5_000, 4, 900)], 1), axis=0)
        t = t[rng.permutation(len(t))].astype(np.int32)
        self.cols = [np.ascontiguousarray(t[:, c]) for c in range(3)]
        self.stream = torch.cuda.Stream()
        self.ctx = tb.tid_ctx_create(0, self.stream.cuda_stream)
        self.store = tb.tid_load(self.ctx, *self.cols)
        tb.tid_ctx_sync(self.ctx)

    def close(self):
        torch.cuda.synchronize()
        tb.tid_store_free(self.store)
        tb.tid_ctx_destroy(self.ctx)

    def captured(self, call):
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=self.stream):
            out = call()
        return g, out


@pytest.fixture()
def prog():
    p = _Program()
    yield p
    p.close()


def test_capture_after_sets_were_freed(prog, orc):
    """A program that made and freed sets captures a search (sets freed but not reused yet are at hand),
    and goes on: the graph and the context answer, and no error is left for the next context."""
    keys = [(0, 2, 0), (17, 0, 0), (0, 1, 5)]
    want = [orc.match(*prog.cols, k) for k in keys]
    for k, w in zip(keys, want):
        assert np.array_equal(_rows(tb.tid_match(prog.ctx, prog.store, k))[:, 0], w)
    freed = [tb.tid_match(prog.ctx, prog.store, k) for k in keys * 5]
    for h in freed:
        tb.tid_set_free(h)
    held = [tb.tid_match(prog.ctx, prog.store, keys[0]) for _ in range(20)]  # (no freed event left)
    tb.tid_set_free(held.pop())
    g, hs = prog.captured(lambda: [tb.tid_match(prog.ctx, prog.store, k) for k in keys])
    g.replay()
    torch.cuda.synchronize()
    for h, w in zip(hs, want):
        assert np.array_equal(_read(h)[:, 0], w)
        tb.tid_set_free(h)
    for h in held:
        assert np.array_equal(_rows(h)[:, 0], want[0])
    second = _Program(20_000)
    assert np.array_equal(_rows(tb.tid_match(second.ctx, second.store, keys[0]))[:, 0], orc.match(*second.cols, keys[0]))
    second.close()


def test_a_captured_set_keeps_its_row_count(prog, orc):
    """A graph writes the row counts of its sets at every run, also of those that were freed: no later
    set may be counted where it writes."""
    few, many = (17, 0, 0), (0, 2, 0)
    want = orc.match(*prog.cols, few)
    _rows(tb.tid_match(prog.ctx, prog.store, few))
    g, _ = prog.captured(lambda: [tb.tid_set_free(tb.tid_match(prog.ctx, prog.store, many)) for _ in range(3)])
    later = [tb.tid_match(prog.ctx, prog.store, few) for _ in range(40)]
    tb.tid_ctx_sync(prog.ctx)
    g.replay()
    torch.cuda.synchronize()
    for h in later:
        assert np.array_equal(_rows(h)[:, 0], want)


def test_capture_before_any_search(prog, orc):
    """The context's first search is captured: the context answers before the graph has run, and the
    graph before, after and beside the context's own work, on another stream."""
    keys = [(0, 2, 0), (17, 0, 0), (0, 1, 5)]
    want = [orc.match(*prog.cols, k) for k in keys]
    first = tb.tid_match(prog.ctx, prog.store, (0, 0, 0))  # (no search: every position)
    g, hs = prog.captured(lambda: [tb.tid_match(prog.ctx, prog.store, keys[0])]
                          + tb.tid_match_multi(prog.ctx, prog.store, keys[1:]))
    for k, w in zip(keys, want):
        assert np.array_equal(_rows(tb.tid_match(prog.ctx, prog.store, k))[:, 0], w), k
    other = torch.cuda.Stream()
    for _ in range(20):
        with torch.cuda.stream(other):
            g.replay()
        for h, w in [(tb.tid_match(prog.ctx, prog.store, k), w) for k, w in zip(keys, want)]:
            assert np.array_equal(_rows(h)[:, 0], w)
    torch.cuda.synchronize()
    for h, w in zip(hs, want):
        assert np.array_equal(_read(h)[:, 0], w)
        tb.tid_set_free(h)
    tb.tid_set_free(first)


def test_two_threads_on_one_context(orc):
    """Extractions and joins of two threads interleave on one context: every thread gets its own column
    bounds (values of one thread's columns lie far outside the other's) and look-back words."""
    p = _Program(260_000, seed=8)
    wide = [np.random.default_rng(9).permutation(np.arange(60_000, dtype=np.int32) * 35_000 + 1) for _ in range(2)]
    other = [wide[0], np.full(60_000, 2, np.int32), wide[1]]
    stores = [(p.store, p.cols), (tb.tid_load(p.ctx, *other), other)]
    errors = []

    def worker(store, cols):
        try:
            pat = tb.make_pattern(0, 2, 0, var=(0, -1, 1))
            subj = tb.make_pattern(0, 2, 0, var=(0, -1, -1))
            idx = orc.match(*cols, (0, 2, 0))
            want, keys = (orc.bind(*cols, (0, 2, 0), v, idx) for v in ((0, -1, 1), (0, -1, -1)))
            first = orc.filter(want, 0, "le", int(want.rows[len(want.rows) // 50, 0]))
            pair = orc.join(first, keys, method="sortmerge")
            for _ in range(40):
                h = tb.tid_match(p.ctx, store, pat)
                b, k = tb.tid_bind(p.ctx, store, pat, h), tb.tid_bind(p.ctx, store, subj, h)
                f = tb.tid_filter(p.ctx, b, [(0, "le", int(want.rows[len(want.rows) // 50, 0]), 0)])
                j = tb.tid_join(p.ctx, f, k)
                for s, w in ((b, want), (k, keys), (f, first), (j, pair)):
                    if not np.array_equal(_rows(s), w.rows):
                        errors.append((len(cols[0]), w.vars, w.n))
                tb.tid_set_free(h)
        except Exception as e:  # reported below
            errors.append(repr(e))

    ths = [threading.Thread(target=worker, args=a) for a in stores]
    for t in ths:
        t.start()
    for t in ths:
        t.join()
    tb.tid_store_free(stores[1][0])
    p.close()
    assert not errors, errors[:5]


def test_a_set_freed_under_capture_outlives_the_graph(prog, orc):
    """A graph that filters a set which is freed while it is captured: the set's memory is no other's,
    however much the context allocates before the graph runs."""
    key, pat = (0, 2, 0), tb.make_pattern(0, 2, 0, var=(0, -1, 1))
    bound = orc.bind(*prog.cols, key, (0, -1, 1), orc.match(*prog.cols, key))
    want = orc.filter(bound, 1, "le", 300).rows
    idx = tb.tid_match(prog.ctx, prog.store, pat)
    b = tb.tid_bind(prog.ctx, prog.store, pat, idx)
    assert np.array_equal(_rows(tb.tid_filter(prog.ctx, b, [(1, "le", 300, 0)])), want)  # (its row count is known)

    def call():
        f = tb.tid_filter(prog.ctx, b, [(1, "le", 300, 0)])
        tb.tid_set_free(b)
        return f
    g, f = prog.captured(call)
    others = [tb.tid_set_from_host(prog.ctx, bound.rows + 7, (0, 1)) for _ in range(8)]
    g.replay()
    torch.cuda.synchronize()
    assert np.array_equal(_read(f), want)
    for h in others + [f, idx]:
        tb.tid_set_free(h)


def test_look_backs_answer_after_one_gave_up(prog, orc):
    """The wait that is made to run out is an operator's own: it shares their status words, and a selection
    that looks back answers right after it."""
    rows = np.stack([np.arange(1, 8001), np.arange(8000) % 37], 1).astype(np.int32)  # four tiles
    h = tb.tid_set_from_host(prog.ctx, rows, (0, 1))
    want = orc.filter(orc.TupleSet((0, 1), rows), 1, "lt", 9).rows
    for _ in range(3):
        assert tb.tid_ctx_test_bounded_wait(prog.ctx, 50) == tb.TID_ERR_TIMEOUT
        assert np.array_equal(_rows(tb.tid_filter(prog.ctx, h, [(1, "lt", 9, 0)])), want)
    tb.tid_ctx_sync(prog.ctx)
    tb.tid_set_free(h)


def test_captured_operators(prog, orc):
    """Operators that need no row count from the device, captured on long and short sets: FILTER, SELECT
    DISTINCT (a prefix, and columns reordered), a join with keys and a union; run twice."""
    key, pat = (0, 2, 0), tb.make_pattern(0, 2, 0, var=(0, -1, 1))
    big = orc.bind(*prog.cols, key, (0, -1, 1), orc.match(*prog.cols, key))
    small = orc.TupleSet((0, 1), big.rows[:900])
    keys = orc.TupleSet((0,), np.unique(big.rows[::50, :1], axis=0))
    hb, hs, hk = (tb.tid_set_from_host(prog.ctx, s.rows, s.vars) for s in (big, small, keys))
    tb.tid_ctx_sync(prog.ctx)
    for h in (hb, hs, hk):
        tb.tid_set_rows(h)

    def call():
        out = []
        for h in (hb, hs):
            out += [tb.tid_filter(prog.ctx, h, [(1, "le", 300, 0)]), tb.tid_project(prog.ctx, h, (0,)),
                    tb.tid_project(prog.ctx, h, (1, 0)), tb.tid_join(prog.ctx, hk, h), tb.tid_union(prog.ctx, [h, hs])]
        return out
    want = []
    for s in (big, small):
        want += [orc.filter(s, 1, "le", 300), orc.project(s, (0,)), orc.project(s, (1, 0)),
                 orc.join(keys, s, method="sortmerge"), orc.union([s, small])]
    for h, w in zip(call(), want):
        assert np.array_equal(_rows(h), w.rows)
    g, out = prog.captured(call)
    assert np.array_equal(_rows(tb.tid_match(prog.ctx, prog.store, pat))[:, 0], orc.match(*prog.cols, key))
    for _ in range(2):
        g.replay()
        torch.cuda.synchronize()
        for h, w in zip(out, want):
            assert np.array_equal(_read(h), w.rows)
    for h in out + [hb, hs, hk]:
        tb.tid_set_free(h)
