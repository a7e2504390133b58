"""SELECT DISTINCT of a reordered result whose rows repeat, as a store with repeated
triples gives them: every repeat is dropped, wherever it lies."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1807_01409_gb300 import binding as tb

pytestmark = pytest.mark.gpu


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


def _bound(ctx, rows, again, rng):
    """The result vector of (?x ?p ?y) over the triples `rows`, those of the sorted positions `again` twice."""
    t = np.unique(rows, axis=0)
    t = np.concatenate([t, t[[a % len(t) for a in again]]]) if len(again) else t
    t = t[rng.permutation(len(t))].astype(np.int32)
    cols = [np.ascontiguousarray(t[:, c]) for c in range(3)]
    st = tb.tid_load(ctx, *cols)
    pat = tb.make_pattern(0, 0, 0, var=(0, 1, 2))
    idx = tb.tid_match(ctx, st, pat)
    h = tb.tid_bind(ctx, st, pat, idx)
    assert tb.tid_set_rows(h) == len(t)
    tb.tid_set_free(idx)
    tb.tid_store_free(st)
    return h


# steps of 1024 rows; one CTA up to 4096 rows; a repeat at the edges of steps and lanes, first and last
@pytest.mark.parametrize("again", [[], [0], [2], [3], [1022], [1023], [1151], [4094], [-1], [-1, 0, 1023, 2047], list(range(0, 4090, 7))])
@pytest.mark.parametrize("n", [4000, 4096, 4097, 5120, 9999, 300_007])
@pytest.mark.parametrize("high", [1000, 2**31 - 1])          # packed rows; rows wider than 64 bits
def test_reordered_rows_are_distinct(ctx, orc, n, again, high):
    rng = np.random.default_rng([n, len(again), high])
    rows = np.stack([rng.integers(1, high, n), rng.integers(1, min(high, 2**31 - 1), n), rng.integers(1, high, n)], 1)
    h = _bound(ctx, rows, again, rng)
    s = orc.TupleSet((0, 1, 2), np.unique(rows, axis=0).astype(np.int32))
    for order in ((2, 0, 1), (1, 0, 2)):
        assert np.array_equal(_rows(tb.tid_project(ctx, h, order)), orc.project(s, order).rows), order
    tb.tid_set_free(h)


def test_right_outer_join_of_repeated_rows(ctx, orc):
    """Its rows are those of a left join, reordered with DISTINCT."""
    rng = np.random.default_rng(4)
    rows = np.stack([rng.integers(1, 3000, 20_000), rng.integers(1, 50, 20_000), rng.integers(1, 3000, 20_000)], 1)
    h = _bound(ctx, rows, list(range(0, 19_000, 5)), rng)
    R = orc.TupleSet((0, 1, 2), np.unique(rows, axis=0).astype(np.int32))
    L = orc.TupleSet((0, 3), orc.canonical(np.stack([rng.integers(1, 6000, 900), rng.integers(1, 9, 900)], 1).astype(np.int32)))
    hl = tb.tid_set_from_host(ctx, L.rows, L.vars)
    want = orc.right_join(L, R)
    assert np.array_equal(_rows(tb.tid_join(ctx, hl, h, "right")), want.rows)
    tb.tid_set_free(hl)
    tb.tid_set_free(h)
