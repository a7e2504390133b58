"""The forms of a rule's last step that a small schema does not reach, against the
CPU oracle, bit-exact."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1807_01409_gb300 import binding as tb

pytestmark = pytest.mark.gpu
VOCAB = {"type": 1, "domain": 2, "range": 3, "subprop": 4, "subclass": 5}


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


def _store(ctx, rng, schema, data):
    t = np.unique(np.concatenate([np.array(schema), data]), axis=0)
    t = t[rng.permutation(len(t))].astype(np.int32)
    cols = [np.ascontiguousarray(t[:, c]) for c in range(3)]
    return tb.tid_load(ctx, *cols), cols


def _allocations(ctx, call):
    for after in range(200):
        tb.tid_ctx_inject_alloc_failure(ctx, after)
        try:
            call()
            return after
        except tb.TidError as e:
            assert e.code == tb.TID_ERR_OOM
        finally:
            tb.tid_ctx_inject_alloc_failure(ctx, -1)
    raise AssertionError("200 allocations")


def test_a_joined_conclusion_is_sorted_once(ctx, orc):
    """Several schema rows per key and terms too far apart for a bit matrix: the joined rows are sorted with
    the bounds that the extraction left, whether two of the conclusion's terms vary or three (a second sort,
    or a pass for the bounds, would show as further allocations)."""
    rng = np.random.default_rng(2)
    n = 60_000
    schema = [(100 + c, 5, 100 + (c * 7 + j) % 50) for c in range(50) for j in range(3)]
    schema += [(6 + c, 4, 6 + (c + j) % 9) for c in range(9) for j in (1, 2)]
    data = np.stack([rng.integers(1, 2**31 - 1, n), np.where(rng.random(n) < 0.5, 1, rng.integers(6, 15, n)),
                     rng.integers(100, 150, n)], 1)
    st, cols = _store(ctx, rng, schema, data)
    made = {}
    for rule in (7, 9):
        h, stats = tb.tid_entail(ctx, st, rule, VOCAB)
        want, wstats = orc.entail(*cols, rule, VOCAB)
        assert stats == wstats and np.array_equal(_rows(h), want.rows), rule
        made[rule] = _allocations(ctx, lambda: tb.tid_set_free(tb.tid_entail(ctx, st, rule, VOCAB)[0]))
    assert made[9] <= made[7], made
    tb.tid_store_free(st)


@pytest.mark.parametrize("keys", [16_000, 16_384, 16_385, 60_000])   # flags in shared memory up to 16384 key numbers
@pytest.mark.parametrize("spread", [1, 30_011])                       # a range of bits; a table (32768 slots and more)
@pytest.mark.parametrize("rule", [7, 9, 11])
def test_many_keys(ctx, orc, keys, spread, rule):
    """Key sets around and above what a CTA flags in shared memory, all keys or one in ten occurring."""
    rng = np.random.default_rng([keys, spread, rule])
    v = VOCAB
    t, n = (np.arange(keys) + 10), 120_000
    up = rng.permutation(t)
    term = v["subprop"] if rule == 7 else v["subclass"]
    schema = np.stack([t, np.full(keys, term), up], 1)
    seen = t[::10] if keys == 60_000 else t
    if rule == 7:
        data = np.stack([rng.integers(10, 9_000, n), rng.choice(seen, n), rng.integers(10, 9_000, n)], 1)
    else:
        data = np.stack([rng.integers(10, 40_000, n), np.full(n, v["type"]), rng.choice(seen, n)], 1)
    rows = np.concatenate([schema, data])
    rows = np.where(rows < 10, rows, (rows - 9) * spread + 9)
    assert rows.max() < 2**31 - 1
    st, cols = _store(ctx, rng, rows[:keys], rows[keys:])
    h, stats = tb.tid_entail(ctx, st, rule, v)
    want, wstats = orc.entail(*cols, rule, v)
    assert stats == wstats
    assert np.array_equal(_rows(h), want.rows)
    tb.tid_store_free(st)
