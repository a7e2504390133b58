"""Batched search in every kernel shape the autotuner may choose, against the CPU
oracle, bit-exact: all masks on ragged stores, candidates dense and sparse, and more
keys than one sub-batch."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1807_01409_gb300 import binding as tb
from paper_1807_01409_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_1807_01409_gb300 import build
    build.build()
    c = tb.tid_ctx_create(0, None)
    yield c
    tb.tid_ctx_destroy(c)


@pytest.fixture(params=sorted(tb.BATCH_SHAPES), ids=lambda s: tb.BATCH_SHAPES[s])
def shape(request, ctx):
    yield request.param
    tb.tid_ctx_test_batch_shape(ctx, -1)


_known = {}  # the oracle's lists, one set for the four shapes


def _check(ctx, orc, cols, keys, shape, per, name):
    tb.tid_ctx_test_batch_shape(ctx, shape, per)
    st = tb.tid_load(ctx, *cols)
    hs = tb.tid_match_batch(ctx, st, keys)
    used = tb.tid_batch_tuning(ctx)
    assert used["shape"] == tb.BATCH_SHAPES[shape] and used["keys_per_sub_batch"] == per
    distinct = len(set(keys) - {(0, 0, 0)})
    assert used["sub_batches"] >= -(-distinct // per)
    for k, h in zip(keys, hs):
        got = tb.tid_set_to_host(h)[:, 0]
        tb.tid_set_free(h)
        if (name, k) not in _known:
            _known[name, k] = orc.match(*cols, k)
        assert np.array_equal(got, _known[name, k]), k
    tb.tid_store_free(st)


@pytest.mark.parametrize("n", [1, 31, 33, 255, 257, 4097, 100_003, 1_000_001])
def test_every_mask(ctx, orc, shape, n):
    """Seven masks at every triple: each slot of 32 adds up to 224 candidates to a warp's queue."""
    rng = np.random.default_rng(n)
    cols = [rng.integers(1, hi, n).astype(np.int32) for hi in (4, 3, 5)]
    keys = [(s, p, o) for s in range(5) for p in range(4) for o in range(6)]
    _check(ctx, orc, cols, keys, shape, tb.TID_BATCH_KEYS, ("every", n))


@pytest.mark.parametrize("n", [1000, 300_001, 5_000_003])
def test_few_candidates(ctx, orc, shape, n):
    """A queue that waits over many slots, and what is left in it at the end of a warp's triples."""
    rng = np.random.default_rng(n + 1)
    cols = [rng.integers(1, hi, n).astype(np.int32) for hi in (n // 3 + 2, 30, n // 5 + 2)]
    rows = list(rng.integers(0, n, 40)) + [0, n - 1]
    keys = [tuple(int(c[r]) if m >> j & 1 else 0 for j, c in enumerate(cols)) for i, r in enumerate(rows)
            for m in (1, 4, 5, 3 + 3 * (i % 2), 7)]
    _check(ctx, orc, cols, keys, shape, tb.TID_BATCH_KEYS, ("few", n))


@pytest.mark.parametrize("per", [1, 100, 1152, tb.TID_BATCH_KEYS])
def test_sub_batches(ctx, orc, shape, per):
    st = synth.tiny_store()
    rng = np.random.default_rng(per)
    rows = rng.integers(0, st.n, min(5 * tb.TID_BATCH_KEYS // 2, 8 * per))
    cols = (st.s, st.p, st.o)
    keys = [tuple(int(c[r]) if (1 + i % 7) >> j & 1 else 0 for j, c in enumerate(cols)) for i, r in enumerate(rows)]
    _check(ctx, orc, cols, keys, shape, per, "tiny")


def test_bad_shapes_are_refused(ctx):
    for s, k in ((len(tb.BATCH_SHAPES), 10), (0, 0), (0, tb.TID_BATCH_KEYS + 1)):
        with pytest.raises(tb.TidError) as e:
            tb.tid_ctx_test_batch_shape(ctx, s, k)
        assert e.value.code == tb.TID_ERR_ARG
