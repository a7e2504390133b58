"""Row selections and entailment from the size where a CTA's range is 32 steps of 1024
rows instead of 8 (eight ranges per SM: 39.8M rows on 152 SMs), ragged, against torch."""
import pytest

torch = pytest.importorskip("torch")

from paper_1807_01409_gb300 import binding as tb

pytestmark = pytest.mark.gpu


class _Dev:
    def __init__(self, ptr, n):
        self.__cuda_array_interface__ = {"shape": (n,), "typestr": "<i4", "data": (ptr, False), "version": 2}


@pytest.fixture(scope="module")
def ctx():
    from paper_1807_01409_gb300 import build
    build.build()
    c = tb.tid_ctx_create(0, None)
    yield c
    tb.tid_ctx_destroy(c)


@pytest.fixture(scope="module")
def n():
    return torch.cuda.get_device_properties(0).multi_processor_count * 256 * 1024 + 57 * 1024 + 7


def _same(h, want):
    """The set's columns equal the tensors `want`; frees it."""
    rows, info = tb.tid_set_rows(h), tb.tid_set_info(h)
    torch.cuda.synchronize()  # (the context's stream is its own)
    assert rows == want[0].shape[0] and info["cols"] == len(want)
    for p, w in zip(info["dev_cols"], want):
        assert rows == 0 or torch.equal(torch.as_tensor(_Dev(p, rows), device="cuda"), w.int())
    tb.tid_set_free(h)


def _shuffled(g, *cols):
    order = torch.randperm(cols[0].shape[0], generator=g, device="cuda")
    return [c[order].int().contiguous() for c in cols]


def test_selections(ctx, n):
    """bind (one tested slot, two, none with DISTINCT), FILTER, a distinct prefix and the join with keys."""
    g = torch.Generator(device="cuda").manual_seed(5)
    i = torch.arange(n, device="cuda")
    s, o = i // 3 + 1, (i % 3) * 1000 + 1 + torch.randint(0, 1000, (n,), generator=g, device="cuda")  # in (s, o) order
    S, O = _shuffled(g, s, o)
    P = torch.ones_like(S)
    torch.cuda.synchronize()
    st = tb.tid_load(ctx, S, P, O, copy=0)
    pat = tb.make_pattern(0, 1, 0, var=(0, -1, 1))
    idx = tb.tid_match(ctx, st, pat)
    b = tb.tid_bind(ctx, st, pat, idx)
    edge = int(s[n // 2])
    for preds, keep in ([(1, "eq", 1500, 0)], o == 1500), ([(1, "le", 1700, 0)], o <= 1700), ([(1, "ge", 1, 0)], o >= 1), \
            ([(1, "gt", 5000, 0)], o > 5000), ([(0, "ge", edge, 0), (1, "le", 1200, 0)], (s >= edge) & (o <= 1200)):
        want = [s[keep], o[keep]]
        _same(tb.tid_bind(ctx, st, pat, idx, preds), want)
        _same(tb.tid_filter(ctx, b, preds), want)
    distinct = torch.unique(s)
    _same(tb.tid_project(ctx, b, (0,)), [distinct])
    _same(tb.tid_bind(ctx, st, tb.make_pattern(0, 1, 0, var=(0, -1, -1)), idx), [distinct])
    keys = distinct[torch.randperm(distinct.shape[0], generator=g, device="cuda")[:distinct.shape[0] // 20]].sort().values
    hk = tb.tid_set_from_host(ctx, keys.int().cpu().numpy().reshape(-1, 1), (0,))
    keep = torch.isin(s, keys)
    _same(tb.tid_join(ctx, hk, b), [s[keep], o[keep]])
    for h in (hk, b, idx):
        tb.tid_set_free(h)
    tb.tid_store_free(st)


@pytest.mark.parametrize("form", ["matrix", "map", "join"])
def test_entailment(ctx, n, form):
    """Marks over the store, then the bit matrix (classes and subjects near each other), the key map (subjects
    spread over int32, one superclass) or the hash join (two superclasses)."""
    g = torch.Generator(device="cuda").manual_seed(6)
    v = {"type": 1, "domain": 2, "range": 3, "subprop": 4, "subclass": 5}
    classes = torch.arange(100, 140, device="cuda")
    ups = [100 + (classes - 100) // 2] + ([100 + (classes + 7) % 40] if form == "join" else [])
    sub = n // 2
    s = torch.randint(1000, 1000 + sub, (n,), generator=g, device="cuda")
    o = torch.randint(100, 400, (n,), generator=g, device="cuda")
    key = torch.unique((s << 10) | o)                        # a set of triples
    s, o = (key >> 10), key & 1023
    p = torch.where((s + o) % 4 == 0, 1, 6 + o % 3)
    if form != "matrix":
        s = (s - 999) * ((2**31 - 2) // (sub + 1))
    while s.shape[0] <= n - 57 * 1024:                       # repeats dropped: filled up with other subjects' triples
        m = n - s.shape[0]
        s, p, o = torch.cat([s, s[:m]]), torch.cat([p, torch.full_like(p[:m], 9)]), torch.cat([o, 500 + o[:m]])
    hit = (p == 1) & (o < 140)
    near = torch.cat([torch.stack([s[hit], u[o[hit] - 100]], 1) for u in ups])
    concl = torch.unique((near[:, 0] << 10) | near[:, 1])
    schema = torch.unique(torch.cat([(classes << 10) | u for u in ups]))
    a, b = schema >> 10, schema & 1023
    S, P, O = _shuffled(g, torch.cat([s, a]), torch.cat([p, torch.full_like(a, 5)]), torch.cat([o, b]))
    torch.cuda.synchronize()
    st = tb.tid_load(ctx, S, P, O, copy=0)
    h, stats = tb.tid_entail(ctx, st, 9, v)
    assert stats == {"res1": a.shape[0], "dist1": 40, "res2": int(hit.sum()), "dist2": int(torch.unique(o[hit]).shape[0]),
                     "all": concl.shape[0]}
    _same(h, [concl >> 10, torch.ones_like(concl), concl & 1023])
    tb.tid_store_free(st)
