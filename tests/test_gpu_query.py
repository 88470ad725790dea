"""Query-level parity through the C-ABI: relational results bit-exact against
the oracle, label logits within the margin tolerance, decisions on every
clear row, and aggregates equal to the oracle's aggregation of the GPU's own
decision vector (Table 2 Q1/Q2 shapes, the reviews-movies join of Section 4,
the multi-label GROUP BY)."""
from dataclasses import replace

import numpy as np
import pytest

import synth
from helpers import compare_logits, gpu_ctx, oracle_preds, weights_list
from oracle import query as oq
from oracle import relational as rel
from oracle import transformer as tf
from paper_2608_10139_gb300 import aiq

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = gpu_ctx()
    yield c
    c.close()


def _load(ctx, t: synth.Table):
    text = (t.offsets, t.tokens) if t.offsets is not None else None
    return ctx.load_table(t.cols, text, n_rows=t.n_rows)


# ------------------------------------------------------------ relational ---

def _random_table(n, seed):
    rng = np.random.default_rng(seed)
    return synth.Table(n, {"a": rng.integers(0, 10, n).astype(np.int32),
                           "b": rng.integers(-2**40, 2**40, n).astype(np.int64),
                           "c": rng.standard_normal(n).astype(np.float32)})


PRED_SETS = [
    [],
    [("a", rel.GE, 5)],
    [("a", rel.LT, 3), ("b", rel.GT, 0)],
    [("a", rel.NE, 4), ("c", rel.LE, 0.25), ("b", rel.LE, 2**39)],
    [("a", rel.EQ, 7)],
    [("a", rel.GT, 100)],          # nothing survives
    [("a", rel.GE, -2**40)],       # constant outside the int32 range: everything survives
]


@pytest.mark.parametrize("n", [0, 1, 31, 2047, 2048, 2049, 100_003, (1 << 22) + 777, 1 << 24])
def test_filter_compaction_bit_exact(ctx, n):
    t = _random_table(n, n)
    ref_t = ctx.load_table(t.cols, n_rows=n)
    try:
        for preds in PRED_SETS:
            r = ctx.run_select(ref_t, 0, preds, [], [0, 1], flags=aiq.FLAG_RELATIONAL_ONLY)
            want = rel.compact(rel.predicate_mask(t.cols, preds, n))
            assert r.n_candidates == len(want)
            assert np.array_equal(r.cand_row_ids, want), preds
    finally:
        ctx.free_table(ref_t)


MIXES = [  # every count of int64 and 4-byte terms that has a kernel of its own, and five terms
    "b", "bb", "bbb", "bbbb", "ab", "abb", "babb", "abc", "cabb", "aabc", "ac", "aca", "acca", "abcab",
]


@pytest.mark.parametrize("n", [1, 8191, 8193, 16384, 16385, 70_001, (1 << 24) + 1])
def test_filter_term_mixes(ctx, n):
    """Conjunctions over columns of every type in any order, at the sizes where the
    filter changes kernels: one block (16,384 rows), the last block's scan (2^24),
    and the allocation-free call on the same columns."""
    torch = pytest.importorskip("torch")
    t = _random_table(n, n + 5)
    ref_t = ctx.load_table(t.cols, n_rows=n)
    dev = {k: torch.from_numpy(v).cuda() for k, v in t.cols.items()}
    code = {"a": aiq.INT32, "b": aiq.INT64, "c": aiq.FLOAT32}
    ids = torch.empty(n, dtype=torch.int32, device="cuda")
    count = torch.empty(1, dtype=torch.int64, device="cuda")
    consts = {"a": [(rel.GE, 2), (rel.NE, 7)], "b": [(rel.GT, -2**39), (rel.LE, 2**39), (rel.NE, 3), (rel.LT, 2**40)],
              "c": [(rel.LE, 0.75), (rel.GT, -1.5)]}
    try:
        for mix in MIXES if n < 1 << 24 else MIXES[::4]:
            preds = [(k, *consts[k][mix[:i].count(k)]) for i, k in enumerate(mix)]
            want = rel.compact(rel.predicate_mask(t.cols, preds, n))
            r = ctx.run_select(ref_t, 0, preds, [], [0, 1], flags=aiq.FLAG_RELATIONAL_ONLY)
            assert np.array_equal(r.cand_row_ids, want), mix
            if n <= 1 << 24:
                torch.cuda.synchronize()
                aiq.filter_compact_static([(dev[k].data_ptr(), code[k], o, v) for k, o, v in preds], n,
                                          ids.data_ptr(), count.data_ptr(), 0)
                torch.cuda.synchronize()
                assert int(count) == len(want) and np.array_equal(ids[:len(want)].cpu().numpy(), want), mix
    finally:
        ctx.free_table(ref_t)


@pytest.mark.parametrize("n", [16385, 2048 * 9, 2048 * 488, 2048 * 488 + 1, 2048 * 490 + 5, 2048 * 491, 2048 * 3000 - 1,
                               (1 << 24) - 3, 1 << 24])
def test_static_filter_tile_groups(n):
    """The allocation-free filter's compaction adds up the tile counts itself: sizes
    around its switch from a block to a warp per tile (488 tiles), groups of four
    tiles with 1 .. 4 of them present, and the largest table, with all, some and no
    rows kept."""
    torch = pytest.importorskip("torch")
    g = torch.Generator(device="cuda").manual_seed(n)
    col = torch.randint(0, 10, (n,), dtype=torch.int32, device="cuda", generator=g)
    ids = torch.empty(n, dtype=torch.int32, device="cuda")
    count = torch.empty(1, dtype=torch.int64, device="cuda")
    for terms in ([], [(rel.GE, 9)], [(rel.GE, 3)] * 5, [(rel.LT, 0)]):
        keep = torch.ones(n, dtype=torch.bool, device="cuda")
        for op, v in terms:
            keep &= col >= v if op == rel.GE else col < v
        want = keep.nonzero().flatten().int()
        torch.cuda.synchronize()
        aiq.filter_compact_static([(col.data_ptr(), aiq.INT32, op, v) for op, v in terms], n, ids.data_ptr(),
                                  count.data_ptr(), 0)
        torch.cuda.synchronize()
        assert int(count) == len(want) and torch.equal(ids[:len(want)], want), terms


def test_static_filter_under_capture():
    """The allocation-free filter recorded into a graph between the caller's own kernels,
    in its one-launch and two-launch forms: every replay filters what the column then holds."""
    torch = pytest.importorskip("torch")
    for n in (9000, 70_001):
        col = torch.zeros(n, dtype=torch.int32, device="cuda")
        base = torch.arange(n, dtype=torch.int32, device="cuda")
        ids = torch.empty(n, dtype=torch.int32, device="cuda")
        count = torch.zeros(1, dtype=torch.int64, device="cuda")
        twice = torch.zeros(1, dtype=torch.int64, device="cuda")
        call = lambda: aiq.filter_compact_static([(col.data_ptr(), aiq.INT32, rel.GE, 6)], n, ids.data_ptr(),
                                                 count.data_ptr(), torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        call()   # the device address is looked up before any capture
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            torch.remainder(base, 10, out=col)
            call()
            torch.add(count, count, out=twice)
        for step in range(3):
            base += 3
            ids.fill_(-1)
            g.replay()
            torch.cuda.synchronize()
            want = (base % 10 >= 6).nonzero().flatten().int()
            assert int(count) == len(want) and int(twice) == 2 * len(want)
            assert torch.equal(ids[:len(want)], want)


@pytest.mark.parametrize("n", [9000, 70_001])
@pytest.mark.parametrize("before", ["nothing", "copy", "memset", "join of two streams", "a call"])
def test_static_filter_captured_after(n, before):
    """Recorded behind each kind of graph node: none, copies and memsets (which let no
    kernel start early), two branches, and a call of its own."""
    torch = pytest.importorskip("torch")
    src = torch.arange(n, dtype=torch.int32, device="cuda")
    col = torch.full((n,), 9, dtype=torch.int32, device="cuda")
    other = torch.zeros(n, dtype=torch.int32, device="cuda")
    ids = torch.empty(n, dtype=torch.int32, device="cuda")
    count = torch.zeros(1, dtype=torch.int64, device="cuda")
    call = lambda: aiq.filter_compact_static([(col.data_ptr(), aiq.INT32, rel.GE, 6)], n, ids.data_ptr(),  # noqa: E731
                                             count.data_ptr(), torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    call()
    torch.cuda.synchronize()
    g, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(g):
        if before == "copy":
            col.copy_(src)
        elif before == "memset":
            col.zero_()
        elif before == "join of two streams":
            side.wait_stream(torch.cuda.current_stream())
            with torch.cuda.stream(side):
                torch.add(src, 1, out=other)
            torch.remainder(src, 10, out=col)
            torch.cuda.current_stream().wait_stream(side)
        elif before == "a call":
            call()
        call()
    for _ in range(2):
        col.fill_(9)
        ids.fill_(-1)
        g.replay()
        torch.cuda.synchronize()
        want = {"copy": src >= 6, "memset": src < 0, "join of two streams": src % 10 >= 6}.get(before, src >= 0)
        want = want.nonzero().flatten().int()
        assert int(count) == len(want) and torch.equal(ids[:len(want)], want)


@pytest.mark.parametrize("room", [64 << 20, 14 << 20, 10 << 20, 3 << 20])
def test_join_table_without_room(room):
    """A join whose table for all build rows (15.7 MB) does not fit under the byte cap,
    or only half of it, is sized for the rows that pass their term instead."""
    from helpers import gpu_ctx
    rng = np.random.default_rng(2)
    m, n = 300_000, 20_000
    build = {"k": rng.permutation(m).astype(np.int64), "y": rng.integers(0, 100, m).astype(np.int32)}
    probe = {"k": rng.integers(0, m, n).astype(np.int64)}
    c = gpu_ctx()   # a context of its own: no workspace left by larger queries
    try:
        tb, tp = c.load_table(build), c.load_table(probe)
        c.set_option("device_bytes_max", m * 12 + n * 8 + 65536 + room)
        r = c.run_join_select(tb, "k", [("y", rel.EQ, 7)], tp, "k", 0, [], [], [0, 1], agg=aiq.AGG_COUNT,
                              flags=aiq.FLAG_RELATIONAL_ONLY)
        row_of = np.full(m, -1)
        row_of[build["k"]] = np.arange(m)
        b = row_of[probe["k"]]
        want = np.flatnonzero(build["y"][b] == 7)
        assert np.array_equal(r.cand_row_ids, want) and np.array_equal(r.cand_build_rows, b[want])
    finally:
        c.close()


@pytest.mark.parametrize("m,n", [(1, 3), (40, 2047), (3000, 70_001), ((1 << 22) + 3, 20_000)])
def test_join_probe_sizes(ctx, m, n):
    """Build sides hashed straight from their columns and (the largest) compacted
    first; crowded tables, absent keys and the empty-slot sentinel among the probes."""
    rng = np.random.default_rng(m)
    keys = rng.permutation(np.arange(-(m // 2), m - m // 2, dtype=np.int64)) * 3
    build = {"k": keys, "y": rng.integers(0, 4, m).astype(np.int32)}
    probe = {"k": rng.integers(-2 * m - 2, 2 * m + 2, n).astype(np.int64), "a": rng.integers(0, 10, n).astype(np.int32)}
    probe["k"][::97] = -2**63
    tb, tp = ctx.load_table(build), ctx.load_table(probe)
    try:
        for bp, pp in [([], []), ([("y", rel.GE, 1)], [("a", rel.LT, 8)])]:
            r = ctx.run_join_select(tb, "k", bp, tp, "k", 0, pp, [], [0, 1], agg=aiq.AGG_COUNT,
                                    flags=aiq.FLAG_RELATIONAL_ONLY)
            ok_b = rel.predicate_mask(build, bp, m)
            order = np.argsort(keys)
            at = np.searchsorted(keys[order], probe["k"]).clip(0, m - 1)
            hit = order[at]
            sel = (keys[hit] == probe["k"]) & ok_b[hit] & rel.predicate_mask(probe, pp, n)
            assert np.array_equal(r.cand_row_ids, np.nonzero(sel)[0])
            assert np.array_equal(r.cand_build_rows, hit[sel])
    finally:
        ctx.free_table(tb)
        ctx.free_table(tp)


def test_join_small_with_orphans_and_repeats(ctx):
    rng = np.random.default_rng(3)
    m, n = 300, 5000
    keys = synth.distinct_int63(rng, m)
    keys[:3] = [-7, 0, 2**62]                      # negative / zero keys hash too
    build = synth.Table(m, {"k": keys, "year": rng.integers(1950, 2025, m).astype(np.int32)})
    fk = np.where(rng.random(n) < 0.8, keys[rng.integers(0, m, n)], rng.integers(0, 2**62, n))
    probe = synth.Table(n, {"k": fk.astype(np.int64), "a": rng.integers(0, 10, n).astype(np.int32)})
    tb, tp = ctx.load_table(build.cols, n_rows=m), ctx.load_table(probe.cols, n_rows=n)
    for bpreds, ppreds in [([], []), ([("year", rel.GE, 2010)], []), ([("year", rel.LT, 1990)], [("a", rel.GE, 5)])]:
        r = ctx.run_join_select(tb, "k", bpreds, tp, "k", 0, ppreds, [], [0, 1], agg=aiq.AGG_COUNT,
                                flags=aiq.FLAG_RELATIONAL_ONLY)
        cand, cand_b = oq.join_candidates(probe, build, "k", "k", ppreds, bpreds,
                                          brute_force=(bpreds == [] and ppreds == []))
        assert np.array_equal(r.cand_row_ids, cand)
        assert np.array_equal(r.cand_build_rows, cand_b)
    ctx.free_table(tb)
    ctx.free_table(tp)


def test_join_rejects_duplicate_and_sentinel_build_keys(ctx):
    for keys in ([5, 9, 5], [1, -2**63, 3]):
        build = ctx.load_table({"k": np.array(keys, np.int64)})
        probe = ctx.load_table({"k": np.array([5, 1], np.int64)})
        with pytest.raises(aiq.AiqError) as e:
            ctx.run_join_select(build, "k", [], probe, "k", 0, [], [], [0, 1], agg=aiq.AGG_COUNT,
                                flags=aiq.FLAG_RELATIONAL_ONLY)
        assert e.value.status == aiq.ERR_INVALID_ARG
        ctx.free_table(build)
        ctx.free_table(probe)
    # the context stays usable afterwards
    t = ctx.load_table({"a": np.arange(10, dtype=np.int32)})
    r = ctx.run_select(t, 0, [("a", rel.GE, 5)], [], [0, 1], flags=aiq.FLAG_RELATIONAL_ONLY)
    assert r.cand_row_ids.tolist() == [5, 6, 7, 8, 9]


# ------------------------------------------------------------ full query ---

def _model(ctx, shape, seed):
    W = synth.make_weights(shape, seed)
    return ctx.load_model(shape, weights_list(shape, W)), W


def _select_parity(ctx, w, budget=None):
    q = synth.make_inputs(w)
    mh, W = _model(ctx, w.model, w.weight_seed)
    t = _load(ctx, q.table)
    if budget:
        ctx.set_option("token_budget", budget)
    try:
        r = ctx.run_select(t, mh, oracle_preds(w.preds), q.prefix, w.label_ids, agg=w.agg, flags=aiq.FLAG_LOGITS)
    finally:
        ctx.set_option("token_budget", 131072)
    o = oq.run_select(q.table, q.prefix, oracle_preds(w.preds), w.label_ids, w.agg, tf.Model(w.model, W, True))
    assert np.array_equal(r.cand_row_ids, o.cand_rows)
    compare_logits(r.label_logits, o.logits, w.name)
    agg = oq.aggregate(w.agg, r.decisions, o.cand_rows, len(w.label_ids))
    if len(w.label_ids) == 2:
        assert r.count == agg["count"]
        assert np.array_equal(r.decisions, rel.decide(r.label_logits.astype(np.float64)))
    if w.agg == synth.AGG_ROW_IDS:
        assert np.array_equal(r.row_ids, agg["row_ids"])
    if w.agg == synth.AGG_GROUP_LABEL:
        assert np.array_equal(r.label_counts, agg["label_counts"])
    n_tok = sum(len(q.prefix) + len(q.table.text(i)) for i in o.cand_rows)
    assert r.n_tokens == n_tok
    if len(o.cand_rows):   # the shared prefix runs once; each row runs only its own tokens
        assert r.n_prefill_tokens == n_tok - len(q.prefix) * (len(o.cand_rows) - 1)
    ctx.free_table(t)
    ctx.free_model(mh)
    return r


def test_c1_tiny_select_full_parity(ctx):
    _select_parity(ctx, synth.C1_TINY)


def test_c1_chunking_is_invisible(ctx):
    w = synth.C1_TINY
    a = _select_parity(ctx, w)
    b = _select_parity(ctx, w, budget=130)   # every chunk holds a couple of rows
    assert b.n_chunks > 10
    assert np.array_equal(a.label_logits, b.label_logits)   # rows never interact: bit-identical


def test_two_term_mlp_activations(ctx):
    """mlp_split forced on for a small model (by default only models of 32
    layers and d 4096 load with it): the query still matches the oracle, on a
    tighter bound than the one-term path reaches, and its AI_TRANSFORM path
    (the decode loop's MLP GEMMs) runs too."""
    w = synth.C1_TINY
    gqa = replace(w.model, d_model=256, n_heads=8, n_kv_heads=2, head_dim=64, d_ffn=512)
    ctx.set_option("mlp_split", 1)
    try:
        for shape in (w.model, gqa):
            r = _select_parity(ctx, replace(w, model=shape))
            assert r.n_candidates > 0
        q = synth.make_inputs(w)
        mh, W = _model(ctx, gqa, w.weight_seed)
        t = _load(ctx, q.table)
        g = ctx.run_transform(t, mh, oracle_preds(w.preds), q.prefix, 3)
        assert g.n_candidates > 0 and g.gen_tokens.shape[1] == 3
        ctx.free_table(t)
        ctx.free_model(mh)
    finally:
        ctx.set_option("mlp_split", -1)


def test_tiny_row_ids_query(ctx):
    w = replace(synth.C2_SELECT, name="c2_tiny", n_rows=3000, model=synth.TINY,
                text=synth.TextRecipe("lognormal", 16, 200, median=60.0), prefix_len=32)
    _select_parity(ctx, w)


def test_tiny_multilabel_group_by(ctx):
    w = replace(synth.C4_MULTILABEL, name="c4_tiny", n_rows=2000, model=synth.TINY,
                text=synth.TextRecipe("lognormal", 32, 300, median=80.0), prefix_len=24)
    _select_parity(ctx, w)


def test_tiny_join_group_by_build_key(ctx):
    w = replace(synth.C3_JOIN, name="c3_tiny", n_rows=4000, join_build_rows=500, model=synth.TINY,
                text=synth.TextRecipe("lognormal", 16, 120, median=40.0), prefix_len=16)
    q = synth.make_inputs(w)
    mh, W = _model(ctx, w.model, w.weight_seed)
    tb, tp = _load(ctx, q.build), _load(ctx, q.table)
    bp = oracle_preds(w.join_build_preds)
    r = ctx.run_join_select(tb, "movie_id", bp, tp, "movie_id", mh, [], q.prefix, w.label_ids,
                            agg=synth.AGG_GROUP_BUILD_KEY, flags=aiq.FLAG_LOGITS)
    o = oq.run_join_select(q.table, q.build, "movie_id", "movie_id", [], bp, q.prefix, w.label_ids,
                           w.agg, tf.Model(w.model, W, True))
    assert np.array_equal(r.cand_row_ids, o.cand_rows)
    assert np.array_equal(r.cand_build_rows, o.cand_build_rows)
    compare_logits(r.label_logits, o.logits, w.name)
    agg = oq.aggregate(w.agg, r.decisions, o.cand_rows, 2, o.cand_build_rows, q.build.cols["movie_id"])
    assert np.array_equal(r.group_build_rows, agg["group_build_rows"])
    assert np.array_equal(r.group_keys, agg["group_keys"])
    assert np.array_equal(r.group_counts, agg["group_counts"])
    assert int(r.group_counts.sum()) == r.count


def test_rows_with_empty_text(ctx):
    """A row whose text is empty is decided on the prefix alone; with no prefix
    such a row's prompt would be empty, which is refused."""
    w = synth.C1_TINY
    q = synth.make_inputs(w)
    lens = np.diff(q.table.offsets)
    lens[::7] = 0                                   # every 7th row loses its text
    offsets = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    tokens = np.concatenate([q.table.text(i)[:lens[i]] for i in range(q.table.n_rows)]).astype(np.int32)
    table = synth.Table(q.table.n_rows, q.table.cols, offsets, tokens)
    mh, W = _model(ctx, w.model, w.weight_seed)
    t = _load(ctx, table)
    preds = oracle_preds(w.preds)
    r = ctx.run_select(t, mh, preds, q.prefix, w.label_ids, agg=w.agg, flags=aiq.FLAG_LOGITS)
    o = oq.run_select(table, q.prefix, preds, w.label_ids, w.agg, tf.Model(w.model, W, True))
    assert np.array_equal(r.cand_row_ids, o.cand_rows)
    compare_logits(r.label_logits, o.logits, "empty-text rows")
    empty = np.diff(offsets)[o.cand_rows] == 0
    assert empty.sum() > 5 and np.all(r.label_logits[empty] == r.label_logits[empty][0])
    with pytest.raises(aiq.AiqError) as e:
        ctx.run_select(t, mh, preds, np.zeros(0, np.int32), w.label_ids)
    assert e.value.status == aiq.ERR_INVALID_ARG
    ctx.free_table(t)
    ctx.free_model(mh)


@pytest.mark.parametrize("P", [1, 63, 65, 1024, 1025])
@pytest.mark.parametrize("gqa", [False, True])
def test_prefix_lengths_and_chunks(ctx, P, gqa):
    """The prefix as the first chunk's first sequence (up to 1024 tokens) and in a
    pass of its own, for both attention kernels, rows without text included: the
    oracle's logits, and the same bits whether the rows take one chunk or several."""
    w = synth.C1_TINY
    shape = replace(w.model, d_model=256, n_heads=8, n_kv_heads=2, head_dim=64, d_ffn=512) if gqa else w.model
    rng = np.random.default_rng(P)
    n = 40
    lens = rng.integers(0, 90, n)
    lens[[0, 7, 39]] = 0
    offsets = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    table = synth.Table(n, {"rating": np.ones(n, np.int32)}, offsets,
                        rng.integers(0, shape.vocab, int(offsets[-1])).astype(np.int32))
    prefix = rng.integers(0, shape.vocab, P).astype(np.int32)
    mh, W = _model(ctx, shape, w.weight_seed)
    t = _load(ctx, table)
    got = []
    try:
        for budget in (131072, max(P, 64) + 70):
            ctx.set_option("token_budget", budget)
            got.append(ctx.run_select(t, mh, [], prefix, w.label_ids, agg=w.agg, flags=aiq.FLAG_LOGITS))
    finally:
        ctx.set_option("token_budget", 131072)
    assert got[0].n_chunks == 1 and got[1].n_chunks > 1
    assert np.array_equal(got[0].label_logits, got[1].label_logits)
    o = oq.run_select(table, prefix, [], w.label_ids, w.agg, tf.Model(shape, W, True))
    compare_logits(got[0].label_logits, o.logits, f"prefix of {P}")
    ctx.free_table(t)
    ctx.free_model(mh)


@pytest.mark.parametrize("P,budget,chunks", [(0, 1024, 1), (63, 1024, 1), (64, 1024, 1), (65, 1024, 2), (960, 1024, 2),
                                             (961, 1024, 1), (64, 200, 8), (150, 200, 8)])
def test_prefix_counts_in_the_token_budget(ctx, P, budget, chunks):
    """The first chunk's tokens are within the budget, the prefix's among them: 15 rows
    of 64 tokens behind prefixes that just fit with them and just do not; a prefix
    that would fill a chunk takes a pass of its own.  The same logits as in one chunk."""
    w = synth.C1_TINY
    rng = np.random.default_rng(P)
    offsets = np.arange(16, dtype=np.int64) * 64
    table = synth.Table(15, {"rating": np.ones(15, np.int32)}, offsets,
                        rng.integers(0, w.model.vocab, 960).astype(np.int32))
    prefix = rng.integers(0, w.model.vocab, P).astype(np.int32)
    mh, _ = _model(ctx, w.model, w.weight_seed)
    t = _load(ctx, table)
    got = []
    try:
        for b in (131072, budget):
            ctx.set_option("token_budget", b)
            got.append(ctx.run_select(t, mh, [], prefix, w.label_ids, agg=w.agg, flags=aiq.FLAG_LOGITS))
    finally:
        ctx.set_option("token_budget", 131072)
    assert [r.n_chunks for r in got] == [1, chunks]
    assert np.array_equal(got[0].label_logits, got[1].label_logits)
    # with the rows, the prefix's final layer runs its output projection and MLP for one token only
    d, f, step = w.model.d_model, w.model.d_ffn, budget - 63
    alone = max(P - 1, 0) * 2 * (d * d + 3 * d * f)
    assert got[1].prefill_flops - got[0].prefill_flops == (alone if P >= step else 0)
    ctx.free_table(t)
    ctx.free_model(mh)


def test_row_plan_sizes(ctx):
    """Up to 8192 rows one block measures and places the rows' texts, above that a
    chain of kernels: token counts, work counts and logits agree on both sides, at
    the edges of a thread's four rows and of a block's 4096."""
    w = synth.C1_TINY
    rng = np.random.default_rng(8)
    n = 8193
    lens = rng.integers(0, 10, n)
    lens[[0, 1, n - 1]] = [0, 3, 0]
    offsets = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    table = synth.Table(n, {"rating": np.arange(n, dtype=np.int32)}, offsets,
                        rng.integers(0, w.model.vocab, int(offsets[-1])).astype(np.int32))
    prefix = rng.integers(0, w.model.vocab, 17).astype(np.int32)
    mh, _ = _model(ctx, w.model, w.weight_seed)
    t = _load(ctx, table)
    run = lambda k: ctx.run_select(t, mh, [("rating", rel.LT, k)], prefix, w.label_ids, flags=aiq.FLAG_LOGITS)
    all_rows = run(n)
    for k in (1, 2, 4, 5, 4095, 4096, 4097, 8192):
        r = run(k)
        assert r.n_candidates == k and r.n_tokens == 17 * k + offsets[k]
        assert np.array_equal(r.label_logits, all_rows.label_logits[:k]), k
    # the last row has no text: the same tokens and attention pairs, and one row more in what
    # runs on last tokens alone (the final layer's output projection and MLP, the label scores)
    d, f = w.model.d_model, w.model.d_ffn
    assert all_rows.prefill_flops - r.prefill_flops == 2 * (d * d + 3 * d * f) + 2 * d * len(w.label_ids)
    ctx.free_table(t)
    ctx.free_model(mh)


def test_more_rows_than_tokens():
    """A chunk whose rows are all but a few without text has more rows than
    tokens: the per-row buffers are sized for the rows."""
    from helpers import gpu_ctx
    w = synth.C1_TINY
    q = synth.make_inputs(w)
    n = q.table.n_rows
    lens = np.zeros(n, np.int64)
    lens[[3, 200, 311]] = [2, 5, 1]
    offsets = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    table = synth.Table(n, q.table.cols, offsets, np.arange(8, dtype=np.int32))
    c = gpu_ctx()   # a context of its own: no workspace left by larger queries
    try:
        mh, W = _model(c, w.model, w.weight_seed)
        t = _load(c, table)
        r = c.run_select(t, mh, [], q.prefix, w.label_ids, agg=w.agg, flags=aiq.FLAG_LOGITS)
        o = oq.run_select(table, q.prefix, [], w.label_ids, w.agg, tf.Model(w.model, W, True))
        assert np.array_equal(r.cand_row_ids, o.cand_rows) and r.n_candidates == n
        compare_logits(r.label_logits, o.logits, "more rows than tokens")
        assert np.all(r.label_logits[lens == 0] == r.label_logits[0])
        g = c.run_transform(t, mh, [], q.prefix, 3)
        assert np.all(g.gen_tokens[lens == 0] == g.gen_tokens[0])
    finally:
        c.close()


def test_degenerate_queries(ctx):
    w = synth.C1_TINY
    q = synth.make_inputs(w)
    mh, W = _model(ctx, w.model, w.weight_seed)
    t = _load(ctx, q.table)
    # no row survives: empty results, count 0
    r = ctx.run_select(t, mh, [("rating", rel.GT, 5)], q.prefix, w.label_ids, agg=synth.AGG_ROW_IDS)
    assert r.n_candidates == 0 and r.count == 0 and r.row_ids.size == 0
    # empty prefix and a single row
    r = ctx.run_select(t, mh, [("rating", rel.EQ, 3)], np.zeros(0, np.int32), w.label_ids,
                       agg=synth.AGG_COUNT, flags=aiq.FLAG_LOGITS)
    o = oq.run_select(q.table, np.zeros(0, np.int32), [("rating", rel.EQ, 3)], w.label_ids, w.agg,
                      tf.Model(w.model, W, True))
    compare_logits(r.label_logits, o.logits, "no prefix")
    # invalid inputs are rejected with a status, not a fault
    for kw in [dict(labels=[100, 5000]), dict(prefix=[4096])]:
        with pytest.raises(aiq.AiqError) as e:
            ctx.run_select(t, mh, [], kw.get("prefix", q.prefix), kw.get("labels", w.label_ids))
        assert e.value.status == aiq.ERR_INVALID_ARG
    with pytest.raises(aiq.AiqError) as e:
        ctx.run_select(t, 12345, [], q.prefix, w.label_ids)
    assert e.value.status == aiq.ERR_NOT_FOUND
    ctx.free_table(t)
    ctx.free_model(mh)


def test_sum_aggregate_matches_oracle_on_gpu_decisions(ctx):
    """Fig. 2's SELECT SUM(values) ... WHERE AI_IF(...) = 1: integer sums exact,
    the float sum within fp64 rounding of the correctly rounded sum."""
    w = synth.C1_TINY
    q = synth.make_inputs(w)
    W = synth.make_weights(w.model, w.weight_seed)
    rng = np.random.default_rng(17)
    n = q.table.n_rows
    cols = dict(q.table.cols)
    cols["v32"] = rng.integers(-2 ** 31, 2 ** 31 - 1, n).astype(np.int32)
    cols["v64"] = rng.integers(-2 ** 50, 2 ** 50, n).astype(np.int64)
    cols["vf"] = (rng.standard_normal(n) * 1e3).astype(np.float32)
    m = ctx.load_model(w.model, weights_list(w.model, W))
    t = ctx.load_table(cols, (q.table.offsets, q.table.tokens))
    preds = oracle_preds(w.preds)
    for name in ("v32", "v64", "vf"):
        r = ctx.run_select(t, m, preds, q.prefix, w.label_ids, agg=aiq.AGG_SUM, flags=aiq.FLAG_LOGITS,
                           sum_column=name)
        want = rel.masked_sum(r.decisions, r.cand_row_ids, cols[name])
        assert r.count == rel.count_yes(r.decisions)
        if name == "vf":
            bound = 1e-12 * float(np.abs(cols[name]).astype(np.float64).sum())
            assert abs(r.sum - want) <= bound, (r.sum, want)
        else:
            assert r.sum == want
    e = ctx.run_select(t, m, [("rating", rel.GT, 100)], q.prefix, w.label_ids, agg=aiq.AGG_SUM, sum_column="v64")
    assert e.count == 0 and e.sum == 0
    with pytest.raises(aiq.AiqError):
        ctx.run_select(t, m, preds, q.prefix, w.label_ids, agg=aiq.AGG_SUM, sum_column="text")
    ctx.free_table(t)
    ctx.free_model(m)
