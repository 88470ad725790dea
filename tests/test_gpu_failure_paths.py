"""Failure paths reported as statuses, with no GPU fault: the context's device
byte cap (AIQ_ERR_OOM), a weight outside the fp16 operand range
(AIQ_ERR_UNSUPPORTED at load), and an activation that leaves the fp16 range
inside the forward pass (the kernels' own range check sets the device error
word: AIQ_ERR_DEVICE_CHECK).  After each failure the same context answers the
normal query exactly as a fresh context does.

The overflowing activation is an ordinary input (embedding rows of 1e5, a
bf16 value), not a fault: every kernel it passes through only does arithmetic
on it; no index, loop bound or wait depends on activation values, and the
decision of a NaN logit pair is "no" (a strict comparison)."""
import os

import numpy as np
import pytest

import synth
from helpers import gpu_ctx, weights_list
from paper_2608_10139_gb300 import aiq

pytestmark = pytest.mark.gpu

W_TINY = synth.C1_TINY


@pytest.fixture(scope="module")
def inputs():
    q = synth.make_inputs(W_TINY)
    W = synth.make_weights(W_TINY.model, W_TINY.weight_seed)
    return q, W


def _query(ctx, q, W, weights=None):
    t = ctx.load_table(q.table.cols, (q.table.offsets, q.table.tokens))
    m = None
    try:
        m = ctx.load_model(W_TINY.model, weights_list(W_TINY.model, weights if weights is not None else W))
        preds = [(p.column, p.op, p.value) for p in W_TINY.preds]
        return ctx.run_select(t, m, preds, q.prefix, W_TINY.label_ids, agg=aiq.AGG_ROW_IDS,
                              flags=aiq.FLAG_LOGITS)
    finally:
        if m is not None:
            ctx.free_model(m)
        ctx.free_table(t)


@pytest.fixture(scope="module")
def fresh(inputs):
    c = gpu_ctx()
    try:
        yield _query(c, *inputs)
    finally:
        c.close()


def _same(a, b):
    assert a.count == b.count and np.array_equal(a.row_ids, b.row_ids)
    assert np.array_equal(a.cand_row_ids, b.cand_row_ids)
    assert np.array_equal(a.label_logits, b.label_logits)


def test_byte_cap_option_gives_oom_then_the_context_recovers(inputs, fresh):
    ctx = gpu_ctx()
    try:
        q, W = inputs
        t = ctx.load_table(q.table.cols, (q.table.offsets, q.table.tokens))
        m = ctx.load_model(W_TINY.model, weights_list(W_TINY.model, W))
        preds = [(p.column, p.op, p.value) for p in W_TINY.preds]
        ctx.set_option("device_bytes_max", 1)           # below what the table and model hold
        for _ in range(2):
            with pytest.raises(aiq.AiqError) as e:
                ctx.run_select(t, m, preds, q.prefix, W_TINY.label_ids, agg=aiq.AGG_ROW_IDS, flags=aiq.FLAG_LOGITS)
            assert e.value.status == aiq.ERR_OOM and "AIQ_DEVICE_BYTES_MAX" in str(e.value)
        ctx.set_option("device_bytes_max", 0)           # lift the cap
        r = ctx.run_select(t, m, preds, q.prefix, W_TINY.label_ids, agg=aiq.AGG_ROW_IDS, flags=aiq.FLAG_LOGITS)
        _same(r, fresh)
        ctx.free_model(m)
        ctx.free_table(t)
    finally:
        ctx.close()


def test_byte_cap_from_the_environment(inputs, fresh):
    q, W = inputs
    old = os.environ.get("AIQ_DEVICE_BYTES_MAX")
    os.environ["AIQ_DEVICE_BYTES_MAX"] = "4096"
    try:
        ctx = gpu_ctx()
    finally:
        if old is None:
            del os.environ["AIQ_DEVICE_BYTES_MAX"]
        else:
            os.environ["AIQ_DEVICE_BYTES_MAX"] = old
    try:
        with pytest.raises(aiq.AiqError) as e:
            ctx.load_table(q.table.cols, (q.table.offsets, q.table.tokens))
        assert e.value.status == aiq.ERR_OOM
        ctx.set_option("device_bytes_max", 0)
        _same(_query(ctx, q, W), fresh)
    finally:
        ctx.close()


def test_weight_outside_the_fp16_range_is_rejected_at_load(inputs, fresh):
    q, W = inputs
    bad = dict(W)
    wq = W["l1.wq"].copy()
    wq[3, 5] = synth.f32_to_bf16_bits(np.array([-1.0e5], np.float32))[0]   # |w| > 65504
    bad["l1.wq"] = wq
    ctx = gpu_ctx()
    try:
        with pytest.raises(aiq.AiqError) as e:
            ctx.load_model(W_TINY.model, weights_list(W_TINY.model, bad))
        assert e.value.status == aiq.ERR_UNSUPPORTED and "fp16 range" in str(e.value)
        _same(_query(ctx, q, W), fresh)
    finally:
        ctx.close()


def test_activation_overflow_is_reported_then_the_context_recovers(inputs, fresh):
    q, W = inputs
    bad = dict(W)
    emb = W["embed"].copy()
    # every prefix token's embedding row at 1e5: the residual stream's fp16
    # copy (the operand of the first QKV GEMM) cannot hold it
    emb[np.unique(q.prefix)] = synth.f32_to_bf16_bits(np.array([1.0e5], np.float32))[0]
    bad["embed"] = emb
    ctx = gpu_ctx()
    try:
        for _ in range(2):
            with pytest.raises(aiq.AiqError) as e:
                _query(ctx, q, W, bad)
            assert e.value.status == aiq.ERR_DEVICE_CHECK and "fp16 range" in str(e.value)
        _same(_query(ctx, q, W), fresh)
    finally:
        ctx.close()


def test_refused_transforms_hold_no_more_memory(inputs):
    """A transform refused for want of room keeps nothing that it made half of: under a
    cap that rises by 8 KB a try (less than any buffer of the full-vocabulary head, so
    that some tries get its first and not its second), it runs once the cap reaches
    what it needs."""
    q, W = inputs
    c = gpu_ctx()
    try:
        t = c.load_table(q.table.cols, (q.table.offsets, q.table.tokens))
        m = c.load_model(W_TINY.model, weights_list(W_TINY.model, W))
        for cap in range(1 << 20, 64 << 20, 8 << 10):
            c.set_option("device_bytes_max", cap)
            try:
                c.run_transform(t, m, [("rating", aiq.GE, 5)], q.prefix, 2)
                return
            except aiq.AiqError as e:
                assert e.status == aiq.ERR_OOM
        pytest.fail("64 MB were not enough for a transform of 15 MB")
    finally:
        c.close()


def test_room_of_a_failed_joins_table(inputs):
    """A join that fails (a repeated build key) leaves its table (15.7 MB) behind; a
    transform under a cap that needs the table's room takes it back."""
    q, W = inputs
    m = 300_000
    keys = np.arange(m, dtype=np.int64)
    keys[-1] = 0

    def context():
        c = gpu_ctx()
        text = c.load_table(q.table.cols, (q.table.offsets, q.table.tokens))
        build, probe = c.load_table({"k": keys}), c.load_table({"k": keys[:1000]})
        return c, text, build, probe, c.load_model(W_TINY.model, weights_list(W_TINY.model, W))

    def transform(c, text, model, cap):
        c.set_option("device_bytes_max", cap)
        return c.run_transform(text, model, [("rating", aiq.GE, 5)], q.prefix, 2)

    c, text, _, _, model = context()
    try:
        loaded = sum(v.nbytes for v in (*q.table.cols.values(), q.table.offsets, q.table.tokens, keys, *weights_list(W_TINY.model, W)))
        for cap in range(loaded, loaded + (1 << 30), 1 << 20):   # the least room it runs in, to 1 MB
            try:
                want = transform(c, text, model, cap)
                break
            except aiq.AiqError as e:
                assert e.status == aiq.ERR_OOM
    finally:
        c.close()
    c, text, build, probe, model = context()
    try:
        with pytest.raises(aiq.AiqError) as e:
            c.run_join_select(build, "k", [], probe, "k", 0, [], [], [0, 1], agg=aiq.AGG_COUNT,
                              flags=aiq.FLAG_RELATIONAL_ONLY)
        assert e.value.status == aiq.ERR_INVALID_ARG
        got = transform(c, text, model, cap + (1 << 20))
        assert np.array_equal(got.gen_tokens, want.gen_tokens)
    finally:
        c.close()


def test_query_runs_in_the_room_that_it_needs(inputs):
    """A query whose prefix would run with the first chunk (2,088 tokens of 2,216) fits
    where it does with a pass of its own (1,216 tokens at a time): the sum of that
    route's buffers, whatever smaller caps were tried before."""
    _, W = inputs
    g, P, n, L = W_TINY.model, 1000, 19, 64
    rng = np.random.default_rng(4)
    T, offsets = n * L, np.arange(n + 1, dtype=np.int64) * L
    tokens = rng.integers(0, g.vocab, T).astype(np.int32)
    prefix = rng.integers(0, g.vocab, P).astype(np.int32)
    d, qd, kd, f = g.d_model, g.n_heads * g.head_dim, g.n_kv_heads * g.head_dim, g.d_ffn
    per_token = 4 * 4 + 4 * d + 2 * d + 2 * (qd + 2 * kd) + 2 * qd + 2 * f + 4 * (d // 128)
    need = T * per_token + g.n_layers * P * 2 * kd * 2 + 2 * 4 * 2048 * (g.head_dim // 2)   # with the RoPE tables
    small = 64 << 10   # per-row buffers, work lists, 256 bytes at least for each
    want = None
    for tries in ([], [2.0, 0.5], [0.3, 0.6, 0.9, 0.95]):   # of the room, before
        c = gpu_ctx()
        try:
            t = c.load_table({"rating": np.ones(n, np.int32)}, (offsets, tokens))
            m = c.load_model(g, weights_list(g, W))
            c.set_option("token_budget", 2100)
            run = lambda: c.run_select(t, m, [], prefix, W_TINY.label_ids, flags=aiq.FLAG_LOGITS)  # noqa: E731
            c.set_option("device_bytes_max", 1)
            with pytest.raises(aiq.AiqError) as e:
                run()
            held = int(str(e.value).split("(")[1].split()[0]) - 256   # "(held + asked for > cap)"
            for part in tries:
                c.set_option("device_bytes_max", held + int(part * need))
                try:
                    run()
                except aiq.AiqError as e:
                    assert e.status == aiq.ERR_OOM and part < 1
            c.set_option("device_bytes_max", held + need + small)
            r = run()
            assert want is None or np.array_equal(r.label_logits, want)
            want = r.label_logits
        finally:
            c.close()


def test_loads_take_back_a_joins_room(inputs):
    """After a join (a table of 15.7 MB for 300,000 build rows) a table and a model load
    under a cap that has room for them and not for what the join left behind."""
    _, W = inputs
    c = gpu_ctx()
    try:
        keys = np.arange(300_000, dtype=np.int64)
        build, probe = c.load_table({"k": keys}), c.load_table({"k": keys[:1000]})
        c.run_join_select(build, "k", [], probe, "k", 0, [], [], [0, 1], agg=aiq.AGG_COUNT, flags=aiq.FLAG_RELATIONAL_ONLY)
        held = keys.nbytes + 8000
        c.set_option("device_bytes_max", held + keys.nbytes + (64 << 10))
        t = c.load_table({"k": keys})
        c.free_table(t)
        r = c.run_join_select(build, "k", [("k", aiq.LT, 10)], probe, "k", 0, [], [], [0, 1], agg=aiq.AGG_COUNT,
                              flags=aiq.FLAG_RELATIONAL_ONLY)
        assert np.array_equal(r.cand_row_ids, np.arange(10))
        c.set_option("device_bytes_max", 0)
        c.run_join_select(build, "k", [], probe, "k", 0, [], [], [0, 1], agg=aiq.AGG_COUNT, flags=aiq.FLAG_RELATIONAL_ONLY)
        c.set_option("device_bytes_max", held + (12 << 20))
        c.free_model(c.load_model(W_TINY.model, weights_list(W_TINY.model, W)))
    finally:
        c.close()
