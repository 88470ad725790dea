"""Bits that a change of kernels is not to move.

A sum formed in another order is as good a sum, but one fp16 rounding that it
flips travels through every later layer, so that a program comparing its logits
with yesterday's sees all of them differ.  The checksums below are of the
outputs that the first kernels of this library gave on the same inputs; every
kernel that took their place since keeps their order of summation."""
import zlib
from dataclasses import replace

import numpy as np
import pytest

import synth
from helpers import gpu_ctx, weights_list
from paper_2608_10139_gb300 import aiq

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = gpu_ctx()
    yield c
    c.close()


def _crc(a):
    a = a.cpu().numpy() if isinstance(a, torch.Tensor) else a
    return zlib.crc32(np.ascontiguousarray(a).tobytes())


def rmsnorm_crc(ctx, d):
    """Rows enough for both RMSNorm kernels (a warp per row, and up to 2432 rows a
    block per row), the second run on the first's leading rows."""
    rng = np.random.default_rng(d)
    T = 4000
    x = torch.from_numpy((rng.standard_normal((T, d)) * 3).astype(np.float32)).cuda()
    g = synth.f32_to_bf16_bits((1 + 0.02 * rng.standard_normal(d)).astype(np.float32))
    g = torch.from_numpy(g.view(np.int16)).cuda()
    crcs = []
    for n in (T, 2000):
        out = torch.zeros((n, d), dtype=torch.float16, device="cuda")
        torch.cuda.synchronize()
        ctx.op_rmsnorm(x.data_ptr(), n, d, g.data_ptr(), 1e-5, out.data_ptr())
        torch.cuda.synchronize()
        crcs.append(_crc(out))
    return tuple(crcs)


RMSNORM = {128: (3904390063, 2493164157), 256: (3067552901, 692534954), 512: (1052675502, 2626568877),
           768: (3262264995, 1646734802), 1024: (3444412211, 2397995067), 2048: (2797889848, 2232699657),
           4096: (2969633955, 1237979846)}


@pytest.mark.parametrize("d", [128, 256, 512, 768, 1024, 2048, 4096])
def test_rmsnorm_bits(ctx, d):
    assert rmsnorm_crc(ctx, d) == RMSNORM[d]


SHAPES = {"one layer": replace(synth.C1_TINY.model, n_layers=1),
          "one wide layer": replace(synth.C1_TINY.model, n_layers=1, d_model=1152, d_ffn=256),
          "tiny": synth.C1_TINY.model,
          "grouped": replace(synth.C1_TINY.model, n_layers=3, d_model=512, n_heads=8, n_kv_heads=2, head_dim=64, d_ffn=1024)}
BUDGETS = (131072, 4000, 300)   # tokens: one chunk of some 16,000, several, chunks of a few rows


def logits_crc(ctx, shape, budget, k):
    w = synth.C1_TINY
    q = synth.make_inputs(w)
    W = synth.make_weights(SHAPES[shape], w.weight_seed)
    m = ctx.load_model(SHAPES[shape], weights_list(SHAPES[shape], W))
    t = ctx.load_table(q.table.cols, (q.table.offsets, q.table.tokens))
    try:
        ctx.set_option("token_budget", budget)
        return _crc(ctx.run_select(t, m, [], q.prefix, [100, 101, 77][:k], agg=aiq.AGG_GROUP_LABEL,
                                   flags=aiq.FLAG_LOGITS).label_logits)
    finally:
        ctx.set_option("token_budget", 131072)
        ctx.free_table(t)
        ctx.free_model(m)


LOGITS = {("one layer", 2): 903127134, ("one layer", 3): 2015117514,
          ("one wide layer", 2): 878337199, ("one wide layer", 3): 1545911119,
          ("tiny", 2): 4004519680, ("tiny", 3): 843533209,
          ("grouped", 2): 665073265, ("grouped", 3): 355354920}


@pytest.mark.parametrize("budget", BUDGETS)
@pytest.mark.parametrize("shape", SHAPES)
def test_query_logits_bits(ctx, shape, budget):
    for k in (2, 3):   # labels
        assert logits_crc(ctx, shape, budget, k) == LOGITS[shape, k]
