"""Row counts at which a bf16 tile of the CTA-pair kernel changes shape: the accumulator's columns go in steps of 16, half of
them per CTA, the boxes that load a down tile's rows are 8, 32 or 128 high, the epilogue takes 32 tokens at a time."""
import numpy as np
import pytest
import torch

import oracle
import paper_2607_18002_b200 as moe
from workloads import synth

from gpu_util import assert_close, bind_ops, make_ctx, oracle_weights, weights_to

pytestmark = pytest.mark.gpu

COUNTS = [1, 7, 8, 9, 15, 16, 17, 31, 32, 33, 48, 63, 64, 65, 80, 95, 96, 97, 127, 128, 129, 143, 144, 145, 159, 160, 161,
          191, 192, 193, 207, 208, 209, 223, 224, 225, 239, 240, 241, 254, 255, 256, 257, 272, 0, 289]


@pytest.mark.parametrize("layout", ["gathered", "masked"])
def test_every_tile_shape_matches_oracle(layout):
    E, H, I = len(COUNTS), 512, 256
    ids = np.random.default_rng(9).permutation(np.repeat(np.arange(E), COUNTS)).astype(np.int32).reshape(-1, 1)
    T = ids.shape[0]
    spec = synth.Spec("cols", synth.Shape(E, 1, H, I), ((synth.PREFILL, T),), "uniform", None, 1.0, -1.0, 61)
    W = synth.make_weights(spec)
    Wd, OW = weights_to(W), oracle_weights(spec, W)
    if layout == "gathered":
        x, _ = synth.make_x(spec, T, 0, 0)
        op = synth.Op(synth.PREFILL, x, ids, np.ones(ids.shape, np.float32))
        ctx = make_ctx(spec)
        b = bind_ops(ctx, [op], Wd)[0]
        ctx.plan(0, b)
        ctx.run([0], fuse_combine=True)
        ctx.check()
        assert_close(b.y.float().cpu().numpy(), oracle.forward(OW, x, None, ids, op.w)["y"])
        return
    slab = 296
    x, _ = synth.make_x(spec, E * slab, 0, 0)
    ctx = make_ctx(spec, max_tokens=E * slab)
    b = moe.bind_masked_op(moe.MOE_CLASS_DECODE, x.view(E, slab, H).cuda(), torch.tensor(COUNTS, dtype=torch.int32).cuda(),
                           Wd.w_gate_up, Wd.w_down)
    ctx.plan(0, b)
    ctx.run([0], fuse_combine=True)
    ctx.check()
    rows_e = np.repeat(np.arange(E), COUNTS).astype(np.int32)
    flat = rows_e * slab + np.concatenate([np.arange(c) for c in COUNTS]).astype(np.int32)
    y = b.y.float().cpu().numpy().reshape(E * slab, H)
    assert_close(y[flat], oracle.ffn_rows(OW, x, None, flat, rows_e))
    untouched = np.ones(E * slab, dtype=bool)
    untouched[flat] = False
    assert np.all(y[untouched] == 0.0)


@pytest.mark.parametrize("T", [1, 15, 31, 32, 33, 64, 127, 128, 129])
def test_small_ops_on_their_deeper_pipelines(T):
    """Ops of up to 32 and up to 128 tokens run with smaller work tiles and more stages.  Tokens may name an expert several times, so
    an expert can still get more rows than the op has tokens: its rows are then cut into several work tiles."""
    E, k, H, I = 6, 4, 512, 256
    spec = synth.Spec("deep", synth.Shape(E, k, H, I), ((synth.DECODE, T),), "uniform", None, 1.0, -1.0, 62)
    W = synth.make_weights(spec)
    rng = np.random.default_rng(T)
    ids = rng.integers(0, E, size=(T, k)).astype(np.int32)
    ids[: T // 2] = 5                                                # half of the tokens name one expert k times
    x, _ = synth.make_x(spec, T, 0, 0)
    op = synth.Op(synth.DECODE, x, ids, rng.random((T, k), dtype=np.float32))
    ctx = make_ctx(spec)
    b = bind_ops(ctx, [op], weights_to(W))[0]
    for fuse in (True, False):
        b.y.fill_(7.0)
        ctx.plan(0, b)
        ctx.run([0], fuse_combine=fuse)
        if not fuse:
            ctx.combine(0)
        ctx.check()
        assert_close(b.y.float().cpu().numpy(), oracle.forward(oracle_weights(spec, W), x, None, ids, op.w)["y"])


@pytest.mark.parametrize("slab", [8, 32, 33, 128, 129])
def test_masked_slabs_on_the_deeper_pipelines(slab):
    E, H, I = 6, 512, 256
    counts = np.array([0, 1, slab // 2, slab - 1, slab, slab], dtype=np.int32)
    spec = synth.Spec("deepm", synth.Shape(E, 1, H, I), ((synth.DECODE, 1),), "uniform", None, 1.0, -1.0, 63)
    W = synth.make_weights(spec)
    x, _ = synth.make_x(spec, E * slab, 0, 0)
    Wd = weights_to(W)
    ctx = make_ctx(spec, max_tokens=E * slab)
    b = moe.bind_masked_op(moe.MOE_CLASS_DECODE, x.view(E, slab, H).cuda(), torch.from_numpy(counts).cuda(), Wd.w_gate_up, Wd.w_down)
    ctx.plan(0, b)
    ctx.run([0], fuse_combine=True)
    ctx.check()
    rows_e = np.repeat(np.arange(E), counts).astype(np.int32)
    flat = rows_e * slab + np.concatenate([np.arange(c) for c in counts]).astype(np.int32)
    y = b.y.float().cpu().numpy().reshape(E * slab, H)
    assert_close(y[flat], oracle.ffn_rows(oracle_weights(spec, W), x, None, flat, rows_e))
    y[flat] = 0.0
    assert np.all(y == 0.0)


@pytest.mark.parametrize("T,I", [(t, i) for t in (1, 24, 90, 180, 250) for i in (128, 768, 1536)])
def test_down_tiles_that_wait_for_their_rows(T, I):
    """Few tiles on many units: every down tile is handed over before its gate/up tiles are done, and its weights wait in the
    stages -- fewer k-blocks than the pipeline has stages, and more -- for activation rows of one to three boxes."""
    E, H = 2, 256
    spec = synth.Spec("wait", synth.Shape(E, 1, H, I), ((synth.DECODE, T),), "uniform", None, 1.0, -1.0, 64)
    W = synth.make_weights(spec)
    ids = (np.arange(T) == 0).astype(np.int32).reshape(-1, 1)        # expert 1 has one row, expert 0 the others
    x, _ = synth.make_x(spec, T, 0, 0)
    op = synth.Op(synth.DECODE, x, ids, np.ones(ids.shape, np.float32))
    ctx = make_ctx(spec)
    b = bind_ops(ctx, [op], weights_to(W))[0]
    ref = oracle.forward(oracle_weights(spec, W), x, None, ids, op.w)["y"]
    for _ in range(3):
        b.y.fill_(7.0)
        ctx.plan(0, b)
        ctx.run([0], fuse_combine=True)
        ctx.check()
        assert_close(b.y.float().cpu().numpy(), ref)
