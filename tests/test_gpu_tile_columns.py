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
