"""Combine tiles of one to four tokens: one or two are shared by columns between the CTAs of a pair, more by tokens; rows narrower than the
threads, rows that are no multiple of a thread group, few and many slots.  The fused combine, the stand-alone one and the oracle."""
import numpy as np
import pytest
import torch

import oracle
from workloads import synth

from gpu_util import assert_close, bind_ops, make_ctx, oracle_weights, weights_to

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_ctas", [0, 3], ids=["pairs", "single"])
@pytest.mark.parametrize("H,k", [(256, 2), (256, 12), (768, 8), (1280, 3)])
def test_small_combine_tiles(H, k, n_ctas):
    sizes = (1, 2, 3, 4, 5, 6, 15)
    spec = synth.Spec("columns", synth.Shape(16, k, H, 128, "bf16"), tuple((synth.DECODE, T) for T in sizes), "zipf", 1.0, 1.0, -1.0, 77)
    W = synth.make_weights(spec)
    ctx = make_ctx(spec, max_tokens=max(sizes), max_ops=1, n_ctas=n_ctas)
    OW = oracle_weights(spec, W)
    ops = synth.make_ops(spec)
    for b, o in zip(bind_ops(ctx, ops, weights_to(W)), ops):
        b.y.fill_(7.0)
        ctx.plan(0, b)
        ctx.run([0], fuse_combine=True)
        ctx.check()
        fused = b.y.clone()
        b.y.fill_(7.0)
        ctx.run([0])
        ctx.combine(0)
        ctx.check()
        assert torch.equal(fused, b.y)
        assert_close(fused.float().cpu().numpy(), np.asarray(oracle.forward(OW, o.x, None, o.ids, o.w)["y"]))
