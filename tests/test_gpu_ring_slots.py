"""Tiles so short that the four descriptor slots of a pair go round every few microseconds, on each form of the pair kernel (32, 128
and 256 rows a tile), launch after launch: a descriptor that is overwritten before every role has read it shows in the outputs."""
import numpy as np
import pytest
import torch

import oracle
from workloads import synth

from gpu_util import assert_close, bind_ops, make_ctx, oracle_weights, weights_to

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T", [1, 31, 33, 129, 700])
@pytest.mark.parametrize("n_ctas", [0, 2, 6])
def test_short_tiles_one_after_the_other(T, n_ctas):
    spec = synth.Spec("ring", synth.Shape(256, 4, 256, 128, "bf16"), ((synth.DECODE, T),), "zipf", 1.0, 1.0, -1.0, 97)
    W = synth.make_weights(spec)
    ctx = make_ctx(spec, n_ctas=n_ctas)
    assert ctx.ctas_per_tile == 2
    op = synth.make_ops(spec)[0]
    b = bind_ops(ctx, [op], weights_to(W))[0]
    ctx.plan(0, b)
    ctx.run([0], fuse_combine=True)
    ctx.check()
    first = b.y.clone()
    assert_close(first.float().cpu().numpy(), np.asarray(oracle.forward(oracle_weights(spec, W), op.x, None, op.ids, op.w)["y"]))
    for _ in range(20):
        b.y.fill_(7.0)
        ctx.run([0], fuse_combine=True)
        assert torch.equal(b.y, first)
    ctx.check()
