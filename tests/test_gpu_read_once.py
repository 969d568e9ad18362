"""Entries of experts with one work tile carry a mark beside the expert id: the largest ids, experts with one and with several tiles in one
launch, of an op by itself and of a pair (where an expert's tiles lie in two lists)."""
import numpy as np
import pytest

import oracle
from workloads import synth

from gpu_util import assert_close, bind_ops, make_ctx, oracle_weights, weights_to

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_ctas", [0, 3], ids=["pairs", "single"])
def test_experts_of_one_and_of_several_tiles(n_ctas):
    E, k = 1024, 4
    spec = synth.Spec("once", synth.Shape(E, k, 256, 128, "bf16"), ((synth.PREFILL, 700), (synth.DECODE, 40)), "zipf", 1.0, 1.0, -1.0, 91)
    W = synth.make_weights(spec)
    ops = synth.make_ops(spec)
    for o in ops:                                   # every token meets expert 1023, every other one expert 0, and two of the others
        t = np.arange(len(o.ids))
        o.ids[:, 0] = E - 1
        o.ids[:, 1] = np.where(t % 2 == 0, 0, 1 + 2 * (t % 500))
        o.ids[:, 2] = 2 + 2 * ((17 * t) % 500)
        o.ids[:, 3] = 2 + 2 * ((17 * t + 250) % 500)
    OW = oracle_weights(spec, W)
    want = [np.asarray(oracle.forward(OW, o.x, None, o.ids, o.w)["y"]) for o in ops]
    ctx = make_ctx(spec, max_tokens=740, n_ctas=n_ctas)
    bound = bind_ops(ctx, ops, weights_to(W))
    for pair in (False, True):
        for s, b in enumerate(bound):
            b.y.fill_(7.0)
            ctx.plan(s, b)
        if pair:
            ctx.plan_pair(0, 1)
        ctx.run([0, 1], fuse_combine=True)
        ctx.check()
        for b, y in zip(bound, want):
            assert_close(b.y.float().cpu().numpy(), y)
