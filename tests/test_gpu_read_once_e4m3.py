"""The mark beside the expert id on the e4m3 kernel, which takes the weights' scales by that id: experts with one work tile and with several,
the largest ids, on both forms of the kernel (work tiles of 64 and of 128 rows), and as a pair."""
import numpy as np
import pytest

import oracle
from workloads import synth

from gpu_util import REL_L2_8, RTOL8, assert_close, bind_ops, make_ctx, oracle_weights, weights_to

pytestmark = pytest.mark.gpu

# An intermediate value next to a rounding boundary may be quantised to the neighbour of the oracle's: at the top of a group's range, where
# steps are widest, a step of amax / 14 <= 0.43 (|a| <= 6), times a down weight |w| <= 0.4 (4.5 sigma of N(0, 1/128)), times the
# router weights of the expert's slots, <= 0.67 with two of three on one expert.
ONE_STEP = 0.43 * 0.4 * 0.67


@pytest.mark.parametrize("T,pair", [((60,), False), ((300, 20), False), ((300, 20), True)])
def test_experts_of_one_and_of_several_tiles(T, pair):
    E, k = 1024, 3
    classes = (synth.PREFILL, synth.DECODE)[:len(T)]
    spec = synth.Spec("once8", synth.Shape(E, k, 256, 128, "fp8"), tuple(zip(classes, T)), "zipf", 1.0, 1.0, -1.0, 53)
    W = synth.make_weights(spec)
    ops = synth.make_ops(spec)
    for o in ops:                                   # every token meets expert 1023 (twice in a short op: more rows than a tile), and two of the others
        t = np.arange(len(o.ids))
        o.ids[:, 0] = E - 1
        o.ids[:, 1] = E - 1 if len(T) == 1 else 1 + 2 * (t % 500)
        o.ids[:, 2] = 2 + 2 * ((17 * t) % 500)
    OW = oracle_weights(spec, W)
    want = [np.asarray(oracle.forward(OW, o.x, o.x_scale, o.ids, o.w)["y"]) for o in ops]
    ctx = make_ctx(spec, max_tokens=sum(T))
    bound = bind_ops(ctx, ops, weights_to(W))
    for s, b in enumerate(bound):
        b.y.fill_(7.0)
        ctx.plan(s, b)
    if pair:
        ctx.plan_pair(0, 1)
    ctx.run(range(len(T)), fuse_combine=True)
    ctx.check()
    for b, y in zip(bound, want):
        assert_close(b.y.float().cpu().numpy(), y, ONE_STEP, RTOL8, REL_L2_8)
