"""The plan at the sizes where its split over blocks and warps changes: around the largest op that one launch plans, rows
per block of one and of several thousand, one to 1024 experts, routings that leave most experts empty.  Integer outputs:
bit-exact against the oracle."""
import numpy as np
import pytest
import torch

import oracle
import paper_2607_18002_b200 as moe
from workloads import synth

from gpu_util import (ATOL, ATOL8, REL_L2, REL_L2_8, RTOL, RTOL8, assert_close, bind_ops, check_plan, check_tiles, make_ctx,
                      n_combine_tiles, oracle_weights, weights_to)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,E,k", [(1, 1024, 1), (31, 33, 1), (1023, 256, 8), (1024, 256, 8), (1025, 256, 8), (8193, 8, 1),
                                   (2049, 1000, 4), (131072, 16, 1), (131073, 5, 1), (40001, 40, 5)])
def test_plan_and_queue_list(T, E, k):
    spec = synth.Spec("sizes", synth.Shape(E, k, 256, 128), ((synth.PREFILL, T),), "uniform", None, 1.0, -1.0, 5)
    Wd = weights_to(synth.make_weights(spec))
    ctx = make_ctx(spec)
    rng = np.random.default_rng([T, E, k])
    # a skewed draw with repeats (ids of a token need not differ for the plan), so that many experts stay empty
    ids = np.minimum(rng.zipf(1.3, size=(T, k)) - 1, rng.integers(0, E, size=(T, k))).astype(np.int32)
    op = synth.Op(synth.PREFILL, torch.zeros(T, 256, dtype=torch.bfloat16), ids, np.full(ids.shape, 1.0 / k, np.float32))
    b = bind_ops(ctx, [op], Wd)[0]
    ctx.plan(0, b)
    ctx.check()
    counts = check_plan(b, op, E)
    check_tiles(ctx, 0, counts)
    rows = 256 if ctx.ctas_per_tile == 2 else moe.MOE_TILE_M        # bf16 work tiles on the default grid
    assert ctx.footprint(0)[1] == int((-(-counts // rows)).sum()) * 2 + n_combine_tiles(T)


@pytest.mark.parametrize("dtype,T", [("bf16", 32), ("fp8", 64)])
def test_more_low_tiles_than_mtiles(dtype, T):
    """An op of few tokens is cut into lower tiles.  When its tokens name one expert with every slot it has more of them than m-tiles
    plus experts: list and dependency counters of a context of just that size hold them, the neighbouring slot stays intact."""
    E = k = 8
    spec = synth.Spec("low", synth.Shape(E, k, 256, 128, dtype), ((synth.DECODE, T), (synth.PREFILL, T)), "uniform", None, 1.0, -1.0, 7)
    W = synth.make_weights(spec)
    ids = np.zeros((T, k), np.int32)
    ids[np.arange(7), k - 1] = np.arange(1, 8)                      # the other experts get a row each
    ctx = make_ctx(spec)
    ops = []
    for i, (cls, _) in enumerate(spec.ops):
        x, xs = synth.make_x(spec, T, 0, i)
        ops.append(synth.Op(cls, x, ids, np.full(ids.shape, 1.0 / k, np.float32), xs))
    bound = bind_ops(ctx, ops, weights_to(W))
    for s, b in enumerate(bound):
        ctx.plan(s, b)
    ctx.run([0, 1], fuse_combine=True)
    ctx.check()
    rows = 32 if dtype == "bf16" and ctx.ctas_per_tile == 2 else 64 if dtype == "fp8" else 128
    tol = dict(atol=ATOL, rtol=RTOL, rel_l2=REL_L2) if dtype == "bf16" else dict(atol=ATOL8, rtol=RTOL8, rel_l2=REL_L2_8)
    for s, (b, op) in enumerate(zip(bound, ops)):
        counts = check_plan(b, op, E)
        assert ctx.footprint(s)[1] == int((-(-counts // rows)).sum()) * 2 + n_combine_tiles(T)
        ref = oracle.forward(oracle_weights(spec, W), op.x, op.x_scale, op.ids, op.w,
                             round_A=oracle.ROUND_NONE if dtype == "bf16" else oracle.ROUND_E4M3_1X128)["y"]
        assert_close(b.y.float().cpu().numpy(), ref, **tol)


@pytest.mark.parametrize("E", [1, 8, 33, 256, 1024])
def test_an_op_without_tokens(E):
    """Its blocks own no rows: zero counts and offsets, no tiles, nothing written to the permutation, whatever the slot held before."""
    spec = synth.Spec("empty", synth.Shape(E, 1, 256, 128), ((synth.DECODE, 40), (synth.DECODE, 0)), "uniform", None, 1.0, -1.0, 9)
    ctx = make_ctx(spec, max_ops=1)
    full, empty = bind_ops(ctx, synth.make_ops(spec), weights_to(synth.make_weights(spec)))
    for _ in range(2):
        ctx.plan(0, full)
        for t in (empty.counts, empty.offsets, empty.sorted_to_flat, empty.flat_to_sorted):
            t.fill_(77)
        ctx.plan(0, empty)
        ctx.run([0], fuse_combine=True)
        ctx.check()
        assert ctx.footprint(0) == (0, 0)
        assert not empty.counts.any() and not empty.offsets.any()
        assert empty.sorted_to_flat.tolist() == [77] and empty.flat_to_sorted.tolist() == [77]
