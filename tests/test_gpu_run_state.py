"""Launches hand the run state on from one to the next: each works on one half of it and clears the other.  Whatever a launch did
-- all slots, one slot, a wait that ran out, a plain launch -- the next one starts from zero, also without a host synchronisation."""
import pytest
import torch

import paper_2607_18002_b200 as moe
from workloads import synth

from gpu_util import bind_ops, make_ctx, weights_to

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,n_ctas", [("bf16", 0), ("bf16", 3), ("fp8", 0)], ids=["pairs", "single", "fp8"])
def test_every_kind_of_launch_leaves_a_clean_state(dtype, n_ctas):
    spec = synth.Spec("state", synth.Shape(8, 2, 512, 256, dtype), ((synth.PREFILL, 300), (synth.DECODE, 37)), "zipf", 1.0, 1.0, -1.0, 71)
    W = weights_to(synth.make_weights(spec))
    ctx = make_ctx(spec, n_ctas=n_ctas, wait_limit_us=20000, tile_log_entries=1 << 12)
    bound = bind_ops(ctx, synth.make_ops(spec), W)
    for s, b in enumerate(bound):
        ctx.plan(s, b)
    n = [ctx.footprint(s)[1] for s in range(2)]
    ctx.run([0, 1], fuse_combine=True)
    ctx.check()
    want = [b.y.clone() for b in bound]
    assert len(ctx.tile_log()) == sum(n)
    word = torch.zeros(1, dtype=torch.int32, device="cuda")
    for step in ("both", "one", "late", "both", "both", "one"):
        for b in bound:
            b.y.zero_()
        if step == "late":                       # a ready word that nothing sets: the wait runs out, tiles stay unserved
            bound[1].c.ready = word.data_ptr()
            ctx.plan(1, bound[1])
            ctx.run([0, 1], fuse_combine=True)
            torch.cuda.synchronize()
            assert ctx.status()[0] == moe.MOE_ETIMEOUT
            bound[1].c.ready = None
            ctx.plan(1, bound[1])
            continue
        slots = [0, 1] if step == "both" else [0]
        for _ in range(3):                       # back to back, nothing waits in between
            ctx.run(slots, fuse_combine=True)
        ctx.check()
        assert len(ctx.tile_log()) == sum(n[s] for s in slots)
        for s in slots:
            assert torch.equal(bound[s].y, want[s]), (step, s)
    if ctx.ctas_per_tile == 2 and dtype == "bf16":
        ctx.run_plain(0)
        ctx.run([0, 1], fuse_combine=True)
        ctx.check()
        assert all(torch.equal(b.y, w) for b, w in zip(bound, want))


@pytest.mark.parametrize("dtype,T", [("fp8", 20), ("fp8", 48), ("bf16", 20), ("bf16", 100), ("bf16", 600)])
def test_launches_end_when_they_are_aborted(dtype, T):
    """An index out of range met in the middle of a launch and a ready word that nothing sets both stop it: every role leaves, also the
    epilogue warps that wait for one another, the error is reported, and the launches behind it are right again."""
    spec = synth.Spec("abort", synth.Shape(16, 4, 1024, 512, dtype), ((synth.PREFILL, T), (synth.DECODE, T)), "uniform", None, 1.0, -1.0, 73)
    W = weights_to(synth.make_weights(spec))
    ctx = make_ctx(spec, wait_limit_us=2000)
    bound = bind_ops(ctx, synth.make_ops(spec), W)

    def launch():
        ctx.run([0, 1], fuse_combine=True)
        torch.cuda.synchronize()
        return ctx.status()[0]

    for s, b in enumerate(bound):
        ctx.plan(s, b)
    assert launch() == moe.MOE_OK
    want = [b.y.clone() for b in bound]
    word = torch.zeros(1, dtype=torch.int32, device="cuda")
    for _ in range(3):
        bound[0].sorted_to_flat[3] = 1 << 28
        assert launch() == moe.MOE_EBOUNDS
        ctx.plan(0, bound[0])
        bound[1].c.ready = word.data_ptr()
        ctx.plan(1, bound[1])
        assert launch() == moe.MOE_ETIMEOUT
        bound[1].c.ready = None
        ctx.plan(1, bound[1])
        for b in bound:
            b.y.zero_()
        assert launch() == moe.MOE_OK
        assert all(torch.equal(b.y, w) for b, w in zip(bound, want))


@pytest.mark.parametrize("dtype,n_ctas", [("bf16", 0), ("bf16", 3), ("fp8", 0)], ids=["pairs", "single", "fp8"])
@pytest.mark.parametrize("launches", [1, 2], ids=["one_half", "other_half"])
def test_a_launch_behind_a_rejected_plan_leaves_a_clean_state(dtype, n_ctas, launches):
    """A plan with an expert id out of range sets the abort word before the launch behind it begins.  That launch does nothing, but it
    too has to clear the half of the run state that the next one works on; both halves have been used by then."""
    spec = synth.Spec("rejected", synth.Shape(8, 2, 512, 256, dtype), ((synth.DECODE, 37),), "uniform", None, 1.0, -1.0, 77)
    ctx = make_ctx(spec, n_ctas=n_ctas, tile_log_entries=1 << 12)
    b = bind_ops(ctx, synth.make_ops(spec), weights_to(synth.make_weights(spec)))[0]
    ctx.plan(0, b)
    for _ in range(1 + launches):                     # both halves, and either parity for what follows
        ctx.run([0], fuse_combine=True)
    ctx.check()
    want, n, good = b.y.clone(), len(ctx.tile_log()), b.topk_ids.clone()
    for _ in range(2):
        b.topk_ids[5, 1] = 99
        ctx.plan(0, b)
        ctx.run([0], fuse_combine=True)
        torch.cuda.synchronize()
        assert ctx.status()[0] == moe.MOE_EBADID
        assert len(ctx.tile_log()) == 0
        b.topk_ids.copy_(good)
        ctx.plan(0, b)
        for _ in range(2):
            b.y.zero_()
            ctx.run([0], fuse_combine=True)
            ctx.check()
            assert len(ctx.tile_log()) == n and torch.equal(b.y, want)


def test_a_plain_run_without_tiles_has_an_empty_log():
    spec = synth.Spec("nolog", synth.Shape(8, 2, 512, 256), ((synth.DECODE, 37), (synth.DECODE, 0)), "uniform", None, 1.0, -1.0, 79)
    ctx = make_ctx(spec, tile_log_entries=1 << 12)
    bound = bind_ops(ctx, synth.make_ops(spec), weights_to(synth.make_weights(spec)))
    for s, b in enumerate(bound):
        ctx.plan(s, b)
    for _ in range(3):
        ctx.run([0], fuse_combine=True)
        ctx.check()
        n = len(ctx.tile_log())
        assert n == ctx.footprint(0)[1]
        ctx.run_plain(1)
        ctx.check()
        assert len(ctx.tile_log()) == 0
        ctx.run_plain(0)
        ctx.check()
        assert 0 < len(ctx.tile_log()) < n            # without the combine
