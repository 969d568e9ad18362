"""Captured calls replayed after the slot has been bound to something else: a captured plan brings its op along, a launch captured by
itself serves whatever the slot is planned for by then -- other sizes (the kernels for small ops have room for small tiles only),
another class, another ready word."""
import pytest
import torch

import paper_2607_18002_b200 as moe
from workloads import synth

from gpu_util import bind_ops, make_ctx, upload, weights_to

pytestmark = pytest.mark.gpu


def _setup(dtype, sizes, **kw):
    spec = synth.Spec("capture", synth.Shape(8, 2, 512, 256, dtype), tuple((c, T) for c, T in sizes), "zipf", 1.0, 1.0, -1.0, 51)
    W = weights_to(synth.make_weights(spec))
    ctx = make_ctx(spec, max_tokens=sum(T for _, T in sizes), max_ops=2, **kw)
    bound = bind_ops(ctx, synth.make_ops(spec), W)
    want = []
    for b in bound:
        ctx.plan(0, b)
        ctx.run([0], fuse_combine=True)
        ctx.check()
        want.append(b.y.clone())
    return spec, W, ctx, bound, want


def _capture(fn):
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    g = torch.cuda.CUDAGraph()
    with torch.cuda.stream(side):
        with torch.cuda.graph(g, stream=side):
            fn()
    torch.cuda.current_stream().wait_stream(side)
    return g


def _expect(ctx, b, y, go):
    b.y.fill_(7.0)
    go()
    ctx.check()
    assert torch.equal(b.y, y)


SIZES = ((synth.DECODE, 16), (synth.PREFILL, 500), (synth.DECODE, 60), (synth.PREFILL, 129))


@pytest.mark.parametrize("dtype,n_ctas", [("bf16", 0), ("bf16", 3), ("fp8", 0)], ids=["pairs", "single", "fp8"])
def test_a_captured_launch_serves_the_plan_it_finds(dtype, n_ctas):
    spec, W, ctx, bound, want = _setup(dtype, SIZES, n_ctas=n_ctas)
    ctx.plan(0, bound[0])
    g = _capture(lambda: ctx.run([0], fuse_combine=True))
    for i in (1, 0, 2, 3, 1):
        ctx.plan(0, bound[i])
        _expect(ctx, bound[i], want[i], g.replay)
    # an op with a ready word, its word unset: the launch waits for it instead of taking the captured op's word for it
    d = upload(synth.make_ops(spec)[1], None)
    word = torch.zeros(1, dtype=torch.int32, device="cuda")
    late = make_ctx(spec, max_tokens=500, max_ops=1, n_ctas=n_ctas, wait_limit_us=2000)
    late.plan(0, bound[0])
    g = _capture(lambda: late.run([0], fuse_combine=True))
    b = late.bind(synth.PREFILL, d["x"], d["ids"], d["w"], W.w_gate_up, W.w_down, x_scale=d["x_scale"], s_gate_up=W.s_gate_up,
                  s_down=W.s_down, ready=word)
    late.plan(0, b)
    g.replay()
    torch.cuda.synchronize()
    assert late.status()[0] == moe.MOE_ETIMEOUT
    word.fill_(1)
    _expect(late, b, want[1], g.replay)


@pytest.mark.parametrize("dtype,n_ctas", [("bf16", 0), ("bf16", 3), ("fp8", 0)], ids=["pairs", "single", "fp8"])
def test_captured_steps_that_share_a_slot(dtype, n_ctas):
    """A graph per batch size on one slot, in any order and with direct calls in between; plan and launch in one graph or in two."""
    spec, W, ctx, bound, want = _setup(dtype, SIZES, n_ctas=n_ctas)

    def step(b):
        ctx.plan(0, b)
        ctx.run([0], fuse_combine=True)

    whole = [_capture(lambda b=b: step(b)) for b in bound]
    plans = [_capture(lambda b=b: ctx.plan(0, b)) for b in bound]
    launch = _capture(lambda: ctx.run([0], fuse_combine=True))
    order = (0, 1, 3, 2, 0, 3, 1)
    for i, j in zip(order, order[1:] + order[:1]):
        _expect(ctx, bound[i], want[i], whole[i].replay)
        _expect(ctx, bound[j], want[j], lambda: step(bound[j]))
        _expect(ctx, bound[i], want[i], lambda: (plans[i].replay(), launch.replay()))
        _expect(ctx, bound[j], want[j], lambda: (plans[j].replay(), ctx.run([0], fuse_combine=True)))
        _expect(ctx, bound[j], want[j], lambda: (step(bound[i]), whole[j].replay()))


@pytest.mark.parametrize("dtype,n_ctas", [("bf16", 0), ("bf16", 3), ("fp8", 0)], ids=["pairs", "single", "fp8"])
def test_a_captured_launch_counts_for_the_words_it_finds(dtype, n_ctas):
    """Committed tiles are counted only where an op of the launch has a done or a notify word or a successor: whether one has is read
    from the plan that the launch finds, not from the op that it was captured with."""
    spec, W, ctx, bound, want = _setup(dtype, SIZES, n_ctas=n_ctas)
    ctx.plan(0, bound[0])
    g = _capture(lambda: ctx.run([0], fuse_combine=True))
    words = torch.zeros(2, dtype=torch.int32, device="cuda")
    d = upload(synth.make_ops(spec)[1], None)
    args = (synth.PREFILL, d["x"], d["ids"], d["w"], W.w_gate_up, W.w_down)
    scales = dict(x_scale=d["x_scale"], s_gate_up=W.s_gate_up, s_down=W.s_down)
    for kw in (dict(done=words[:1]), dict(notify=words[1:], notify_after=3), dict(done=words[:1], notify=words[1:], notify_after=1)):
        words.zero_()
        b = ctx.bind(*args, **scales, **kw)
        ctx.plan(0, b)
        _expect(ctx, b, want[1], g.replay)
        assert words.tolist() == [int("done" in kw), int("notify" in kw)]
        words.zero_()
        ctx.plan(0, bound[0])
        _expect(ctx, bound[0], want[0], g.replay)
        assert words.tolist() == [0, 0]


def test_a_captured_pair_and_its_ops_by_themselves():
    spec, W, ctx, bound, want = _setup("bf16", SIZES)

    def paired(p, d):
        ctx.plan(0, bound[p])
        ctx.plan(1, bound[d])
        ctx.plan_pair(0, 1)
        ctx.run([0, 1], fuse_combine=True)

    pairs = [(1, 0), (3, 2)]
    graphs = [_capture(lambda pd=pd: paired(*pd)) for pd in pairs]
    for n in (0, 1, 0, 0, 1, 1):
        for i in pairs[n]:
            bound[i].y.fill_(7.0)
        graphs[n].replay()
        ctx.check()
        assert all(torch.equal(bound[i].y, want[i]) for i in pairs[n])
        paired(*pairs[1 - n])
        ctx.check()
        assert all(torch.equal(bound[i].y, want[i]) for i in pairs[1 - n])


def test_a_plan_too_tall_for_the_launched_kernel_is_reported():
    """A direct plan for a small op, a replayed plan for a large one, a direct launch: the launch was chosen for the small op.  It has no
    room for the tiles it finds and says so instead of running them."""
    spec, W, ctx, bound, want = _setup("bf16", SIZES)
    g = _capture(lambda: ctx.plan(0, bound[1]))
    ctx.plan(0, bound[0])
    g.replay()
    bound[1].y.fill_(7.0)
    ctx.run([0], fuse_combine=True)
    torch.cuda.synchronize()
    assert ctx.status()[0] == moe.MOE_EBOUNDS
    assert torch.all(bound[1].y == 7.0)
    ctx.plan(0, bound[0])
    _expect(ctx, bound[0], want[0], lambda: ctx.run([0], fuse_combine=True))


def test_a_launch_ahead_of_the_replay_of_its_plan_does_nothing():
    spec, W, _, bound, want = _setup("bf16", SIZES)
    ctx = make_ctx(spec, max_tokens=705, max_ops=2)

    def plans():
        ctx.plan(0, bound[1])
        ctx.plan(1, bound[0])
        ctx.plan_pair(0, 1)

    g = _capture(plans)
    for b in bound[:2]:
        b.y.fill_(7.0)
    ctx.run([0], fuse_combine=True)
    ctx.run([0, 1], fuse_combine=True)
    ctx.combine(0)
    ctx.check()
    assert all(torch.all(b.y == 7.0) for b in bound[:2])
    g.replay()
    ctx.run([0, 1], fuse_combine=True)
    ctx.check()
    assert all(torch.equal(b.y, w) for b, w in zip(bound[:2], want))
