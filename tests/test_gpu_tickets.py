"""What one claim of the CTA-pair kernel takes from a queue: in large launches of layers with even numbers of n-blocks two neighbouring entries
that run together, in all others one entry.  Read from the tile log: the entries of a ticket have the same unit and claim time."""
import numpy as np
import pytest
import torch

import paper_2607_18002_b200 as moe
from workloads import synth

from gpu_util import bind_ops, make_ctx, weights_to

pytestmark = pytest.mark.gpu


def tickets(log, slot):
    """The op's GEMM entries by ticket: a list of lists of log records."""
    mine = log[(log["slot"] == slot) & (log["kind"] != 2)]
    by = {}
    for r in mine[np.argsort(mine["tile"], kind="stable")]:
        by.setdefault((int(r["cta"]), int(r["t_claim"])), []).append(r)
    return list(by.values())


def run(spec, n_ctas, budget=0, **kw):
    ctx = make_ctx(spec, max_tokens=sum(T for _, T in spec.ops), n_ctas=n_ctas, tile_log_entries=1 << 14, **kw)
    bound = bind_ops(ctx, synth.make_ops(spec), weights_to(synth.make_weights(spec)))
    ctx.set_budget(budget)
    for s, b in enumerate(bound):
        ctx.plan(s, b)
    ctx.run(range(len(bound)), fuse_combine=True)
    ctx.check()
    return ctx, bound


@pytest.mark.parametrize("H,I,twos", [(1024, 1024, True), (1280, 1152, False), (1024, 1152, False), (1280, 1024, False)])
def test_two_entries_of_a_ticket_always_run_together(H, I, twos):
    spec = synth.Spec("tickets", synth.Shape(6, 2, H, I), ((synth.PREFILL, 1500),), "zipf", 1.0, 1.0, -1.0, 83)
    ctx, _ = run(spec, n_ctas=6)
    got = tickets(ctx.tile_log(), 0)
    two = [t for t in got if len(t) > 1]
    assert len(two) * 2 > len(got) if twos else not two
    for a, b in two:                                    # n-blocks 2 p and 2 p + 1 of a work tile lie at places 2 t and 2 t + 1 of the list
        assert a["kind"] == b["kind"] and a["tile"] % 2 == 0 and b["tile"] == a["tile"] + 1


@pytest.mark.parametrize("E,T,twos", [(32, 1000, True), (16, 1000, False), (16, 2000, True)])
def test_two_at_a_time_where_units_have_many_tiles(E, T, twos):
    """Ten rounds of the 16 units by the rows, five where experts get 64 rows or fewer: 5.3, 5.3 and 11 rounds here."""
    spec = synth.Spec("rounds", synth.Shape(E, 2, 1024, 1024), ((synth.PREFILL, T),), "zipf", 1.0, 1.0, -1.0, 89)
    ctx, _ = run(spec, n_ctas=32)
    assert any(len(t) > 1 for t in tickets(ctx.tile_log(), 0)) == twos


@pytest.mark.parametrize("decode,masked", [(40, False), (300, False), (48, True)])
def test_decode_entries_go_one_by_one_next_to_prefill(decode, masked):
    """In a launch that hands prefill entries out in twos, the decode op's tickets are single entries.  Its tiles (rows below and above the 128 up to
    which two k-blocks share a stage, gathered or consecutive) and those at the end of the prefill list give bit for bit what each op gives
    by itself in the plain launch, or the masked op in a launch of its own."""
    E, H, I = 6, 1024, 768
    spec = synth.Spec("latency", synth.Shape(E, 2, H, I), ((synth.PREFILL, 1800), (synth.DECODE, decode)), "zipf", 1.0, 1.0, -1.0, 97)
    W = weights_to(synth.make_weights(spec))
    ops = synth.make_ops(spec)
    ctx = make_ctx(spec, max_tokens=1800, n_ctas=6, tile_log_entries=1 << 14)
    bound = bind_ops(ctx, ops, W)
    alone = make_ctx(spec, max_tokens=1800, max_ops=1)
    if masked:
        x = torch.randn(E, decode, H, generator=torch.Generator().manual_seed(5)).to(torch.bfloat16).cuda()
        counts = torch.tensor([48, 0, 1, 17, 33, 40], dtype=torch.int32, device="cuda")
        bound[1] = moe.bind_masked_op(moe.MOE_CLASS_DECODE, x, counts, W.w_gate_up, W.w_down)
        valid = torch.arange(decode, device="cuda")[None, :] < counts[:, None]
    else:
        valid = slice(None)
    want = []
    for s, b in enumerate(bound):
        b.y.fill_(7.0)
        alone.plan(0, b)
        alone.run([0]) if masked and s == 1 else alone.run_plain(0)
        alone.check()
        want.append(b.y.clone())
    ctx.set_budget(2)
    for s, b in enumerate(bound):
        b.y.fill_(7.0)
        ctx.plan(s, b)
    for _ in range(2):
        ctx.run([0, 1], fuse_combine=True)
    ctx.check()
    log = ctx.tile_log()
    assert any(len(t) == 2 for t in tickets(log, 0)) and all(len(t) == 1 for t in tickets(log, 1))
    assert torch.equal(bound[0].y, want[0]) and torch.equal(bound[1].y[valid], want[1][valid])


def test_a_unit_next_to_another_class_claims_late():
    """In a launch with both classes a unit asks for its next ticket half-way through the loads of two prefill tiles, so that it holds a ticket
    for one and a half times what one takes.  (Asked for at their start it is held for two.)"""
    spec = synth.Spec("late", synth.Shape(4, 2, 3072, 1536), ((synth.PREFILL, 1500), (synth.DECODE, 8)), "uniform", None, 1.0, -1.0, 101)
    ctx, _ = run(spec, n_ctas=6, budget=2)
    got = [t for t in tickets(ctx.tile_log(), 0) if len(t) == 2 and t[0]["kind"] == 0]       # 48 k-blocks each
    held, period = [], []
    for u in {int(t[0]["cta"]) for t in got} - {0}:                    # the unit inside the budget starts with decode tiles
        mine = sorted((t for t in got if t[0]["cta"] == u), key=lambda t: t[0]["t_claim"])[2:]
        end = [max(int(r["t_commit"]) for r in t) for t in mine]
        held += [e - int(t[0]["t_claim"]) for e, t in zip(end, mine)]
        period += list(np.diff(end))
    assert len(period) > 10 and np.median(held) < 1.75 * np.median(period), (np.median(held), np.median(period))


def test_masked_entries_in_twos():
    """A masked op next to a large gathered op of its own class: its gate/up tiles (consecutive rows of x) and down tiles run in twos as well, at 1 to
    200 rows; bit for bit the op in a launch of its own."""
    E, H, I, slab = 6, 1024, 768, 200
    spec = synth.Spec("masked2", synth.Shape(E, 2, H, I), ((synth.DECODE, 1800), (synth.DECODE, 600)), "zipf", 1.0, 1.0, -1.0, 103)
    W = weights_to(synth.make_weights(spec))
    ctx = make_ctx(spec, max_tokens=1800, n_ctas=6, tile_log_entries=1 << 14)
    x = torch.randn(E, slab, H, generator=torch.Generator().manual_seed(7)).to(torch.bfloat16).cuda()
    counts = torch.tensor([200, 1, 0, 129, 128, 33], dtype=torch.int32, device="cuda")
    op = moe.bind_masked_op(moe.MOE_CLASS_DECODE, x, counts, W.w_gate_up, W.w_down)
    alone = make_ctx(spec, max_tokens=600, max_ops=1)
    alone.plan(0, op)
    alone.run([0])
    alone.check()
    want = op.y.clone()
    op.y.fill_(7.0)
    ctx.plan(0, bind_ops(ctx, synth.make_ops(spec)[:1], W)[0])
    ctx.plan(1, op)
    ctx.run([0, 1], fuse_combine=True)
    ctx.check()
    two = [t for t in tickets(ctx.tile_log(), 1) if len(t) == 2]
    assert {int(t[0]["kind"]) for t in two} == {1, 3}
    valid = torch.arange(slab, device="cuda")[None, :] < counts[:, None]
    assert torch.equal(op.y[valid], want[valid]) and torch.all(op.y[~valid] == 7.0)


def test_a_captured_step_in_twos_and_an_entry_out_of_range():
    """A layer step of both classes that runs two tiles at a time, captured and replayed on other routing in the same buffers: the same as when called.
    A permutation entry out of range, met by the warp that lists the rows of the next tiles, ends the launch with MOE_EBOUNDS, and the step behind
    it is right again."""
    spec = synth.Spec("cap2", synth.Shape(6, 2, 1024, 768), ((synth.PREFILL, 1800), (synth.DECODE, 40)), "zipf", 1.0, 1.0, -1.0, 107)
    W = weights_to(synth.make_weights(spec))
    ctx = make_ctx(spec, max_tokens=1800, n_ctas=6, tile_log_entries=1 << 14, wait_limit_us=20000)
    bound = bind_ops(ctx, synth.make_ops(spec), W)

    def step():
        ctx.set_budget(2)
        for s, b in enumerate(bound):
            ctx.plan(s, b)
        ctx.run([0, 1], fuse_combine=True)

    step()
    ctx.check()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        step()
    for shift in (0, 1):
        for b in bound:
            b.topk_ids.copy_((b.topk_ids + shift) % 6)
        step()
        ctx.check()
        want = [b.y.clone() for b in bound]
        for b in bound:
            b.y.fill_(7.0)
        graph.replay()
        ctx.check()
        assert any(len(t) == 2 for t in tickets(ctx.tile_log(), 0))
        assert all(torch.equal(b.y, w) for b, w in zip(bound, want))
    for at in (0, 700, 3599):
        bound[0].sorted_to_flat[at] = 1 << 28
        ctx.run([0, 1], fuse_combine=True)
        torch.cuda.synchronize()
        assert ctx.status()[0] == moe.MOE_EBOUNDS
        step()
        ctx.check()
        assert all(torch.equal(b.y, w) for b, w in zip(bound, want))


@pytest.mark.parametrize("n_ctas,T,H,I", [(6, 1800, 1024, 1024), (6, 1800, 1024, 1152), (0, 16384, 4096, 512)])
def test_a_unit_holds_at_most_five_tickets(n_ctas, T, H, I):
    """Four in the descriptor ring and the one that waits for a place, also where the epilogue is behind (combine tiles of many long rows, all units
    at once) and in launches that run two tiles at a time."""
    spec = synth.Spec("held", synth.Shape(6, 2, H, I), ((synth.PREFILL, T), (synth.DECODE, 300)), "zipf", 1.0, 1.0, -1.0, 109)
    ctx, _ = run(spec, n_ctas=n_ctas, budget=2)
    log = ctx.tile_log()
    for u in np.unique(log["cta"]):
        mine = log[log["cta"] == u]
        claim = np.unique(mine["t_claim"])
        end = np.array([mine["t_commit"][mine["t_claim"] == t].max() for t in claim])
        held = [int((end[:i] > t).sum()) + 1 for i, t in enumerate(claim)]
        assert len(claim) > 8 and max(held) <= 5, max(held)
