"""What one claim of the CTA-pair kernel takes from a queue: in large launches of layers with even numbers of n-blocks two neighbouring entries
that run together, in all others one entry.  Read from the tile log: the entries of a ticket have the same unit and claim time."""
import numpy as np
import pytest
import torch

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
