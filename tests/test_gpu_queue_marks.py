"""Which entries of a queue list carry the mark that their weights are read once: those of experts with one work tile in the op's list
and, for a pair, none in the other op's.  The lists are read back from the workspace; the tiles are counted here from the ids."""
import numpy as np
import pytest
import torch

import paper_2607_18002_b200 as moe
from workloads import synth

from gpu_util import bind_ops, make_ctx, weights_to

pytestmark = pytest.mark.gpu

E, K, H, I, TP, TD = 1024, 4, 256, 128, 700, 40
NT1, NT2 = I // 128, H // 256
# the op descriptors in the workspace, and the pointers to its list and plan state in one
OPS_AT, OP_BYTES, LIST_AT, PLAN_AT = 1024, 1920, 1536 + 184, 1536 + 200


def _entries(ctx, slot, paired, max_ops):
    """(work_rows, GEMM entries [n, 4]) of the slot's list."""
    base = (ctx.workspace.data_ptr() + 1023) // 1024 * 1024
    raw = ctx.workspace[base - ctx.workspace.data_ptr():].cpu().numpy()
    op = raw[OPS_AT + OP_BYTES * (slot + (max_ops if paired else 0)):][:OP_BYTES]
    at = lambda o: int(op[o:o + 8].view(np.uint64)[0]) - base
    state = raw[at(PLAN_AT):][:32].view(np.int32)
    assert state[3] == 1                                    # planned
    return int(state[5]), raw[at(LIST_AT):][:16 * state[1]].view(np.int32).reshape(-1, 4)


def _check(entries, tiles, once):
    """tiles[e]: work tiles of expert e in this list; once[e]: its weights are read by one of them only."""
    expert, mark = entries[:, 3] & 0xffff, entries[:, 3] >> 16
    assert np.array_equal(np.bincount(expert, minlength=E), tiles * (NT1 + NT2))
    assert np.array_equal(mark, once[expert].astype(np.int32))


def _ops():
    rest = lambda t, first: first + t % 256
    t, d = np.arange(TP), np.arange(TD)
    p_ids = np.stack([np.full(TP, E - 1), np.select([t < 250, t < 350, t < 380], [5, 7, 11], rest(t, 700)), rest(t, 100), rest(t, 400)], 1)
    d_ids = np.stack([np.full(TD, E - 1), np.select([d < 20, d < 30, d < 35], [5, 9, 11], rest(d, 700)), rest(d, 100), rest(d, 400)], 1)
    return p_ids.astype(np.int32), d_ids.astype(np.int32)


@pytest.mark.parametrize("n_ctas", [0, 3], ids=["pairs", "single"])
def test_marked_entries(n_ctas):
    spec = synth.Spec("marks", synth.Shape(E, K, H, I, "bf16"), ((synth.PREFILL, TP), (synth.DECODE, TD)), "zipf", 1.0, 1.0, -1.0, 91)
    ops = synth.make_ops(spec)
    for o, ids in zip(ops, _ops()):
        o.ids[:] = ids
    cp, cd = (np.bincount(o.ids.reshape(-1), minlength=E) for o in ops)
    ctx = make_ctx(spec, max_tokens=TP + TD, n_ctas=n_ctas)
    marks = ctx.ctas_per_tile == 2
    for s, b in enumerate(bind_ops(ctx, ops, weights_to(synth.make_weights(spec)))):
        ctx.plan(s, b)
    ctx.check()
    for s, cnt in enumerate((cp, cd)):
        rows, entries = _entries(ctx, s, False, 2)
        tiles = -(-cnt // rows)
        _check(entries, tiles, (tiles == 1) & marks)
    ctx.plan_pair(0, 1)
    ctx.check()
    # the decode list takes the prefill rows behind the last full tile where they fit beside the decode rows
    room = np.where(cd > 0, -cd % 256, 0)
    take = np.where(cp % 256 <= room, cp % 256, 0)
    wp, wd = -(-(cp - take) // 256), -(-(cd + take) // 256)
    assert [(wp[e], wd[e]) for e in (E - 1, 5, 7, 9, 11)] == [(2, 1), (1, 1), (1, 0), (0, 1), (0, 1)]
    _check(_entries(ctx, 0, True, 2)[1], wp, (wp == 1) & (wd == 0) & marks)
    _check(_entries(ctx, 1, True, 2)[1], wd, (wd == 1) & (wp == 0) & marks)


def test_marked_entries_of_slabs():
    slab = 300
    counts = np.zeros(E, np.int32)
    counts[[0, 3, 8, E - 1]] = 300, 1, 256, 257
    ctx = moe.Context(E, K, H, I, E * slab // K, 1)
    x = torch.zeros(E, slab, H, dtype=torch.bfloat16, device="cuda")
    w1, w2 = (torch.zeros(E, *s, dtype=torch.bfloat16, device="cuda") for s in ((2 * I, H), (H, I)))
    ctx.plan(0, moe.bind_masked_op(moe.MOE_CLASS_DECODE, x, torch.from_numpy(counts).cuda(), w1, w2))
    ctx.check()
    rows, entries = _entries(ctx, 0, False, 1)
    tiles = -(-counts // rows)
    assert rows == 256 and list(tiles[[0, 3, 8, E - 1]]) == [2, 1, 1, 2]
    _check(entries, tiles, tiles == 1)
