"""Launches that run two neighbouring n-blocks of a work tile at a time: experts of one, two and several work tiles, even and odd numbers of
n-blocks, tiles of 1 to 256 rows, lists whose last entries go one by one, paired ops and ops behind one another.  Bit for bit the
plain launch, which runs tile by tile, with every entry logged once; the outputs against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from workloads import synth

from gpu_util import assert_close, bind_ops, make_ctx, oracle_weights, weights_to

pytestmark = pytest.mark.gpu

ROWS = (1, 16, 17, 130, 255, 256, 257, 300, 512, 700, 31, 33, 97, 240)      # prefill rows of the experts


def _ids(T, E, shift):
    """[T, 2] distinct experts; expert (e + shift) % E gets ROWS[e] tokens in the first column, the second column goes round."""
    first = np.concatenate([np.full(n, (e + shift) % E) for e, n in enumerate(ROWS)])[:T]
    return np.stack([first, (first + 1 + np.arange(T) % (E - 1)) % E], 1).astype(np.int32)


@pytest.mark.parametrize("form", ["one", "two", "chain", "pair"])
@pytest.mark.parametrize("H,I", [(1024, 1024), (1280, 1152)])
def test_two_tiles_at_a_time(H, I, form):
    E, k = len(ROWS) + 2, 2
    T = (sum(ROWS), 40)
    spec = synth.Spec("dual", synth.Shape(E, k, H, I, "bf16"), ((synth.PREFILL, T[0]), (synth.DECODE, T[1])), "zipf", 1.0, 1.0, -1.0, 61)
    W = synth.make_weights(spec)
    Wd, OW = weights_to(W), oracle_weights(spec, W)
    ops = synth.make_ops(spec)
    for i, o in enumerate(ops):
        o.ids[:] = _ids(T[0], E, i)[:: T[0] // T[i]][:T[i]]
    ops = ops[:1] if form == "one" else ops
    plain = make_ctx(spec, max_tokens=T[0], max_ops=1)
    ys = []
    for b in bind_ops(plain, ops, Wd):
        plain.plan(0, b)
        plain.run_plain(0)
        plain.check()
        ys.append(b.y)
    for n_ctas in (0, 2, 6):
        ctx = make_ctx(spec, max_tokens=sum(T), max_ops=2, n_ctas=n_ctas, tile_log_entries=1 << 13)
        bound = bind_ops(ctx, ops[:1], Wd)
        if len(ops) > 1:
            bound += bind_ops(ctx, ops[1:], Wd, **({"after_op": 0} if form == "chain" else {}))
        ctx.set_budget(2)
        for s, b in enumerate(bound):
            b.y.fill_(7.0)
            ctx.plan(s, b)
        if form == "pair":
            ctx.plan_pair(0, 1)
        for _ in range(2):
            ctx.run(range(len(ops)), fuse_combine=True)
        ctx.check()
        log = ctx.tile_log()
        for s in range(len(ops)):
            mine = log[log["slot"] == s]
            assert sorted(mine["tile"].tolist()) == list(range(len(mine)))
            gemm = mine[mine["kind"] != 2]
            assert len(gemm) % (I // 128 + H // 256) == 0 and len(gemm) > 0
            up, down = gemm[gemm["kind"] == 0], gemm[gemm["kind"] == 1]
            assert len(up) * (H // 256) == len(down) * (I // 128)
        assert all(torch.equal(b.y, y) for b, y in zip(bound, ys))
    for y, o in zip(ys, ops):
        keep = np.unique(np.r_[0, len(o.ids) - 1, np.arange(0, len(o.ids), 7)])
        got = y.float().cpu().numpy()[keep]
        assert_close(got, np.asarray(oracle.forward_tokens(OW, o.x, None, o.ids, o.w, keep)))
