"""What one MoE layer costs a program that uses this library, from router logits to outputs.

A case is one layer on one GPU: a decode batch, a prefill batch, or both in one launch, as a serving loop issues
them -- moe_route per op, moe_set_budget where two classes share the launch, moe_plan per op, moe_plan_pair where
the two ops travel together, and one moe_run with the fused combine.  The masked layout starts at its dispatched
slabs (it has neither router nor combine).  Shapes are those of workloads/synth.py, the tests and bench.py.

Inputs are drawn on the GPU from the seed: activations N(0,1), weights N(0, 0.02), logits whose top-k follows a
Zipf(s) popularity over a random expert order (s = 0: uniform), for e4m3 quantised per 128x128 block and 1x128 group.
"""
import math

import torch

import paper_2607_18002_b200 as moe

E4M3_MAX = 448.0


def _case(name, dtype, experts, top_k, hidden, inter, prefill, decode, zipf=0.0, active=0, budget=0, pair=False, masked=False):
    """active: experts the tokens may choose from (0: all); budget: decode SM budget of a co-scheduled launch."""
    return dict(name=name, dtype=dtype, experts=experts, top_k=top_k, hidden=hidden, inter=inter, prefill=prefill, decode=decode,
                zipf=zipf, active=active, budget=budget, pair=pair, masked=masked)


def listed():
    big, big8 = (256, 8, 3072, 1536), (256, 8, 6144, 2048)
    return [
        # a toy layer: nothing but launches and latencies
        _case("tiny_layer", "bf16", 8, 2, 256, 512, 48, 16, budget=16),
        # one user's decode step: 8 experts' weights are read for one token
        _case("decode_1", "bf16", *big, 0, 1),
        # a decode batch on one GPU of an expert-parallel group: its tokens meet only 8 of the experts
        _case("decode_128_on_8", "bf16", *big, 0, 128, active=8),
        # a decode batch over all experts: the whole layer's weights are streamed
        _case("decode_128", "bf16", *big, 0, 128),
        # a decode batch that a dispatch step left in per-expert slabs
        _case("decode_masked_96_on_32", "bf16", *big, 0, 96, active=32, masked=True),
        # the last, odd-sized chunk of a prompt
        _case("prefill_777", "bf16", *big, 777, 0, zipf=1.0),
        # a full prefill chunk with a skewed expert popularity
        _case("prefill_8192", "bf16", *big, 8192, 0, zipf=1.2),
        # a 64-expert layer shared by both classes, each with its own tiles
        _case("mixed_4096_64", "bf16", 64, 8, 3072, 1536, 4096, 64, zipf=1.1, budget=32),
        # the largest co-scheduled layer, decode rows carried along with prefill rows
        _case("mixed_16384_256_paired", "bf16", *big, 16384, 256, zipf=1.1, budget=64, pair=True),
        # e4m3: a decode batch, an odd-sized prefill chunk, and both together
        _case("fp8_decode_48", "fp8", *big8, 0, 48),
        _case("fp8_prefill_2000", "fp8", *big8, 2000, 0, zipf=1.0),
        _case("fp8_mixed_4096_512_paired", "fp8", *big8, 4096, 512, zipf=1.0, budget=96, pair=True),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    dtype = rng.choice(["bf16", "bf16", "fp8"])
    kind = rng.choice(["decode", "decode", "prefill", "mixed"])
    shapes = [(8, 2, 256, 512), (32, 4, 1024, 512)] + [(e, 8, 3072, 1536) for e in (64, 64, 128, 256, 256, 256)]
    if dtype == "fp8":
        shapes = [(16, 4, 768, 384)] + [(e, 8, 6144, 2048) for e in (32, 64, 128, 256, 256)]
    experts, top_k, hidden, inter = rng.choice(shapes)
    c = dict(dtype=dtype, experts=experts, top_k=top_k, hidden=hidden, inter=inter, prefill=0, decode=0, zipf=0.0, active=0,
             budget=0, pair=False, masked=False)
    most = 4096 if dtype == "fp8" else 12288
    if kind != "decode":
        c["prefill"] = _log_int(rng, 64, most)
        c["zipf"] = round(rng.uniform(0.6, 1.6), 2)
    if kind != "prefill":
        c["decode"] = _log_int(rng, 1, 512 if kind == "decode" else 256)
    if kind == "mixed":
        c["budget"] = rng.choice([16, 32, 64, 96])
        c["pair"] = rng.random() < 0.5
    if kind == "decode":
        c["zipf"] = round(rng.uniform(0.0, 1.2), 2)
        if rng.random() < 0.4:
            c["active"] = _log_int(rng, top_k, experts)
        c["masked"] = rng.random() < 0.25
    return c


# ------------------------------------------------------------------ inputs

def _quant(v, br, bc):
    """fp32 [..., r, c] -> (e4m3 codes as uint8, fp32 scales per br x bc block)."""
    r, c = v.shape[-2:]
    blk = v.view(*v.shape[:-2], r // br, br, c // bc, bc)
    scale = blk.abs().amax(dim=(-3, -1), keepdim=True).clamp_(min=1e-20) / E4M3_MAX
    q = (blk / scale).clamp_(-E4M3_MAX, E4M3_MAX).to(torch.float8_e4m3fn).view(torch.uint8).view(v.shape)
    return q, scale.squeeze(-1).squeeze(-2).contiguous()


def _weights(c, g, dev):
    E, H, I = c["experts"], c["hidden"], c["inter"]
    if c["dtype"] == "bf16":
        return [torch.empty(E, r, k, dtype=torch.bfloat16, device=dev).normal_(0.0, 0.02, generator=g) for r, k in ((2 * I, H), (H, I))] + [None, None]
    ws, ss = [], []
    for r, k in ((2 * I, H), (H, I)):
        w = torch.empty(E, r, k, dtype=torch.uint8, device=dev)
        s = torch.empty(E, r // 128, k // 128, dtype=torch.float32, device=dev)
        for e in range(0, E, 8):
            n = min(8, E - e)
            w[e:e + n], s[e:e + n] = _quant(torch.empty(n, r, k, device=dev).normal_(0.0, 0.02, generator=g), 128, 128)
        ws.append(w)
        ss.append(s)
    return ws + ss


def _activations(c, rows, g, dev):
    v = torch.empty(rows, c["hidden"], device=dev).normal_(0.0, 1.0, generator=g)
    return (v.to(torch.bfloat16), None) if c["dtype"] == "bf16" else _quant(v, 1, 128)


def _log_popularity(c, g, dev):
    """log popularity of every expert: Zipf(s) over a random order, -60 for experts outside the pool."""
    E, n = c["experts"], c["active"] or c["experts"]
    rank = torch.randperm(E, generator=g, device=dev)
    lp = -c["zipf"] * torch.log((rank + 1).float())
    return torch.where(rank < n, lp, torch.full_like(lp, -60.0))


def _logits(log_pi, T, g, dev):
    """Gumbel noise on the log popularity: the k largest are k experts drawn without replacement."""
    u = torch.rand(T, log_pi.numel(), generator=g, device=dev).clamp_(1e-7, 1.0 - 1e-7)
    return (log_pi - torch.log(-torch.log(u))).contiguous()


def prepare(case, seed):
    c, dev = case, torch.device("cuda:0")
    g = torch.Generator(device=dev)
    g.manual_seed(seed)
    E, k = c["experts"], c["top_k"]
    w1, w2, s1, s2 = _weights(c, g, dev)
    log_pi = _log_popularity(c, g, dev)
    kw = dict(n_experts=E, top_k=k, hidden=c["hidden"], inter=c["inter"], device=dev,
              dtype=moe.MOE_DTYPE_BF16 if c["dtype"] == "bf16" else moe.MOE_DTYPE_FP8_E4M3)
    if c["masked"]:
        slab = -(-c["decode"] // 8) * 8                      # any expert may be chosen by every token
        top = torch.topk(_logits(log_pi, c["decode"], g, dev), k, dim=1).indices
        counts = torch.bincount(top.reshape(-1), minlength=E).to(torch.int32)
        x, xs = _activations(c, E * slab, g, dev)
        ctx = moe.Context(max_tokens_per_op=-(-E * slab // k), max_ops=1, **kw)
        op = moe.bind_masked_op(moe.MOE_CLASS_DECODE, x.view(E, slab, -1), counts, w1, w2,
                                x_scale=None if xs is None else xs.view(E, slab, -1), s_gate_up=s1, s_down=s2)
        return dict(case=c, ctx=ctx, ops=[op], logits=[None])
    todo = [(cls, T) for cls, T in ((moe.MOE_CLASS_PREFILL, c["prefill"]), (moe.MOE_CLASS_DECODE, c["decode"])) if T > 0]
    tokens = [T for _, T in todo]
    ctx = moe.Context(max_tokens_per_op=sum(tokens) if c["pair"] else max(tokens), max_ops=len(todo), **kw)
    ops, logits = [], []
    for cls, T in todo:
        x, xs = _activations(c, T, g, dev)
        ids = torch.zeros(T, k, dtype=torch.int32, device=dev)
        wt = torch.zeros(T, k, dtype=torch.float32, device=dev)
        logits.append(_logits(log_pi, T, g, dev))
        ops.append(ctx.bind(cls, x, ids, wt, w1, w2, x_scale=xs, s_gate_up=s1, s_down=s2))
    return dict(case=c, ctx=ctx, ops=ops, logits=logits)


# ------------------------------------------------------------------ one pass

def run(state):
    c, ctx, ops = state["case"], state["ctx"], state["ops"]
    stream = torch.cuda.current_stream().cuda_stream
    if c["budget"]:
        ctx.set_budget(c["budget"])
    for slot, (op, z) in enumerate(zip(ops, state["logits"])):
        if z is not None:
            moe.moe_route(z.data_ptr(), z.shape[0], c["experts"], c["top_k"], op.topk_ids.data_ptr(), op.topk_w.data_ptr(), stream)
        ctx.plan(slot, op)
    if c["pair"]:
        ctx.plan_pair(0, 1)
    ctx.run(range(len(ops)), fuse_combine=True)
    if c["masked"]:
        return [dict(y=op.y, offsets=op.offsets) for op in ops]
    return [dict(y=op.y, ids=op.topk_ids, w=op.topk_w, counts=op.counts, offsets=op.offsets, sorted_to_flat=op.sorted_to_flat,
                 flat_to_sorted=op.flat_to_sorted) for op in ops]


# ------------------------------------------------------------------ what a pass cannot do without

def _expected_active(c):
    """Expected number of experts that the launch's tokens meet (k draws without replacement per token)."""
    n, k = c["active"] or c["experts"], c["top_k"]
    pi = [(r + 1) ** -c["zipf"] for r in range(n)]
    if n == k:
        return float(n)
    lo, hi = 0.0, 1e9                                        # rate at which a token has chosen k experts on average
    for _ in range(100):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if sum(1.0 - math.exp(-mid * p) for p in pi) < k else (lo, mid)
    T = c["prefill"] + c["decode"]
    return sum(1.0 - math.exp(-T * lo * p) for p in pi)


def work(case):
    c = case
    E, k, H, I, T = c["experts"], c["top_k"], c["hidden"], c["inter"], case["prefill"] + case["decode"]
    el = 2 if c["dtype"] == "bf16" else 1
    rows_in = T * k if c["masked"] else T                    # the masked layout holds a row per routed (token, expert)
    per_expert = 3 * H * I * el + (0 if el == 2 else 3 * (H // 128) * (I // 128) * 4)
    rows = rows_in * (H * (el + 2) + (0 if el == 2 else H // 128 * 4))
    routing = 8 * E if c["masked"] else T * E * 4 + T * k * 4 * 4 + 8 * E
    return {"bytes": _expected_active(c) * per_expert + rows + routing, "flops": 6.0 * T * k * H * I}


def tolerance(case):
    """Outputs pass three bf16 roundings (intermediate, expert output, result), for e4m3 one 1x128 re-quantisation of
    the intermediate on top; plan outputs and expert ids are whole numbers and exact.  Against a 64-bit evaluation (with
    that re-quantisation) the outputs are off by 2.9e-3 (2-norm), the worst value by 1.6e-2 of the rms."""
    return {"rel": 1e-2, "max": 0.06}
