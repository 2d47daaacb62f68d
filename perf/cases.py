"""The work that a user of this library has it do, as timed cases.

Each case is one pass through the public entry points of `paper_2503_17922_b200.binding`, as an inference
engine drives them while it prefills: a whole layer group in one call or replayed from a plan, layer by
layer, into a compact, packed or paged cache or inside the layer's own buffer, from device or host memory.

Fields of a case:
  kind       which entry points the pass uses, one of KINDS
  dtype      "bf16" or "f32"
  batch      sequences;  ragged: True = packed [T, H_kv, d] of different lengths, False = dense, all of length n
  q_heads, kv_heads, d   attention shape
  n          context length (the longest, when ragged)
  alpha      observation window;  window: review window;  task: 0 localization, 1 aggregation
  layers     layers of the group
  budget     retained tokens per layer in thousandths of the sequence's length
  layout     "bhnd" or "bnhd" (token-major) for dense keys and values
"""
import math
import random

import numpy as np
import torch

from paper_2503_17922_b200 import binding as wkv

KINDS = ("group", "plan", "stream", "inplace", "paged", "score", "host")

_LARGEST = {"bytes": 3.5e9, "flops": 1.9e11}     # what the largest listed case cannot do without

_LLAMA = dict(dtype="bf16", batch=1, ragged=False, q_heads=32, kv_heads=8, d=128, layout="bhnd")


def _case(kind, **kw):
    c = dict(_LLAMA, kind=kind, alpha=32, window=16, task=1, layers=4, budget=120)
    c.update(kw)
    return c


def listed():
    return [
        # a unit test's or a toy model's group in fp32: nothing but latency
        _case("group", name="tiny-fp32-group", dtype="f32", q_heads=4, kv_heads=2, d=64, n=1024, alpha=8, window=8,
              task=0, layers=2, budget=125),
        # a needle lookup in a short prompt, 128 tokens kept
        _case("group", name="needle-4k-group", n=4096, alpha=16, window=8, task=0, budget=32),
        # an ordinary prompt, one call per group
        _case("group", name="llama-8k-group", n=8192, window=8, task=0),
        # the same model at full context, its group recorded once and replayed per prompt
        _case("plan", name="llama-32k-plan", n=32768),
        # a serving batch of long documents, ragged and packed: the largest
        _case("group", name="batch-64k-group", batch=8, ragged=True, n=65536, alpha=64, window=32, layers=8),
        # a model with six query heads per key head and seven layers per group, ragged prompts of odd lengths,
        # packed compact cache
        _case("group", name="g6-ragged-group", batch=3, ragged=True, q_heads=12, kv_heads=2, n=12289, alpha=16, window=32,
              layers=7),
        # prefill layer by layer with the attention's own normalisers: leader's selection, then each layer's gather
        _case("stream", name="llama-32k-stream", n=32768),
        # prefill that keeps each layer's compact cache in the layer's own buffer, layer by layer
        _case("inplace", name="llama-16k-inplace", n=16384),
        # a serving engine with token-major tensors and a block table
        _case("paged", name="paged-24k", n=24576, layout="bnhd", batch=2),
        # scores for inspection (per token too) and a separate selection; wide windows, head dimension 64, odd length
        _case("score", name="wide-window-20k-score", batch=2, q_heads=16, d=64, n=20011, window=128),
        # a model kept in fp32
        _case("group", name="fp32-6k-group", dtype="f32", q_heads=16, kv_heads=4, d=64, n=6000, alpha=16, window=8),
        # keys and values offloaded to pinned host memory
        _case("host", name="llama-8k-host", n=8192, window=8, task=0),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(KINDS + ("group", "group", "fp32"))
    c = _case("group" if kind == "fp32" else kind, task=rng.randrange(2), window=rng.choice((8, 16, 32)),
              alpha=rng.choice((8, 16, 32, 64)), layers=rng.randint(2, 8), budget=_log(rng, 30, 240))
    heads = rng.choice(((32, 8), (32, 8), (12, 2), (28, 4), (16, 8)))
    c["q_heads"], c["kv_heads"] = heads
    if heads[0] // heads[1] * c["alpha"] > 256:
        c["alpha"] = 32
    if kind == "fp32":
        c.update(dtype="f32", d=64, n=_log(rng, 600, 6000), q_heads=rng.choice((4, 8, 16)), kv_heads=rng.choice((2, 4)),
                 alpha=rng.choice((8, 16)), window=8)
    elif kind == "group":
        c["n"] = _log(rng, 1500, 65536)
        c["batch"] = rng.randint(1, 8)
        c["ragged"] = c["batch"] > 1
    elif kind == "score":
        c.update(n=_log(rng, 2000, 40000), batch=rng.randint(1, 4), d=rng.choice((64, 128)),
                 window=rng.choice((16, 32, 64, 128)))
    elif kind == "paged":
        c.update(n=_log(rng, 4000, 32768), batch=rng.randint(1, 4), layout="bnhd")
    elif kind == "host":
        c.update(n=_log(rng, 2000, 12000), layers=rng.randint(2, 4))
    else:                       # plan, stream, inplace: one prompt at a time
        c["n"] = _log(rng, 2000, 65536)
    # room for a few windows even in the shortest sequence of the batch
    c["budget"] = max(c["budget"], -(-1000 * (c["alpha"] + 4 * c["window"]) // (c["n"] // 2)))
    while c["batch"] > 1 and any(v > _LARGEST[m] for m, v in work(c).items()):
        c["batch"] -= 1
    return c


def _lengths(c):
    """The sequences' lengths: part of the case, not of its inputs."""
    if not c["ragged"]:
        return [c["n"]] * c["batch"]
    r = random.Random(c["n"] * 1000 + c["batch"])
    return [c["n"]] + [r.randint(c["n"] // 2, c["n"]) for _ in range(c["batch"] - 1)]


def _budgets(c):
    return [n * c["budget"] // 1000 for n in _lengths(c)]


def _keep(c):
    """Per sequence: rows of the compact cache of one head."""
    return [min((b - c["alpha"]) // c["window"] * c["window"] if b > c["alpha"] else 0, n - c["alpha"]) + c["alpha"]
            for n, b in zip(_lengths(c), _budgets(c))]


_DT = {"bf16": torch.bfloat16, "f32": torch.float32}


def _log_normalisers(c, q, k, lens, offs):
    """Natural-log normalisers of the observation rows' causal softmax, as a prefill attention leaves them."""
    B, H, G, a, d = c["batch"], c["kv_heads"], c["q_heads"] // c["kv_heads"], c["alpha"], c["d"]
    out = torch.empty((B, c["q_heads"], a), dtype=torch.float32, device="cuda")
    for b, n in enumerate(lens):
        kb = k[b] if offs is None else k[offs[b]:offs[b] + n].transpose(0, 1)
        if c["layout"] == "bnhd" and offs is None:
            kb = kb.transpose(0, 1)
        for h in range(H):
            s = q[b, h * G:(h + 1) * G].reshape(G * a, d).float() @ kb[h].float().T / math.sqrt(d)
            hide = torch.ones((a, a), dtype=torch.bool, device="cuda").triu(1).repeat(G, 1)
            s[:, n - a:].masked_fill_(hide, float("-inf"))
            out[b, h * G:(h + 1) * G] = torch.logsumexp(s, dim=1).view(G, a)
    return out


def _inputs(c, seed):
    """Queries of the observation rows, keys and values of every layer.  N(0, 1) with heavy-tailed key norms; the
    leader's keys lean toward or away from the observation queries by an amount of their own for every 16 tokens,
    so that attention mass is spread as unevenly over a prompt as it is in earnest."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    B, H, d, a, G = c["batch"], c["kv_heads"], c["d"], c["alpha"], c["q_heads"] // c["kv_heads"]
    dt, lens = _DT[c["dtype"]], _lengths(c)
    offs = [sum(lens[:b]) for b in range(B)] if c["ragged"] else None
    if c["ragged"]:
        shape = (sum(lens), H, d)
    else:
        shape = (B, H, c["n"], d) if c["layout"] == "bhnd" else (B, c["n"], H, d)

    def normal(*sh, dtype=dt):
        return torch.randn(sh, dtype=dtype, device="cuda", generator=gen)

    q = normal(B, c["q_heads"], a, d)
    ks, vs = [normal(*shape) for _ in range(c["layers"])], [normal(*shape) for _ in range(c["layers"])]
    for b, n in enumerate(lens):
        u = torch.nn.functional.normalize(q[b].float().view(H, G * a, d).sum(1), dim=1) * math.sqrt(G * a)
        lean = normal(H, -(-n // 16), dtype=torch.float32).repeat_interleave(16, dim=1)[:, :n]
        norm = torch.exp(0.5 * normal(H, n, dtype=torch.float32) - 0.125)
        # [H, n, d] view of the sequence's keys in the tensor
        kb = ks[0][offs[b]:offs[b] + n].transpose(0, 1) if c["ragged"] else ks[0][b]
        if c["layout"] == "bnhd" and not c["ragged"]:
            kb = kb.transpose(0, 1)
        for h in range(H):
            kb[h] = (kb[h].float() * norm[h, :, None] + lean[h, :, None] * u[h]).to(dt)
    return q, ks, vs, lens, offs


class _State:
    """What a user's program has in hand: tensors, the problem's shape, workspace, outputs, perhaps a plan."""


def prepare(case, seed):
    c, s = case, _State()
    s.kind, dt = c["kind"], _DT[c["dtype"]]
    s.q, s.k, s.v, lens, offs = _inputs(c, seed)
    cu = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32) if c["ragged"] else None
    s.prob = wkv.Problem(dtype=c["dtype"], batch=c["batch"], n_q_heads=c["q_heads"], n_kv_heads=c["kv_heads"],
                         head_dim=c["d"], l_obs=c["alpha"], window=c["window"], task=c["task"],
                         top_p=max(1, c["window"] // 2), max_seqlen=c["n"], budgets=_budgets(c), cu_seqlens=cu,
                         kv_layout=c["layout"])
    s.work = s.prob.alloc_workspace()
    B, H, d, L, cap = c["batch"], c["kv_heads"], c["d"], c["layers"], s.prob.keep_max

    def zeros(*shape, dtype=dt):
        return torch.zeros(shape, dtype=dtype, device="cuda")

    s.ws = zeros(B, H, s.prob.kw_max, dtype=torch.float32)
    s.idx, s.kept = zeros(B, H, s.prob.k_max, dtype=torch.int32), zeros(B, H, dtype=torch.int32)
    s.cap, s.cu_out = cap, None
    if s.kind == "group" and c["ragged"]:
        # sequences behind one another in the compact cache as they are in the full one
        rows = np.concatenate([[0], np.cumsum(_keep(c))]).astype(np.int32)
        s.cu_out, shape = torch.from_numpy(rows).cuda(), (int(rows[-1]), H, d)
    elif s.kind == "paged":
        # pages of 64 tokens, handed out in no order
        s.page = 64
        per = -(-cap // s.page)
        s.pages, shape = B * per, (B * per, s.page, H, d)
        order = np.random.default_rng(seed).permutation(s.pages).astype(np.int32)
        s.table = torch.from_numpy(order.reshape(B, per)).cuda()
    else:
        shape = (B, H, cap, d)
    outs = 0 if s.kind in ("inplace", "score") else L
    s.k_out, s.v_out = [zeros(*shape) for _ in range(outs)], [zeros(*shape) for _ in range(outs)]
    if s.kind == "stream":
        s.lse = _log_normalisers(c, s.q, s.k[0], lens, offs)
    elif s.kind == "plan":
        s.plan = wkv.GroupPlan(s.prob, s.q, s.k, s.v, s.k_out, s.v_out, s.ws, s.idx, s.kept, s.work, keep_capacity=cap)
    elif s.kind == "inplace":
        wkv.wkv_select_leader_windows(s.prob, s.q, s.k[0], s.ws, s.idx, s.kept, s.work)
    elif s.kind == "score":
        s.k, s.v = s.k[:1], []
        s.tok = zeros(B, H, s.prob.nr_max, dtype=torch.float32)
    elif s.kind == "host":
        def pinned(t, fill=True):
            p = torch.empty(t.shape, dtype=t.dtype, pin_memory=True)
            return p.copy_(t) if fill else p
        s.h_q, s.h_k, s.h_v = pinned(s.q), [pinned(t) for t in s.k], [pinned(t) for t in s.v]
        s.h_k_out, s.h_v_out = [pinned(t) for t in s.k_out], [pinned(t) for t in s.v_out]
        s.h_idx, s.h_kept = pinned(s.idx), pinned(s.kept)
        for t in [s.q] + s.k + s.v:      # staging on the device
            t.zero_()
    return s


def run(s):
    if s.kind == "group":
        wkv.wkv_compress_group(s.prob, s.q, s.k, s.v, s.k_out, s.v_out, s.ws, s.idx, s.kept, s.work,
                               cu_seqlens_out=s.cu_out, keep_capacity=0 if s.cu_out is not None else s.cap)
    elif s.kind == "plan":
        s.plan.launch()
    elif s.kind == "stream":
        wkv.wkv_select_leader_windows(s.prob, s.q, s.k[0], s.ws, s.idx, s.kept, s.work, lse_obs=s.lse)
        for layer in range(len(s.k)):
            wkv.wkv_gather_kv(s.prob, s.k[layer:layer + 1], s.v[layer:layer + 1], s.idx, s.k_out[layer:layer + 1],
                              s.v_out[layer:layer + 1], keep_capacity=s.cap)
    elif s.kind == "inplace":
        for layer in range(len(s.k)):
            wkv.wkv_compact_kv_inplace(s.prob, s.k[layer:layer + 1], s.v[layer:layer + 1], s.idx)
        return {"k": s.k, "v": s.v}
    elif s.kind == "paged":
        H, d = s.k_out[0].shape[2:]
        wkv.wkv_select_leader_windows(s.prob, s.q, s.k[0], s.ws, s.idx, s.kept, s.work)
        wkv.wkv_gather_kv_paged(s.prob, s.k, s.v, s.idx, s.k_out, s.v_out, s.table, s.page, s.pages, s.page * H * d, d,
                                H * d)
    elif s.kind == "score":
        wkv.wkv_score_windows(s.prob, s.q, s.k[0], s.ws, s.tok, s.work)
        wkv.wkv_select_topk_windows(s.prob, s.ws, s.idx, s.kept)
        return {"window_scores": s.ws, "token_scores": s.tok, "window_idx": s.idx, "kept_len": s.kept}
    elif s.kind == "host":
        wkv.wkv_compress_group_host(s.prob, s.h_q, s.h_k, s.h_v, s.h_k_out, s.h_v_out, s.h_idx, s.h_kept, s.q, s.k, s.v,
                                    s.k_out, s.v_out, s.idx, s.kept, s.cap, s.work)
        return {"window_idx": s.h_idx, "kept_len": s.h_kept, "k": s.h_k_out, "v": s.h_v_out}
    return {"window_scores": s.ws, "window_idx": s.idx, "kept_len": s.kept, "k": s.k_out, "v": s.v_out}


def work(case):
    """The leader's keys once, the retained rows of every other tensor read once, all retained rows written once, the
    scores and indices written once; one contraction of the observation rows with the leader's keys.  The retained rows
    of the leader's keys are read already, except where the pass is only a compaction."""
    c = case
    e, H = (2 if c["dtype"] == "bf16" else 4), c["kv_heads"]
    row = c["d"] * e
    keys = sum(_lengths(c)) * H * row
    kept = sum(_keep(c)) * H * row
    windows = sum(-(-(n - c["alpha"]) // c["window"]) for n in _lengths(c)) * H
    chosen = sum((m - c["alpha"]) // c["window"] for m in _keep(c)) * H
    q = c["batch"] * c["q_heads"] * c["alpha"] * row
    flops = 2.0 * c["q_heads"] * c["alpha"] * c["d"] * sum(_lengths(c))
    if c["kind"] == "inplace":
        return {"bytes": 4 * c["layers"] * kept + 4 * chosen, "flops": 0}
    if c["kind"] == "score":
        return {"bytes": keys + q + 4 * windows + 4 * chosen + 4 * H * sum(n - c["alpha"] for n in _lengths(c)), "flops": flops}
    return {"bytes": keys + q + 4 * windows + 4 * chosen + (4 * c["layers"] - 1) * kept, "flops": flops}


def tolerance(case):
    """Rows are copied bit for bit and scores are 32-bit sums.  Two windows whose scores lie within the sums' rounding
    of one another at the budget's edge may change places, which moves the rest of that head's list by one."""
    if case["kind"] == "inplace":
        return "exact"
    return {"rel": 1e-5, "max": 1e-4, "differ": 0.01}
