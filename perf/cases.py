"""Performance cases of the generation-step library: what a program that decodes with it has it do.

A case is one of five kinds of work, all through the functions of the package's binding:

  cycle       one generation cycle on the append commit: the diffusion view through all layers, the
              AR view through all layers, the greedy consensus on the AR logits, the commit of the
              accepted rows of all layers
  in_place    the same cycle on the write-then-truncate commit, as the decoder around the library
              runs it: rotary write and attention per layer and view, the consensus taken from the
              last hidden states and the LM head, the commit a length bump.  With `views` = 1 and
              `block` = 1 it is one step of plain autoregressive decoding
  sample      the sampled consensus (temperature > 0) on the logits of both views
  lm_head     the greedy consensus from hidden states and LM head
  multi       the multi-block diffusion attention of the training-time mask, anchors increasing

Inputs are random tensors of the shapes and scales of `paper_2605_12825_b200/workloads.py`, drawn on the
GPU.  The prefix lengths of a batch are spread evenly over their range and dealt to the sequences
by the seed, so that every seed is the same amount of work.
"""
import math

import torch

from paper_2605_12825_b200 import binding as B

DEV = "cuda"
BF16 = torch.bfloat16
THETA = 10000.0


def _cycle(name, batch, heads, kv_heads, head_dim, block, vocab, prefix_min, prefix_max, layers, logits="bf16"):
    return dict(name=name, kind="cycle", batch=batch, heads=heads, kv_heads=kv_heads, head_dim=head_dim, block=block,
                vocab=vocab, prefix_min=prefix_min, prefix_max=prefix_max, layers=layers, logits=logits)


def _in_place(name, batch, heads, kv_heads, block, vocab, hidden, prefix_min, prefix_max, room, layers, views):
    return dict(name=name, kind="in_place", batch=batch, heads=heads, kv_heads=kv_heads, head_dim=128, block=block,
                vocab=vocab, hidden=hidden, prefix_min=prefix_min, prefix_max=prefix_max, room=room, layers=layers,
                views=views)


def listed():
    return [
        # the smallest model: a short prompt, one layer, every call a few microseconds
        _cycle("tiny", 1, 8, 2, 64, 8, 1000, 512, 512, 1),
        # one conversation on an 8B-class model, all 36 layers: the latency case of the headline metric, whose prefix
        # of about four thousand positions is any length in earnest
        _cycle("8b_batch1", 1, 32, 8, 128, 16, 151936, 4000, 4000, 36),
        # a serving batch of unequal lengths, wide blocks, one layer and the consensus of the whole batch
        _cycle("serving_ragged", 32, 32, 8, 128, 32, 128256, 1024, 8192, 1),
        # long documents, eight query heads per KV head
        _cycle("long_context", 4, 64, 8, 128, 16, 151936, 32768, 32768, 1),
        # a small model with 64-wide heads, odd sizes throughout, logits kept in fp32
        _cycle("odd_d64", 5, 14, 2, 64, 7, 50257, 77, 1531, 6, "fp32"),
        # the end-to-end decoder on the write-then-truncate commit
        _in_place("decoder_loop", 8, 16, 4, 16, 32000, 2048, 1700, 1980, 512, 12, 2),
        # plain autoregressive decoding of two conversations through the same calls
        _in_place("decode_width1", 2, 32, 8, 1, 32000, 2048, 1500, 3900, 128, 24, 1),
        # consensus by rejection sampling: one conversation, then the serving batch
        dict(name="sample_batch1", kind="sample", batch=1, block=16, vocab=151936, temperature=0.7),
        dict(name="sample_serving", kind="sample", batch=32, block=32, vocab=128256, temperature=1.0),
        # consensus straight from the hidden states: one conversation (the LM head is streamed), the serving batch
        # (a dense product)
        dict(name="lm_head_batch1", kind="lm_head", batch=1, block=16, vocab=151936, hidden=4096),
        dict(name="lm_head_serving", kind="lm_head", batch=32, block=32, vocab=128256, hidden=4096),
        # the diffusion view over many anchored blocks per sequence (the forward pass of training)
        dict(name="multi_block", kind="multi", batch=4, heads=32, kv_heads=8, head_dim=128, block=8, blocks=32,
             prefix_max=4096),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, round(math.exp(rng.uniform(math.log(lo), math.log(hi))))))


def _narrow_limit(c):
    """Longest prefix drawn for calls of at most 64 query rows per KV head: four 64-position tiles for each of the
    thread blocks that share a KV head.  The kernel for such calls could lose a barrier phase on longer chunks
    before that was corrected, so that longer ones have no earlier time to compare with."""
    splits = 1
    while splits < 16 and splits * 2 * c["batch"] * c["kv_heads"] <= 2 * 148:
        splits *= 2
    return 64 * (4 * splits - 1)


def draw(rng):
    """Sizes spread over the ranges of the listed cases; a draw that would cost more than the largest of them is
    made smaller in its number of layers, then in its lengths."""
    kind = rng.choice(["cycle", "cycle", "cycle", "in_place", "in_place", "sample", "lm_head", "multi"])
    heads, kv_heads = rng.choice([(8, 2), (14, 2), (16, 4), (16, 8), (32, 8), (64, 8)])
    group, most = heads // kv_heads, 1.2e9
    if kind == "cycle":
        c = _cycle(None, _log_int(rng, 1, 32), heads, kv_heads, rng.choice([64, 128, 128]), _log_int(rng, 4, 32),
                   _log_int(rng, 1000, 152000), 1, _log_int(rng, 100, 32768), _log_int(rng, 1, 36),
                   rng.choice(["bf16", "bf16", "fp32"]))
    elif kind == "in_place":
        views = rng.choice([1, 2, 2])
        c = _in_place(None, _log_int(rng, 1, 32), heads, kv_heads, 1 if views == 1 else _log_int(rng, 4, 32),
                      _log_int(rng, 4000, 152000), 8 * _log_int(rng, 64, 512), 1, _log_int(rng, 100, 16384),
                      _log_int(rng, 64, 512), _log_int(rng, 1, 24), views)
    elif kind == "sample":
        c = dict(kind=kind, batch=_log_int(rng, 1, 32), block=_log_int(rng, 4, 32), vocab=_log_int(rng, 8000, 152000),
                 temperature=round(rng.uniform(0.5, 1.2), 2))
    elif kind == "lm_head":
        c = dict(kind=kind, batch=_log_int(rng, 1, 32), block=_log_int(rng, 1, 32), vocab=_log_int(rng, 8000, 128256),
                 hidden=8 * _log_int(rng, 64, 512))
    else:
        c = dict(kind=kind, batch=_log_int(rng, 1, 8), heads=heads, kv_heads=kv_heads, head_dim=128,
                 block=_log_int(rng, 4, 16), blocks=_log_int(rng, 2, 48), prefix_max=_log_int(rng, 256, 8192))
    c.pop("name", None)
    if kind in ("cycle", "in_place") and c["head_dim"] == 128 and group * c["block"] <= 64:
        if c["block"] > 1 and group > 2 and rng.random() < 0.5:
            c["block"] = rng.randint(64 // group + 1, 32)
        else:
            c["prefix_max"] = min(c["prefix_max"], _narrow_limit(c))
    if "prefix_min" in c:
        c["prefix_min"] = max(1, round(c["prefix_max"] * rng.uniform(0.1, 1.0)))
    while work(c)["bytes"] > most:
        if c.get("layers", 1) > 1:
            c["layers"] //= 2
        elif "prefix_max" in c and c["prefix_max"] > 100:
            c["prefix_max"] //= 2
            c["prefix_min"] = max(1, c["prefix_min"] // 2)
        else:
            c["batch"] = max(1, c["batch"] // 2)
    return c


# ---------------------------------------------------------------------------- inputs

def _generator(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(12825 + seed)
    return g


def _normal(g, shape, std, dtype=BF16):
    return torch.randn(shape, generator=g, device=DEV, dtype=dtype).mul_(std)


def _i32(*shape):
    return torch.zeros(shape, dtype=torch.int32, device=DEV)


def _lengths(c):
    n = c["batch"]
    step = (c["prefix_max"] - c["prefix_min"]) / max(1, n - 1)
    return [round(c["prefix_max"] - step * i) for i in range(n)]


def _capacity(c):
    return (c["prefix_max"] + c["block"] + c.get("room", 0) + 63) // 64 * 64


def _outputs(c):
    b, k = c["batch"], c["block"]
    return dict(n_commit=_i32(b), committed=_i32(b, k), ar_argmax=_i32(b, k), next_anchor=_i32(b))


def _drafts(g, greedy, vocab, rate):
    """Drafts that agree with the greedy tokens at the given rate and are uniform otherwise."""
    coin = torch.rand(greedy.shape, generator=g, device=DEV) < rate
    other = torch.randint(0, vocab, greedy.shape, generator=g, device=DEV)
    return torch.where(coin, greedy, other).to(torch.int32)


def _hidden_and_head(g, c):
    """Last hidden states that lean towards one vocabulary entry each, as a trained model's do, and the LM head."""
    b, k, v, h = c["batch"], c["block"], c["vocab"], c["hidden"]
    head = _normal(g, (v, h), 1.0 / math.sqrt(h))
    greedy = torch.randint(0, v, (b, k), generator=g, device=DEV)
    hidden = _normal(g, (b, k, h), 1.0) + 8.0 * head[greedy]
    return hidden, head, _drafts(g, greedy, v, 0.65)


def _attention_state(g, c, flags):
    """Caches, lengths and per-layer block tensors of both views, in one tensor per kind."""
    b, k, hq, hkv, d, n = c["batch"], c["block"], c["heads"], c["kv_heads"], c["head_dim"], c["layers"]
    views, cap, std = c.get("views", 2), _capacity(c), 1.0 / math.sqrt(d)
    lens = torch.tensor(_lengths(c), dtype=torch.int32, device=DEV)
    lens = lens[torch.randperm(b, generator=g, device=DEV)].contiguous()
    s = dict(len0=lens, cache_len=lens.clone(),
             k_cache=_normal(g, (n, b, hkv, cap, d), std), v_cache=_normal(g, (n, b, hkv, cap, d), std),
             q=_normal(g, (views, n, b, k, hq, d), std), k_blk=_normal(g, (views, n, b, k, hkv, d), std),
             v_blk=_normal(g, (views, n, b, k, hkv, d), std), out=torch.empty((views, n, b, k, hq, d), dtype=BF16, device=DEV))
    # a decoder that lets the cache fill up bounds the lengths by its capacity, others know them
    hint = cap - k if "room" in c else c["prefix_max"]
    s["layers"] = [B.make_layer(s["k_cache"][i], s["v_cache"][i], s["cache_len"], hq, k, hint, 0.0, flags) for i in range(n)]
    # the call behind the kernel that sets the lengths back reads nothing early
    s["first"] = B.make_layer(s["k_cache"][0], s["v_cache"][0], s["cache_len"], hq, k, hint, 0.0,
                              flags & ~B.LAYER_CACHE_QUIESCENT)
    s["ws"] = B.new_workspace(B.orthrus_attend_workspace_bytes(s["layers"][0]))
    return s


def prepare(case, seed):
    c, g = case, _generator(seed)
    b, k = c["batch"], c["block"]
    if c["kind"] == "cycle":
        s = _attention_state(g, c, B.LAYER_CACHE_QUIESCENT)
        s["logits"] = _normal(g, (b, k, c["vocab"]), 2.0, torch.float32 if c["logits"] == "fp32" else BF16)
        s["draft"] = _drafts(g, s["logits"].argmax(-1), c["vocab"], 0.6)
        s["cws"] = B.new_workspace(B.orthrus_consensus_workspace_bytes(b, k, c["vocab"]))
        s["k_ar"], s["v_ar"] = list(s["k_blk"][1]), list(s["v_blk"][1])
        s["res"] = _outputs(c)
        # per view and layer: the arguments of the attention call
        s["calls"] = [[(s["layers"][i] if i or w else s["first"], s["q"][w][i], s["k_blk"][w][i], s["v_blk"][w][i],
                        s["out"][w][i]) for i in range(c["layers"])] for w in (0, 1)]
    elif c["kind"] == "in_place":
        s = _attention_state(g, c, B.LAYER_CACHE_QUIESCENT | B.LAYER_BLOCK_IN_CACHE)
        s["hidden"], s["head"], s["draft"] = _hidden_and_head(g, c)
        s["cws"] = B.new_workspace(B.orthrus_lm_head_consensus_workspace_bytes(b, k, c["vocab"]))
        s["q_rot"] = torch.empty_like(s["q"])
        s["res"] = _outputs(c)
        s["calls"] = [[(s["layers"][i], s["q"][w][i], s["k_blk"][w][i], s["v_blk"][w][i], s["q_rot"][w][i], s["out"][w][i])
                       for i in range(c["layers"])] for w in range(c["views"])]
    elif c["kind"] == "sample":
        shape = (b, k, c["vocab"])
        ar = _normal(g, shape, 2.0)
        diff = ar + _normal(g, shape, 0.4)
        # drafts drawn from the diffusion view's distribution
        gumbel = torch.empty(shape, device=DEV).exponential_(generator=g).log_().neg_()
        draft = gumbel.add_(diff, alpha=1.0 / c["temperature"]).argmax(-1).to(torch.int32)
        s = dict(ar=ar, diff=diff, draft=draft, u=torch.rand((b, k), generator=g, device=DEV),
                 u2=torch.rand((b, k), generator=g, device=DEV), t=c["temperature"],
                 cws=B.new_workspace(B.orthrus_consensus_sample_workspace_bytes(b, k, c["vocab"])), res=_outputs(c))
        del s["res"]["ar_argmax"]
    elif c["kind"] == "lm_head":
        s = dict(res=_outputs(c), cws=B.new_workspace(B.orthrus_lm_head_consensus_workspace_bytes(b, k, c["vocab"])))
        s["hidden"], s["head"], s["draft"] = _hidden_and_head(g, c)
    else:
        n, hq, hkv, d, top = c["blocks"], c["heads"], c["kv_heads"], c["head_dim"], c["prefix_max"]
        std, cap = 1.0 / math.sqrt(d), (top + k + 63) // 64 * 64
        jitter = torch.rand((b, n), generator=g, device=DEV) - 0.5
        anchors = (torch.arange(1, n + 1, device=DEV) + 0.5 * jitter) * (top / n)
        anchors[:, -1] = top
        s = dict(anchors=anchors.to(torch.int32).contiguous(), k_cache=_normal(g, (b, hkv, cap, d), std),
                 v_cache=_normal(g, (b, hkv, cap, d), std), q=_normal(g, (b, n, k, hq, d), std),
                 k_blk=_normal(g, (b, n, k, hkv, d), std), v_blk=_normal(g, (b, n, k, hkv, d), std),
                 len=torch.full((b,), top, dtype=torch.int32, device=DEV))
        s["out"] = torch.empty_like(s["q"])
        s["layer"] = B.make_layer(s["k_cache"], s["v_cache"], s["len"], hq, k, top)
        s["ws"] = B.new_workspace(B.orthrus_multi_block_workspace_bytes(s["layer"], n))
    s["kind"] = c["kind"]
    return s


# ---------------------------------------------------------------------------- one pass

def run(state):
    s = state
    kind = s["kind"]
    if kind == "cycle":
        ws, res = s["ws"], s["res"]
        s["cache_len"].copy_(s["len0"])           # the same cycle again: the lengths of its start
        for layer, q, k, v, out in s["calls"][0]:
            B.orthrus_diffusion_block_attend(layer, q, k, v, out, ws)
        for layer, q, k, v, out in s["calls"][1]:
            B.orthrus_ar_verify_attend(layer, q, k, v, out, ws)
        B.orthrus_consensus_accept(s["logits"], s["draft"], res["n_commit"], res["committed"], res["ar_argmax"],
                                   res["next_anchor"], s["cws"])
        if len(s["layers"]) == 1:
            B.orthrus_kv_append(s["layers"][0], s["k_ar"][0], s["v_ar"][0], res["n_commit"], True, ws)
        else:
            B.orthrus_kv_append_layers(s["layers"], s["k_ar"], s["v_ar"], res["n_commit"], True, ws)
        return dict(res, out=s["out"], k_cache=s["k_cache"], v_cache=s["v_cache"], cache_len=s["cache_len"])
    if kind == "in_place":
        ws, res, calls = s["ws"], s["res"], s["calls"]
        s["cache_len"].copy_(s["len0"])
        if len(calls) == 2:
            for layer, q, k, v, q_rot, out in calls[0]:
                B.orthrus_rope_block_kv_write(layer, q, k, v, THETA, q_rot, ws)
                B.orthrus_diffusion_block_attend(layer, q_rot, None, None, out, ws)
        for layer, q, k, v, q_rot, out in calls[-1]:
            B.orthrus_rope_block_kv_write(layer, q, k, v, THETA, q_rot, ws)
            B.orthrus_ar_verify_attend(layer, q_rot, None, None, out, ws)
        B.orthrus_lm_head_consensus(s["hidden"], s["head"], s["draft"], res["n_commit"], res["committed"],
                                    res["ar_argmax"], res["next_anchor"], s["cws"])
        B.orthrus_commit_len(s["layers"][0], res["n_commit"], ws)
        return dict(res, out=s["out"], q_rot=s["q_rot"], k_cache=s["k_cache"], v_cache=s["v_cache"],
                    cache_len=s["cache_len"])
    if kind == "sample":
        res = s["res"]
        B.orthrus_consensus_sample(s["ar"], s["diff"], s["draft"], s["u"], s["u2"], s["t"], res["n_commit"],
                                   res["committed"], res["next_anchor"], s["cws"])
        return res
    if kind == "lm_head":
        res = s["res"]
        B.orthrus_lm_head_consensus(s["hidden"], s["head"], s["draft"], res["n_commit"], res["committed"],
                                    res["ar_argmax"], res["next_anchor"], s["cws"])
        return res
    B.orthrus_multi_block_attend(s["layer"], s["anchors"], s["q"], s["k_blk"], s["v_blk"], s["out"], s["ws"])
    return s["out"]


# ---------------------------------------------------------------------------- what a pass cannot do without

def work(case):
    c = case
    b, k = c["batch"], c["block"]
    kind, ints = c["kind"], 4 * (3 * b * k + 2 * b)
    nbytes = flops = 0
    if kind in ("cycle", "in_place"):
        hq, hkv, d, n, views = c["heads"], c["kv_heads"], c["head_dim"], c["layers"], c.get("views", 2)
        total = sum(_lengths(c))
        # per view and layer: every prefix row once, the block's K and V, queries in, outputs out
        call = hkv * 4 * d * (total + b * k) + b * k * hq * 4 * d
        if kind == "in_place":                    # raw and rotated queries, the block's rows written
            call += b * k * d * 4 * (hq + hkv)
        nbytes += views * n * call
        flops += views * n * 4 * hq * k * d * (total + b * k)
        if kind == "cycle":                       # logits in, drafts in, tokens out, accepted rows (about 2.5) moved
            nbytes += b * k * c["vocab"] * (4 if c["logits"] == "fp32" else 2) + ints
            nbytes += n * b * min(k, 2.5) * hkv * d * 8
    if kind in ("lm_head", "in_place"):
        nbytes += 2 * c["hidden"] * (c["vocab"] + b * k) + ints
        flops += 2 * b * k * c["vocab"] * c["hidden"]
    if kind == "sample":
        # verification stops at the first rejected draft: about six rows of both views, then the rejected one
        rows = b * min(k, 6)
        nbytes += rows * c["vocab"] * 4 + ints
        flops += rows * c["vocab"] * 4
    if kind == "multi":
        hq, hkv, d, n, top = c["heads"], c["kv_heads"], c["head_dim"], c["blocks"], c["prefix_max"]
        nbytes += b * (hkv * 4 * d * (top + n * k) + n * k * hq * 4 * d + 4 * n)
        flops += 4 * b * hq * k * d * n * (top * (n + 1) / (2 * n) + k)
    return dict(bytes=nbytes, flops=flops)


def tolerance(case):
    """Attention in bf16: probabilities and outputs are rounded to 8 bits.  Greedy tokens of given logits are exact;
    those of the LM-head product and the sampled ones may differ where two candidates are within rounding."""
    if case["kind"] == "cycle":
        return dict(rel=1e-2, max=0.1)
    if case["kind"] == "in_place":
        return dict(rel=1e-2, max=0.1, differ=0.005)
    if case["kind"] == "multi":
        return dict(rel=1e-2, max=0.1)
    return dict(rel=0.0, differ=0.005)
