"""Narrow calls (at most 64 query rows per KV head) over long chunks: every CTA walks dozens of key
tiles through its K and V slots while the memory is busy, so tiles land out of order.  The status
word must stay clear, repeated calls must give identical bytes, and sampled rows must match the oracle."""
import pytest
import torch

import oracle
from paper_2605_12825_b200 import workloads as W
from _gpu_util import assert_close, binding

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,Hq,Hkv,K,lo,hi", [(9, 32, 8, 6, 6492, 13713), (24, 32, 8, 16, 500, 6000), (3, 8, 8, 1, 9000, 20000)])
@pytest.mark.parametrize("flags", [0, 1])
def test_long_chunks(B, Hq, Hkv, K, lo, hi, flags):
    b = binding()
    wl = W.CONFIGS["cfg2_8b_b1"].with_(name=f"narrow_{B}_{K}", batch=B, n_q_heads=Hq, n_kv_heads=Hkv, block=K,
                                       prefix_min=lo, prefix_max=hi)
    g = torch.Generator(device="cuda").manual_seed(B)
    mk = lambda *s: torch.randn(s, generator=g, device="cuda", dtype=torch.bfloat16)
    lens = torch.linspace(lo, hi, B).round().to(torch.int32)[torch.randperm(B)]
    d = dict(k_cache=mk(B, Hkv, wl.capacity, 128), v_cache=mk(B, Hkv, wl.capacity, 128), cache_len=lens.cuda())
    q, kb, vb = mk(B, K, Hq, 128), mk(B, K, Hkv, 128), mk(B, K, Hkv, 128)
    layer = b.make_layer(d["k_cache"], d["v_cache"], d["cache_len"], Hq, K, hi, 0.0, flags)
    ws = b.new_workspace(b.orthrus_attend_workspace_bytes(layer))
    outs = [torch.empty_like(q) for _ in range(60)]
    for o in outs:
        b.orthrus_ar_verify_attend(layer, q, kb, vb, o, ws)
    assert b.orthrus_read_status(ws) == 0
    for o in outs[1:]:
        assert torch.equal(o.view(torch.int16), outs[0].view(torch.int16))
    i = int(lens.argmax())
    one = lambda t: t[i:i + 1].cpu().contiguous()
    ref = oracle.block_attend(oracle.VIEW_AR, one(q), one(kb), one(vb), one(d["k_cache"]), one(d["v_cache"]), lens[i:i + 1].contiguous())
    assert_close(one(outs[0]), ref, torch.bfloat16, f"B={B} K={K}")
