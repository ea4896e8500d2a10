"""The keys kernel with the block's own keys apart from the tiles, which it takes where those keys alone would be a tile more for the
longest CTA (64 rows, bounds just above sixteen CTAs of two tiles less one half): against the oracle over blocks of one to sixteen
positions, both views, the block as a tensor and in the cache, empty and short prefixes under the same bound, NaN behind the
keys, peaked scores; the line of the rule; the same numbers behind a preceding call."""
import pytest
import torch

import oracle
from paper_2605_12825_b200 import workloads as W
from _gpu_util import Guarded, assert_close, binding, captured_launches, oracle_attend, small_workload

pytestmark = pytest.mark.gpu
NAN = float("nan")


def name_of(call):
    (name, _), = captured_launches(call)
    return name


# 33 to 64 rows in one query tile, 68 to 128 in two: (Hq, Hkv, K)
@pytest.mark.parametrize("shape", [(8, 2, 9), (8, 2, 16), (7, 1, 9), (9, 1, 4), (16, 1, 4), (35, 1, 1), (6, 1, 12), (8, 1, 16)])
@pytest.mark.parametrize("view", [oracle.VIEW_DIFFUSION, oracle.VIEW_AR])
@pytest.mark.parametrize("peak", [1.0, 40.0])
@pytest.mark.parametrize("in_cache", [False, True])
def test_apart_from_the_tiles(shape, view, peak, in_cache):
    b = binding()
    Hq, Hkv, K = shape
    bound = 4096
    for lens in ([4096, 0], [4065, 1], [130, 4033]):
        wl = small_workload(2, K, Hq, Hkv, 128, bound, bound, std=0.5, name=f"apart_{Hq}_{Hkv}_{K}")
        t = W.attention_inputs(wl)
        t["cache_len"][:] = torch.tensor(lens, dtype=torch.int32)
        x = "ar" if view == oracle.VIEW_AR else "diff"
        t["q_" + x] *= peak
        for i, p in enumerate(lens):
            t["k_cache"][i, :, p:], t["v_cache"][i, :, p:] = NAN, NAN
        ref = oracle_attend(view, t)
        flags = b.LAYER_CACHE_QUIESCENT
        if in_cache:
            flags |= b.LAYER_BLOCK_IN_CACHE
            for i, p in enumerate(lens):
                t["k_cache"][i, :, p:p + K] = t[f"k_{x}_blk"][i].transpose(0, 1)
                t["v_cache"][i, :, p:p + K] = t[f"v_{x}_blk"][i].transpose(0, 1)
        g = {k: v.cuda() for k, v in t.items()}
        layer = b.make_layer(g["k_cache"], g["v_cache"], g["cache_len"], Hq, K, bound, 0.0, flags)
        ws = b.new_workspace(b.orthrus_attend_workspace_bytes(layer))
        f = b.orthrus_ar_verify_attend if view == oracle.VIEW_AR else b.orthrus_diffusion_block_attend
        blk = [None, None] if in_cache else [g[f"k_{x}_blk"], g[f"v_{x}_blk"]]
        outs = [Guarded(tuple(t["q_" + x].shape), torch.bfloat16) for _ in range(3)]
        assert "apart_attend_keys_kernel" in name_of(lambda: f(layer, g["q_" + x], *blk, outs[0].t, ws))
        for out in outs:
            f(layer, g["q_" + x], *blk, out.t, ws)
        assert b.orthrus_read_status(ws) == 0 and all(o.intact() for o in outs)
        assert_close(outs[0].t.cpu(), ref, torch.bfloat16, f"{shape} {lens} peak={peak} in_cache={in_cache}")
        assert torch.equal(outs[1].t, outs[0].t) and torch.equal(outs[2].t, outs[0].t)


@pytest.mark.parametrize("units,bound,apart", [(8, 4032, False), (8, 4033, True), (8, 4096, True), (8, 4097, False), (9, 4096, True),
                                               (8, 2000, False), (8, 6000, False), (32, 2000, False)])
def test_where_they_are_kept_apart(units, bound, apart):
    b = binding()
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("the lines are drawn for 148 SMs")
    cache = torch.empty(units, 1, bound + 16, 128, dtype=torch.bfloat16, device="cuda")
    ln = torch.zeros(units, dtype=torch.int32, device="cuda")
    q, kb = (torch.empty(units, 16, h, 128, dtype=torch.bfloat16, device="cuda") for h in (4, 1))
    layer = b.make_layer(cache, cache, ln, 4, 16, bound, 0.0, b.LAYER_CACHE_QUIESCENT)
    ws = b.new_workspace(b.orthrus_attend_workspace_bytes(layer))
    name = name_of(lambda: b.orthrus_ar_verify_attend(layer, q, kb, kb, q, ws))
    assert ("apart_attend_keys_kernel" in name) == apart and "attend_keys_kernel" in name
