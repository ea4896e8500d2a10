"""The keys kernel with its first tiles asked for ahead of the preceding kernel, several calls one behind the other: CTAs of
one to many tiles (two of them fold into three slots at head_dim 128; from three on the slots of the ring are used again), the
block's own keys alone in a tile and beside prefix keys, scores that make the references move in the first
tile of each softmax warpgroup (later ones: test_gpu_references.py)."""
import pytest
import torch

import oracle
from paper_2605_12825_b200 import workloads as W
from _gpu_util import assert_close, binding, oracle_attend, small_workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("peak", [1.0, 40.0])
@pytest.mark.parametrize("shape", [(8, 2, 64, 8), (14, 2, 64, 7), (8, 1, 64, 16), (8, 2, 128, 1), (8, 2, 128, 6), (8, 2, 128, 16)])
@pytest.mark.parametrize("splits", [1, 2, 3, 6])
def test_early_tiles_in_a_chain_of_calls(shape, splits, peak, monkeypatch):
    b = binding()
    Hq, Hkv, d, K = shape
    monkeypatch.setenv("ORTHRUS_TC_SMALL_ROWS", "1")
    monkeypatch.setenv("ORTHRUS_SPLITS", str(splits))
    for lens in ([127, 640], [193, 1024], [64, 577], [256, 576], [897, 310]):        # (256, 576, 897: five halves of 64 keys for each of 1, 2, 3 CTAs)
        wl = small_workload(2, K, Hq, Hkv, d, 1024, 1024, std=0.5, name=f"ring_{Hq}_{Hkv}_{d}_{K}")
        t = W.attention_inputs(wl)
        t["cache_len"][:] = torch.tensor(lens, dtype=torch.int32)
        t["q_ar"] *= peak                      # 40: scores of hundreds, far from the first reference on either side
        for i, p in enumerate(lens):
            t["k_cache"][i, :, p:] = float("nan")
            t["v_cache"][i, :, p:] = float("nan")
        ref = oracle_attend(oracle.VIEW_AR, t)
        g = {k: v.cuda() for k, v in t.items()}
        layer = b.make_layer(g["k_cache"], g["v_cache"], g["cache_len"], Hq, K, 1024, 0.0, b.LAYER_CACHE_QUIESCENT)
        ws = b.new_workspace(b.orthrus_attend_workspace_bytes(layer))
        outs = [torch.full_like(g["q_ar"], float("nan")) for _ in range(6)]
        for out in outs:
            b.orthrus_ar_verify_attend(layer, g["q_ar"], g["k_ar_blk"], g["v_ar_blk"], out, ws)
        assert b.orthrus_read_status(ws) == 0
        assert_close(outs[0].cpu(), ref, torch.bfloat16, f"{shape} {lens} splits={splits} peak={peak}")
        for out in outs[1:]:
            assert torch.equal(out, outs[0])
