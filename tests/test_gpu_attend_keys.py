"""The kernel with the keys on the MMA's rows (bf16, "auto" path), head_dim 64 and, up to 32 rows, 128.
Edges of its row counts (16, 32, 64, 128, several tiles of 128), of its key tiles, of the cluster split (CTAs without a
tile included), both masks, the block as a tensor and in the cache, NaN behind the keys.  33 to 64 rows at head_dim 128, which
the library may put there, are in test_gpu_rows_33_to_64.py; the shapes of more rows at 128 belong to the wide
kernel and stand for the other side of the line."""
import pytest
import torch

import oracle
from paper_2605_12825_b200 import workloads as W
from _gpu_util import Guarded, assert_close, binding, oracle_attend, run_attend, small_workload

pytestmark = pytest.mark.gpu
VIEWS = [oracle.VIEW_DIFFUSION, oracle.VIEW_AR]
# (Hq, Hkv, head_dim, K): 1, 4, 16, 17, 32, 33, 49, 64, then 72, 128, 129 and 320 query rows
SHAPES = [(2, 2, 64, 1), (8, 2, 64, 1), (8, 2, 64, 4), (3, 3, 64, 17), (8, 2, 64, 8), (3, 1, 64, 11), (14, 2, 64, 7), (4, 2, 64, 32),
          (1, 1, 128, 1), (8, 2, 128, 1), (8, 2, 128, 4), (2, 2, 128, 17), (16, 4, 128, 8), (7, 1, 128, 4),
          (8, 1, 128, 9), (8, 2, 64, 32), (16, 2, 128, 16), (3, 1, 128, 43), (10, 2, 64, 64)]
NAN = float("nan")


def inputs(shape, lens, hint=1024):
    Hq, Hkv, d, K = shape
    wl = small_workload(len(lens), K, Hq, Hkv, d, hint, hint, std=0.5, name=f"narrow_{Hq}_{Hkv}_{d}_{K}")
    t = W.attention_inputs(wl)
    t["cache_len"][:] = torch.tensor(lens, dtype=torch.int32)
    for b, p in enumerate(lens):
        t["k_cache"][b, :, p:, :] = NAN
        t["v_cache"][b, :, p:, :] = NAN
    return wl, t


@pytest.mark.parametrize("view", VIEWS)
@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("splits", [None, 1, 2, 3, 8, 16])
def test_shapes_and_splits(view, shape, splits):
    for lens in ([0, 1], [15, 64], [65, 130], [700, 257], [1024, 1000]):
        wl, t = inputs(shape, lens)
        got, status, used = run_attend(view, t, wl, max_len_hint=1024, splits=splits, flags=1 if splits == 16 else 0)
        assert used == "tcgen05" and status == 0
        assert_close(got, oracle_attend(view, t), torch.bfloat16, f"{shape} lens={lens} splits={splits}")


@pytest.mark.parametrize("shape", [(14, 2, 64, 7), (8, 2, 64, 1), (8, 2, 128, 1), (16, 4, 128, 8), (8, 2, 128, 20),
                                   (3, 1, 128, 43)])
@pytest.mark.parametrize("view", VIEWS)
def test_block_in_the_cache(view, shape):
    b = binding()
    Hq, Hkv, d, K = shape
    for lens in ([0, 63], [190, 1000]):
        wl, t = inputs(shape, lens)
        kb, vb = ("k_diff_blk", "v_diff_blk") if view == oracle.VIEW_DIFFUSION else ("k_ar_blk", "v_ar_blk")
        q = t["q_diff"] if view == oracle.VIEW_DIFFUSION else t["q_ar"]
        ref = oracle_attend(view, t)
        for i, p in enumerate(lens):
            t["k_cache"][i, :, p:p + K] = t[kb][i].transpose(0, 1)
            t["v_cache"][i, :, p:p + K] = t[vb][i].transpose(0, 1)
        k, v, ln = t["k_cache"].cuda(), t["v_cache"].cuda(), t["cache_len"].cuda()
        layer = b.make_layer(k, v, ln, Hq, K, 1024, 0.0, b.LAYER_BLOCK_IN_CACHE)
        ws = b.new_workspace(b.orthrus_attend_workspace_bytes(layer))
        out = Guarded(tuple(q.shape), torch.bfloat16)
        f = b.orthrus_diffusion_block_attend if view == oracle.VIEW_DIFFUSION else b.orthrus_ar_verify_attend
        f(layer, q.cuda(), None, None, out.t, ws)
        assert b.orthrus_last_path() == "tcgen05" and b.orthrus_read_status(ws) == 0 and out.intact()
        assert_close(out.t.cpu(), ref, torch.bfloat16, f"{shape} {lens}")


@pytest.mark.parametrize("shape", [(16, 4, 64, 8), (32, 8, 128, 1), (16, 4, 128, 13)])
def test_many_units_of_unequal_length(shape):
    """More clusters than fit at once: handed out longest prefix first; scores of a few units to either side."""
    lens = [int(x) for x in torch.randint(0, 3000, (40,), generator=torch.Generator().manual_seed(3))]
    wl, t = inputs(shape, lens, 3000)
    t["q_ar"] *= 8
    got, status, used = run_attend(oracle.VIEW_AR, t, wl, max_len_hint=3000)
    assert used == "tcgen05" and status == 0
    assert_close(got, oracle_attend(oracle.VIEW_AR, t), torch.bfloat16, f"{shape}")
