"""65 to 128 query rows at head_dim 128: with the promise of a quiescent cache few units run as two tiles on the keys kernel, others
on the wide one; parity of both sides of that line with the oracle (rows that do not divide evenly, both masks, the block
in the cache), and of the wide kernel's merge at cluster sizes that share its columns out unevenly.  Batches of more than 32
sequences, whose order by length is searched for bit by bit."""
import pytest
import torch

import oracle
from paper_2605_12825_b200 import workloads as W
from _gpu_util import assert_close, binding, captured_launches, oracle_attend, small_workload

pytestmark = pytest.mark.gpu


def inputs(shape, lens, hint):
    Hq, Hkv, K = shape
    wl = small_workload(len(lens), K, Hq, Hkv, 128, hint, hint, std=0.5, name=f"rows128_{Hq}_{Hkv}_{K}")
    t = W.attention_inputs(wl)
    t["cache_len"][:] = torch.tensor(lens, dtype=torch.int32)
    for b, p in enumerate(lens):
        t["k_cache"][b, :, p:] = float("nan")
        t["v_cache"][b, :, p:] = float("nan")
    return t


def run(t, shape, hint, flags, view=oracle.VIEW_AR, grids=None):
    b = binding()
    Hq, Hkv, K = shape
    x = "ar" if view == oracle.VIEW_AR else "diff"
    g = {k: v.cuda() for k, v in t.items()}
    layer = b.make_layer(g["k_cache"], g["v_cache"], g["cache_len"], Hq, K, hint, 0.0, flags)
    ws = b.new_workspace(b.orthrus_attend_workspace_bytes(layer))
    out = torch.full_like(g["q_" + x], float("nan"))
    f = b.orthrus_ar_verify_attend if view == oracle.VIEW_AR else b.orthrus_diffusion_block_attend
    blk = [None, None] if flags & b.LAYER_BLOCK_IN_CACHE else [g[f"k_{x}_blk"], g[f"v_{x}_blk"]]
    (name, _), = captured_launches(lambda: f(layer, g["q_" + x], *blk, out, ws), grids)
    f(layer, g["q_" + x], *blk, out, ws)
    assert b.orthrus_read_status(ws) == 0
    return out.cpu(), "keys" if "attend_keys_kernel" in name else "wide" if "attend_tc_kernel" in name else name


# 65, 77, 119 and 128 rows; 129 are three tiles of the wide kernel's side
@pytest.mark.parametrize("view", [oracle.VIEW_DIFFUSION, oracle.VIEW_AR])
@pytest.mark.parametrize("shape,few", [((5, 1, 13), "keys"), ((14, 2, 11), "keys"), ((7, 1, 17), "keys"), ((8, 2, 32), "keys"), ((3, 1, 43), "wide")])
def test_both_sides_of_the_promise(view, shape, few):
    b = binding()
    for lens in ([0, 1], [63, 500], [1024, 130]):
        t = inputs(shape, lens, 1024)
        ref = oracle_attend(view, t)
        for flags, kernel in ((b.LAYER_CACHE_QUIESCENT, few), (0, "wide")):
            got, name = run(t, shape, 1024, flags, view)
            assert name == kernel
            assert_close(got, ref, torch.bfloat16, f"{shape} {lens} {kernel}")


def test_block_in_the_cache():
    b = binding()
    shape, lens = (14, 2, 11), [190, 1000]
    t = inputs(shape, lens, 1024)
    ref = oracle_attend(oracle.VIEW_AR, t)
    for i, p in enumerate(lens):
        t["k_cache"][i, :, p:p + 11] = t["k_ar_blk"][i].transpose(0, 1)
        t["v_cache"][i, :, p:p + 11] = t["v_ar_blk"][i].transpose(0, 1)
    got, name = run(t, shape, 1024, b.LAYER_CACHE_QUIESCENT | b.LAYER_BLOCK_IN_CACHE)
    assert name == "keys"
    assert_close(got, ref, torch.bfloat16, "in cache")


def test_which_side_many_units_and_long_prefixes_are_on():
    b = binding()
    z = lambda *s: torch.zeros(s, dtype=torch.bfloat16, device="cuda")
    for B, Hkv, hint, kernel in ((2, 4, 8192, "keys"), (2, 4, 8193, "wide"), (9, 1, 1000, "wide")):
        kc, ln = z(B, Hkv, hint + 32, 128), torch.zeros(B, dtype=torch.int32, device="cuda")
        layer = b.make_layer(kc, kc, ln, 4 * Hkv, 32, hint, 0.0, b.LAYER_CACHE_QUIESCENT)
        ws = b.new_workspace(b.orthrus_attend_workspace_bytes(layer))
        q, kb = z(B, 32, 4 * Hkv, 128), z(B, 32, Hkv, 128)
        (name, _), = captured_launches(lambda: b.orthrus_ar_verify_attend(layer, q, kb, kb, torch.empty_like(q), ws))
        assert ("attend_keys_kernel" if kernel == "keys" else "attend_tc_kernel") in name


def test_few_units_of_33_to_64_rows_without_the_promise():
    """Two tiles for each of sixteen CTAs are the line: bound and block together in 62 halves of 64 keys and one of the block's."""
    b = binding()
    z = lambda *s: torch.zeros(s, dtype=torch.bfloat16, device="cuda")
    for B, Hkv, K, hint, flags, kernel in ((2, 4, 16, 512, 0, "wide"), (2, 4, 16, 513, 0, "keys"), (2, 4, 16, 4016, 0, "keys"),
                                           (2, 4, 16, 4017, 0, "wide"), (9, 1, 9, 4000, 0, "keys"), (10, 1, 9, 2000, 0, "wide"),
                                           (2, 4, 16, 4096, b.LAYER_CACHE_QUIESCENT, "keys"), (3, 8, 16, 1023, b.LAYER_CACHE_QUIESCENT, "wide"),
                                           (3, 8, 16, 1024, b.LAYER_CACHE_QUIESCENT, "keys"), (65, 1, 16, 2000, b.LAYER_CACHE_QUIESCENT, "wide")):
        kc, ln = z(B, Hkv, hint + K, 128), torch.zeros(B, dtype=torch.int32, device="cuda")
        layer = b.make_layer(kc, kc, ln, 4 * Hkv, K, hint, 0.0, flags)
        ws = b.new_workspace(b.orthrus_attend_workspace_bytes(layer))
        q, kb = z(B, K, 4 * Hkv, 128), z(B, K, Hkv, 128)
        (name, _), = captured_launches(lambda: b.orthrus_ar_verify_attend(layer, q, kb, kb, torch.empty_like(q), ws))
        assert ("attend_keys_kernel" if kernel == "keys" else "attend_tc_kernel") in name, (B, Hkv, K, hint, flags)


@pytest.mark.parametrize("splits", [3, 6, 7, 9, 10, 11, 12, 14, 16])
@pytest.mark.parametrize("peak", [1.0, 40.0])
def test_uneven_clusters_of_the_wide_kernel(splits, peak, monkeypatch):
    monkeypatch.setenv("ORTHRUS_SPLITS", str(splits))
    shape, lens = (8, 2, 24), [1000, 70]
    t = inputs(shape, lens, 1024)
    t["q_ar"] *= peak                          # 40: scores of hundreds, far from the first reference on either side
    got, name = run(t, shape, 1024, 0)
    assert name == "wide"
    assert_close(got, oracle_attend(oracle.VIEW_AR, t), torch.bfloat16, f"splits={splits} peak={peak}")


@pytest.mark.parametrize("K", [24, 4])
@pytest.mark.parametrize("B,Hkv", [(33, 16), (70, 8), (97, 8), (128, 4)])
@pytest.mark.parametrize("lens", ["some equal", "all equal"])
def test_batches_in_the_order_of_their_length(K, B, Hkv, lens):
    """More clusters than fit at once on either kernel (two CTAs to an SM), so that they are handed out by length: entries that are there
    for some of a lane's four registers, all lengths alike, the largest an exact power of two."""
    g = torch.Generator().manual_seed(B)
    lens = [256] + [int(x) for x in torch.randint(0, 12, (B - 1,), generator=g) * 20] if lens == "some equal" else [256] * B
    shape = (4 * Hkv, Hkv, K)
    t = inputs(shape, lens, 256)
    grids = []
    got, _ = run(t, shape, 256, 0, grids=grids)
    x, y, z = grids[0]
    assert x * y * z > 2 * torch.cuda.get_device_properties(0).multi_processor_count
    assert_close(got, oracle_attend(oracle.VIEW_AR, t), torch.bfloat16, f"{shape} {B}")
