"""33 to 64 query rows at head_dim 128, which two tcgen05 kernels can serve: both against the oracle at the same
inputs (rows that fill warps of 32 and rows that do not, every merge form, both masks, the block as a tensor and in the
cache, NaN behind the keys), and which of them the library picks at the edges of its rule."""
import pytest
import torch

import oracle
from paper_2605_12825_b200 import workloads as W
from _gpu_util import Guarded, assert_close, binding, captured_launches, oracle_attend, run_attend, small_workload

pytestmark = pytest.mark.gpu
VIEWS = [oracle.VIEW_DIFFUSION, oracle.VIEW_AR]
# (Hq, Hkv, K): 33, 36, 43, 49, 60, 63, 64 and 64 rows
SHAPES = [(3, 1, 11), (8, 2, 9), (1, 1, 43), (14, 2, 7), (8, 2, 15), (7, 1, 9), (8, 2, 16), (1, 1, 64)]
KERNELS = {"keys": "1", "wide": "0"}
NAN = float("nan")


def inputs(shape, lens, hint):
    Hq, Hkv, K = shape
    wl = small_workload(len(lens), K, Hq, Hkv, 128, hint, hint, std=0.5, name=f"rows64_{Hq}_{Hkv}_{K}")
    t = W.attention_inputs(wl)
    t["cache_len"][:] = torch.tensor(lens, dtype=torch.int32)
    for b, p in enumerate(lens):
        t["k_cache"][b, :, p:, :] = NAN
        t["v_cache"][b, :, p:, :] = NAN
    return wl, t


def kernel_of(layer, q, kb, vb, out, ws):
    (name, _), = captured_launches(lambda: binding().orthrus_ar_verify_attend(layer, q, kb, vb, out, ws))
    return "keys" if "attend_keys_kernel" in name else "wide" if "attend_tc_kernel" in name else name


@pytest.mark.parametrize("view", VIEWS)
@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("lens", [[0, 1], [64, 129], [700, 257], [1024, 1000]])
def test_both_kernels_at_every_cut(view, shape, lens, monkeypatch):
    wl, t = inputs(shape, lens, 1024)
    ref = oracle_attend(view, t)
    for kernel, knob in KERNELS.items():
        monkeypatch.setenv("ORTHRUS_TC_SMALL_ROWS", knob)
        for splits in (None, 1, 2, 3, 4, 5, 8, 16):
            got, status, used = run_attend(view, t, wl, max_len_hint=1024, splits=splits, flags=1 if splits == 8 else 0)
            assert used == "tcgen05" and status == 0
            assert_close(got, ref, torch.bfloat16, f"{kernel} {shape} lens={lens} splits={splits}")


@pytest.mark.parametrize("kernel", KERNELS)
@pytest.mark.parametrize("shape", [(8, 2, 9), (1, 1, 43), (8, 2, 16)])
@pytest.mark.parametrize("splits", [None, 2, 4, 16])
def test_block_in_the_cache(kernel, shape, splits, monkeypatch):
    b = binding()
    Hq, Hkv, K = shape
    lens = [190, 1000]
    wl, t = inputs(shape, lens, 1024)
    ref = oracle_attend(oracle.VIEW_AR, t)
    for i, p in enumerate(lens):
        t["k_cache"][i, :, p:p + K] = t["k_ar_blk"][i].transpose(0, 1)
        t["v_cache"][i, :, p:p + K] = t["v_ar_blk"][i].transpose(0, 1)
    monkeypatch.setenv("ORTHRUS_TC_SMALL_ROWS", KERNELS[kernel])
    if splits:
        monkeypatch.setenv("ORTHRUS_SPLITS", str(splits))
    k, v, ln = t["k_cache"].cuda(), t["v_cache"].cuda(), t["cache_len"].cuda()
    layer = b.make_layer(k, v, ln, Hq, K, 1024, 0.0, b.LAYER_BLOCK_IN_CACHE)
    ws = b.new_workspace(b.orthrus_attend_workspace_bytes(layer))
    out = Guarded(tuple(t["q_ar"].shape), torch.bfloat16)
    b.orthrus_ar_verify_attend(layer, t["q_ar"].cuda(), None, None, out.t, ws)
    assert b.orthrus_read_status(ws) == 0 and out.intact()
    assert_close(out.t.cpu(), ref, torch.bfloat16, f"{kernel} {shape}")


@pytest.mark.parametrize("K", [9, 16])
@pytest.mark.parametrize("B", [16, 24, 32])
def test_cuts_that_many_units_pick_by_themselves(B, K, monkeypatch):
    """64, 96 and 128 units: clusters of 4, 2 and 2, which merge through distributed shared memory on either kernel;
    lengths from nothing to the bound, so that CTAs without a tile exchange too."""
    lens = [int(x) for x in torch.linspace(0, 1400, B)]
    wl, t = inputs((16, 4, K), lens, 1400)
    ref = oracle_attend(oracle.VIEW_AR, t)
    for kernel, knob in KERNELS.items():
        monkeypatch.setenv("ORTHRUS_TC_SMALL_ROWS", knob)
        got, status, _ = run_attend(oracle.VIEW_AR, t, wl, max_len_hint=1400)
        assert status == 0
        assert_close(got, ref, torch.bfloat16, f"{kernel} B={B} K={K}")
    b = binding()
    z = lambda *s: torch.zeros(s, dtype=torch.bfloat16, device="cuda")
    kc, ln = z(B, 4, wl.capacity, 128), torch.zeros(B, dtype=torch.int32, device="cuda")
    monkeypatch.setenv("ORTHRUS_TC_SMALL_ROWS", "1")
    layer = b.make_layer(kc, kc, ln, 16, K, 1400)
    ws = b.new_workspace(b.orthrus_attend_workspace_bytes(layer))
    q, kb = z(B, K, 16, 128), z(B, K, 4, 128)
    (name, _), = captured_launches(lambda: b.orthrus_ar_verify_attend(layer, q, kb, kb, torch.empty_like(q), ws))
    assert "attend_keys_kernelILi128ELi64ELb1EE" in name, name          # (the exchanging instance)


# (units, rows, bound, kernel)
PICKS = [(8, 64, 100, "wide"), (8, 64, 300, "wide"), (8, 64, 512, "wide"), (8, 64, 4096, "wide"), (8, 64, 20000, "wide"),
         (32, 64, 500, "wide"), (48, 64, 3000, "wide"), (128, 64, 2000, "wide"), (256, 64, 300, "wide"), (8, 36, 4096, "wide"),
         # clusters of the wide kernel that are not all resident
         (33, 64, 1300, "wide"), (34, 64, 1300, "keys"), (37, 64, 1700, "keys"), (38, 64, 1700, "wide"),
         (160, 64, 960, "wide"), (160, 64, 961, "keys"), (296, 64, 1024, "wide"), (320, 64, 1024, "wide"),
         # half-empty grids
         (12, 64, 4096, "wide"), (12, 64, 4097, "keys"), (44, 64, 4097, "keys"), (46, 64, 4097, "wide"), (80, 64, 4500, "wide"),
         (12, 36, 2048, "wide"), (12, 36, 2049, "keys"), (42, 60, 2049, "keys"), (46, 36, 3000, "wide"),
         # clusters of eight that fill the grid
         (22, 64, 2000, "wide"), (23, 64, 2000, "keys"), (32, 64, 1536, "wide"), (32, 64, 1537, "keys"), (32, 64, 3072, "keys"),
         (32, 64, 3073, "wide"), (32, 36, 1536, "wide"), (32, 36, 3072, "keys")]


@pytest.mark.parametrize("units,rows,bound,kernel", PICKS)
def test_which_kernel_the_library_picks(units, rows, bound, kernel):
    b = binding()
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("the lines are drawn for 148 SMs")
    hkv = 4 if units % 4 == 0 else 2 if units % 2 == 0 else 1
    B, K, cap = units // hkv, rows // 4, bound + 16
    cache = torch.empty(B, hkv, cap, 128, dtype=torch.bfloat16, device="cuda")
    ln = torch.zeros(B, dtype=torch.int32, device="cuda")
    q, kb = (torch.empty(B, K, h * hkv, 128, dtype=torch.bfloat16, device="cuda") for h in (4, 1))
    layer = b.make_layer(cache, cache, ln, 4 * hkv, K, bound)
    ws = b.new_workspace(b.orthrus_attend_workspace_bytes(layer))
    assert kernel_of(layer, q, kb, kb, q, ws) == kernel
