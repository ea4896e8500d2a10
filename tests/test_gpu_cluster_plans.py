"""CTAs per unit of the keys kernel: clusters that are all resident at once whatever the number of units and the bound, and the
choices at the lines of the rule."""
import pytest
import torch

from _gpu_util import binding, captured_launches

pytestmark = pytest.mark.gpu

# clusters of 1 to 16 CTAs that a B200 of 148 SMs keeps resident, two CTAs to an SM and one
TWO = (296, 148, 93, 71, 56, 45, 37, 33, 30, 26, 21, 21, 17, 14, 14, 14)


def planned(units, rows, bound, monkeypatch, flags=0, d=128, kernel="attend_keys_kernel"):
    """(CTAs per unit, query tiles) of a call of `units` units of `rows` = 4 x block query rows."""
    b = binding()
    monkeypatch.setenv("ORTHRUS_TC_SMALL_ROWS", "1" if kernel == "attend_keys_kernel" else "0")
    K = rows // 4
    cache = torch.empty(units, 1, bound + K, d, dtype=torch.bfloat16, device="cuda")
    ln = torch.zeros(units, dtype=torch.int32, device="cuda")
    q, kb = (torch.empty(units, K, h, d, dtype=torch.bfloat16, device="cuda") for h in (4, 1))
    layer = b.make_layer(cache, cache, ln, 4, K, bound, 0.0, flags)
    ws = b.new_workspace(b.orthrus_attend_workspace_bytes(layer))
    grids = []
    (name, _), = captured_launches(lambda: b.orthrus_ar_verify_attend(layer, q, kb, kb, q, ws), grids)
    assert kernel in name
    return grids[0][0], grids[0][1] // (units if kernel == "attend_tc_kernel" else 1)


@pytest.fixture(autouse=True)
def a_full_b200():
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("the lines are drawn for 148 SMs")


@pytest.mark.parametrize("rows", [4, 32, 64])
def test_clusters_are_all_resident(rows, monkeypatch):
    for units in (2, 7, 13, 14, 15, 16, 18, 21, 22, 24, 27, 31, 34, 38, 46, 57, 72, 94):
        for bound in (64, 300, 1000, 4000, 8000):
            S, tiles = planned(units, rows, bound, monkeypatch)
            assert S == 1 or units * tiles <= TWO[S - 1], (units, rows, bound, S)


# 64 rows: units, bound, CTAs per unit
@pytest.mark.parametrize("units,bound,splits", [
    (1, 100, 8), (8, 100, 8), (16, 300, 4), (28, 200, 4), (36, 300, 3), (45, 300, 3), (8, 2000, 9), (8, 4000, 16), (15, 4000, 8),
    (22, 4000, 8), (24, 500, 5), (32, 1000, 8)])
def test_clusters_at_the_lines(units, bound, splits, monkeypatch):
    assert planned(units, 64, bound, monkeypatch) == (splits, 1)


# wide kernel: units, rows, bound, block in the cache, CTAs per unit
@pytest.mark.parametrize("units,rows,bound,in_cache,splits", [
    (6, 128, 8000, 0, 16), (7, 128, 8000, 0, 16), (8, 128, 2000, 0, 10), (8, 128, 16000, 0, 10), (8, 128, 20481, 0, 16), (9, 128, 4000, 0, 10),
    (8, 128, 4000, 1, 8), (8, 128, 8000, 1, 16), (8, 80, 4000, 0, 10), (8, 80, 5000, 0, 16), (8, 64, 3000, 0, 10), (8, 64, 3073, 0, 16),
    (4, 64, 3000, 0, 16)])
def test_clusters_of_sixteen_of_the_wide_kernel(units, rows, bound, in_cache, splits, monkeypatch):
    flags = binding().LAYER_BLOCK_IN_CACHE if in_cache else 0
    assert planned(units, rows, bound, monkeypatch, flags, kernel="attend_tc_kernel") == (splits, 1)


# with the promise of a quiescent cache: units, rows, bound, kernel
@pytest.mark.parametrize("units,rows,bound,kernel", [
    (8, 64, 64, "attend_tc_kernel"), (8, 64, 65, "attend_keys_kernel"), (8, 36, 64, "attend_tc_kernel"), (2, 128, 64, "attend_tc_kernel"),
    (2, 128, 65, "attend_keys_kernel"), (9, 64, 384, "attend_tc_kernel"), (9, 64, 385, "attend_keys_kernel"), (9, 60, 300, "attend_keys_kernel"),
    (23, 64, 1000, "attend_keys_kernel"), (24, 64, 1000, "attend_tc_kernel"), (49, 64, 1024, "attend_keys_kernel"), (50, 64, 1024, "attend_tc_kernel")])
def test_lines_with_the_promise(units, rows, bound, kernel):
    b = binding()
    K = rows // 4
    cache = torch.empty(units, 1, bound + K, 128, dtype=torch.bfloat16, device="cuda")
    ln = torch.zeros(units, dtype=torch.int32, device="cuda")
    q, kb = (torch.empty(units, K, h, 128, dtype=torch.bfloat16, device="cuda") for h in (4, 1))
    layer = b.make_layer(cache, cache, ln, 4, K, bound, 0.0, b.LAYER_CACHE_QUIESCENT)
    ws = b.new_workspace(b.orthrus_attend_workspace_bytes(layer))
    (name, _), = captured_launches(lambda: b.orthrus_ar_verify_attend(layer, q, kb, kb, q, ws))
    assert kernel in name
