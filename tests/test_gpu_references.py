"""The tcgen05 kernels' softmax references, which start at zero and move only when a tile's probabilities are out of proportion
with them: all scores far above or far below zero, one key far above the rest in the first tile (as attention sinks are), in the
middle or at the end, references that rise tile by tile, or of some rows in one tile and of others in another, at the cluster sizes the library uses most and at uneven ones; the packed
multi-block form, whose rows see their first key at different tiles; visible scores that are not finite; the range of values
that the header states."""
import math

import pytest
import torch

import oracle
from paper_2605_12825_b200 import workloads as W
from _gpu_util import assert_close, binding, oracle_attend, small_workload

pytestmark = pytest.mark.gpu

# (query heads, KV heads, head_dim, block): 77 and 96 rows on the wide kernel, 63 rows on either, 4 and 128 rows on the keys kernel
SHAPES = [("wide", 14, 2, 128, 11), ("wide", 8, 2, 128, 24), ("wide", 14, 2, 128, 9), ("keys", 14, 2, 128, 9),
          ("keys", 8, 2, 128, 1), ("keys", 16, 2, 64, 16)]
SCORES = ["above", "below", "sink", "middle", "rising", "falling"]


def shift_scores(score, q, keys, lens):
    """Column 0 of the queries becomes `a`, that of the keys a per-key factor, so that score j is about 60 * factor_j more.  With
    rows of the block tensor behind those of the cache; the factor is a function of the position."""
    d = q.shape[-1]
    a = math.sqrt(60.0 * math.sqrt(d))
    q[..., 0] = a
    for k, start in keys:                                    # [B][Hkv][n][d] views, their first positions
        for b in range(k.shape[0]):
            pos = torch.arange(k.shape[2]) + start[b]
            f = {"above": torch.ones_like(pos, dtype=torch.float), "below": -torch.ones_like(pos, dtype=torch.float),
                 "sink": (pos == 0).float(), "middle": (pos == max(0, lens[b] // 2)).float(),
                 "rising": pos.float() / 100.0, "falling": -pos.float() / 100.0}[score]
            k[b, :, :, 0] = a * f


def inputs(shape, lens, hint, score):
    _, Hq, Hkv, d, K = shape
    wl = small_workload(len(lens), K, Hq, Hkv, d, hint, hint, std=0.5, name=f"refs_{Hq}_{Hkv}_{d}_{K}")
    t = W.attention_inputs(wl)
    t["cache_len"][:] = torch.tensor(lens, dtype=torch.int32)
    if score:
        shift_scores(score, t["q_ar"], [(t["k_cache"], [0] * len(lens)), (t["k_ar_blk"].transpose(1, 2), lens)], lens)
    for b, p in enumerate(lens):
        t["k_cache"][b, :, p:] = float("nan")
        t["v_cache"][b, :, p:] = float("nan")
    return t


def run(t, shape, hint, splits, monkeypatch):
    kernel, Hq, Hkv, d, K = shape
    b = binding()
    M = Hq // Hkv * K
    if d == 128 and M <= 64:
        monkeypatch.setenv("ORTHRUS_TC_SMALL_ROWS", "1" if kernel == "keys" else "0")
    if splits:
        monkeypatch.setenv("ORTHRUS_SPLITS", str(splits))
    g = {k: v.cuda() for k, v in t.items()}
    layer = b.make_layer(g["k_cache"], g["v_cache"], g["cache_len"], Hq, K, hint)
    ws = b.new_workspace(b.orthrus_attend_workspace_bytes(layer))
    out = torch.full_like(g["q_ar"], float("nan"))
    b.orthrus_ar_verify_attend(layer, g["q_ar"], g["k_ar_blk"], g["v_ar_blk"], out, ws)
    assert b.orthrus_read_status(ws) == 0 and b.orthrus_last_path() == "tcgen05"
    return out.cpu()


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("score", SCORES)
@pytest.mark.parametrize("splits", [None, 1, 2, 4, 8, 16, 5])
def test_references_that_move(shape, score, splits, monkeypatch):
    for lens in ([0, 1000], [64, 513]):
        t = inputs(shape, lens, 1024, score)
        got = run(t, shape, 1024, splits, monkeypatch)
        assert_close(got, oracle_attend(oracle.VIEW_AR, t), torch.bfloat16, f"{shape} {score} {lens} splits={splits}")


# references of some rows: further widths of the keys kernel's second operand (32 and 48 rows)
@pytest.mark.parametrize("shape", SHAPES + [("keys", 8, 2, 128, 8), ("keys", 8, 2, 64, 8), ("keys", 8, 2, 64, 12)])
@pytest.mark.parametrize("splits", [1, 2])
@pytest.mark.parametrize("first", [0.0, -60.0])
def test_references_of_some_rows(shape, splits, first, monkeypatch):
    """Every third row meets scores of +60 from key 256 on and of +120 from key 512 on, every other third of +60 from key 640 to
    767 only: with one CTA a unit those are the second and third 128-key tile of one softmax warpgroup of the keys kernel and the
    third of the other.  `first`: the scores of all rows over the first 256 keys, each warpgroup's first tile."""
    t = inputs(shape, [1000, 700], 1024, None)
    _, Hq, Hkv, d, K = shape
    a = math.sqrt(60.0 * math.sqrt(d))
    row = torch.arange(K)[:, None] * (Hq // Hkv) + torch.arange(Hq)[None, :] % (Hq // Hkv)       # a row's place in its query tile
    t["q_ar"][..., 0], t["q_ar"][..., 1], t["q_ar"][..., 2] = a * (row % 3 == 1), a * (row % 3 == 2), a
    for k in ("k_cache", "k_ar_blk"):
        t[k][..., :3] = 0
    k = t["k_cache"]
    k[:, :, :256, 2] = a * first / 60.0
    k[:, :, 256:512, 0], k[:, :, 512:, 0], k[:, :, 640:768, 1] = a, 2 * a, a
    for b, p in enumerate([1000, 700]):
        k[b, :, p:] = float("nan")
    got = run(t, shape, 1024, splits, monkeypatch)
    assert_close(got, oracle_attend(oracle.VIEW_AR, t), torch.bfloat16, f"{shape} splits={splits} first={first}")


# the packed form: blocks per sequence, width, heads (several blocks in a query tile of 128 rows)
@pytest.mark.parametrize("shape", [(12, 8, 8, 2), (5, 24, 4, 2), (7, 16, 2, 2)])
@pytest.mark.parametrize("score", SCORES + [None])
@pytest.mark.parametrize("splits", [None, 1, 3, 4])
@pytest.mark.parametrize("anchors", ["sorted", "random"])
def test_packed_blocks_with_references_that_move(shape, score, splits, anchors, monkeypatch):
    b = binding()
    NB, K, Hq, Hkv = shape
    S, d, L = 2, 128, 600
    g = torch.Generator().manual_seed(NB * K + Hq)
    mk = lambda *s, std=0.5: (torch.randn(*s, generator=g) * std).to(torch.bfloat16)
    q, kb, vb = mk(S, NB, K, Hq, d, std=0.5 if score else 20.0), mk(S, NB, K, Hkv, d), mk(S, NB, K, Hkv, d)
    kc, vc = mk(S, Hkv, 640, d), mk(S, Hkv, 640, d)
    at = torch.randint(0, L + 1, (S, NB), generator=g)
    at[0, 0], at[1, -1] = 0, L
    at = at.sort(dim=1).values if anchors == "sorted" else at
    lens = torch.full((S,), L, dtype=torch.int32)
    if score:
        shift_scores(score, q, [(kc, [0] * S)], [L] * S)
        for j in range(NB):                                  # a block's keys stand where its anchor is
            shift_scores(score, q[:, j], [(kb[:, j].transpose(1, 2), at[:, j].tolist())], [L] * S)
    kc[:, :, L:], vc[:, :, L:] = float("nan"), float("nan")
    at = at.to(torch.int32).contiguous()
    ref = oracle.multi_block_attend(q, kb, vb, kc, vc, lens, at)
    monkeypatch.setenv("ORTHRUS_MULTI_BLOCK_PACK", "1")
    if splits:
        monkeypatch.setenv("ORTHRUS_SPLITS", str(splits))
    dev = [x.cuda() for x in (kc, vc, lens, at, q, kb, vb)]
    layer = b.make_layer(dev[0], dev[1], dev[2], Hq, K, L)
    ws = b.new_workspace(b.orthrus_multi_block_workspace_bytes(layer, NB))
    out = torch.full_like(dev[4], float("nan"))
    b.orthrus_multi_block_attend(layer, dev[3], *dev[4:], out, ws)
    assert b.orthrus_read_status(ws) == 0 and b.orthrus_last_path() == "tcgen05"
    assert_close(out.cpu(), ref, torch.bfloat16, f"{shape} {score} {anchors} splits={splits}")


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("splits", [1, 2, 4, 9])
@pytest.mark.parametrize("value", ["inf", "nan"])
@pytest.mark.parametrize("at", [0, 300])
def test_scores_that_are_not_finite(shape, splits, value, at, monkeypatch):
    """A visible key whose scores are +inf for some query heads and -inf for others, or NaN: rows with +inf or NaN are not numbers
    (as in the definition, where inf - inf appears), rows with -inf leave the key out, and no row disturbs another."""
    t = inputs(shape, [400, 513], 1024, None)
    t["k_cache"][0, 0, at] = 0
    t["k_cache"][0, 0, at, 0] = float(value)
    t["q_ar"][..., 0] = 1.0
    t["q_ar"][:, ::2, :, 0] = -1.0                             # the odd rows of the block see +inf
    ref = oracle_attend(oracle.VIEW_AR, t)
    void = torch.isnan(ref)
    G = shape[1] // shape[2]
    assert void[0, 1::2, :G].all() and not void[1].any() and not void[0, :, G:].any()
    assert void[0, ::2, :G].all() == (value == "nan")
    got = run(t, shape, 1024, splits, monkeypatch)
    assert torch.equal(torch.isnan(got), void)
    assert_close(torch.where(void, torch.zeros_like(got), got), torch.where(void, torch.zeros_like(ref), ref), torch.bfloat16,
                 f"{shape} {value} splits={splits}")


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("splits", [None, 1, 2, 4])
@pytest.mark.parametrize("void", [64, 128, 256, 390])
def test_tiles_of_minus_infinity_ahead_of_low_scores(shape, splits, void, monkeypatch):
    """The first `void` keys have scores of -inf for every row, the others about -90: the first tiles tell nothing of where a
    row's scores are, and the reference moves in the first one that does."""
    t = inputs(shape, [400, 513], 1024, None)
    a = math.sqrt(90.0 * math.sqrt(shape[3]))
    t["q_ar"][..., 0] = a
    for k in ("k_cache", "k_ar_blk"):
        t[k][..., 0] = -a
    t["k_cache"][:, :, :void, 0] = -math.inf
    for b, p in enumerate([400, 513]):
        t["k_cache"][b, :, p:] = float("nan")
    got = run(t, shape, 1024, splits, monkeypatch)
    assert_close(got, oracle_attend(oracle.VIEW_AR, t), torch.bfloat16, f"{shape} void={void} splits={splits}")


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("splits", [1, 2, 8])
@pytest.mark.parametrize("sign,scale", [(1, 70), (-1, -48)])
def test_range_of_values(shape, splits, sign, scale, monkeypatch):
    """Scores at the ends of what an unmoved reference takes (27 and -41, that is, probabilities of 2^39 and 2^-59) with values of 2^70
    and 2^-48 and a thousand keys: the accumulators neither overflow nor lose a bit, so that the result is that of plain values
    times a power of two."""
    t = inputs(shape, [0, 1000], 1024, None)
    d = shape[3]
    a = math.sqrt((27.0 if sign > 0 else 40.5) * math.sqrt(d))
    t["q_ar"] *= 0.1
    t["q_ar"][..., 0] = a
    for k in ("k_cache", "k_ar_blk"):
        t[k] *= 0.1
        t[k][..., 0] = sign * a
    for b, p in enumerate([0, 1000]):
        t["k_cache"][b, :, p:] = float("nan")
    plain = run(t, shape, 1024, splits, monkeypatch)
    assert_close(plain, oracle_attend(oracle.VIEW_AR, t), torch.bfloat16, f"{shape} {sign}")
    for v in ("v_cache", "v_ar_blk"):
        t[v] *= 2.0 ** scale
    got = run(t, shape, 1024, splits, monkeypatch)
    assert torch.equal(got.float() * 2.0 ** -scale, plain.float())


@pytest.mark.parametrize("shape,lens", [((8, 2, 16), [1000, 800]), ((8, 2, 16), [4096, 70]), ((14, 2, 11), [1000, 513]), ((8, 2, 32), [2000, 64])])
def test_the_promise_changes_rounding_at_most(shape, lens):
    """With the promise of a quiescent cache these shapes run on the keys kernel, without it on either: the same probabilities, sums of
    them before or after rounding (2^-9 at most between them), each output rounded to bf16 (2^-9 each)."""
    b = binding()
    Hq, Hkv, K = shape
    t = inputs(("", Hq, Hkv, 128, K), lens, max(lens), None)
    g = {k: v.cuda() for k, v in t.items()}
    outs = []
    for flags in (0, b.LAYER_CACHE_QUIESCENT):
        layer = b.make_layer(g["k_cache"], g["v_cache"], g["cache_len"], Hq, K, max(lens), 0.0, flags)
        ws = b.new_workspace(b.orthrus_attend_workspace_bytes(layer))
        out = torch.empty_like(g["q_ar"])
        b.orthrus_ar_verify_attend(layer, g["q_ar"], g["k_ar_blk"], g["v_ar_blk"], out, ws)
        assert b.orthrus_read_status(ws) == 0
        outs.append(out.double().cpu())
    x, y = outs
    # (fp32 sums of up to 4096 products in another order: 4096 * 2^-24 of the sum of their magnitudes at most, which is below max|V| = 3)
    assert ((x - y).abs() <= 3 * 2.0 ** -9 * torch.maximum(x.abs(), y.abs()) + 3 * 4096 * 2.0 ** -24).all()
