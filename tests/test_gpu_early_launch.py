"""Which launches are programmatic dependents of the kernel before them: all of them by default, none of a call
whose layer has ORTHRUS_LAYER_NO_EARLY_LAUNCH, none of any call with ORTHRUS_NO_EARLY_LAUNCH=1.  Read off the edges
of captured graphs."""
import pytest
import torch

from _gpu_util import binding, captured_launches

pytestmark = pytest.mark.gpu
B, K, V, HQ, HKV, D, CAP, HID = 2, 4, 3000, 4, 2, 64, 256, 64


def calls(b, flags, dtype=torch.bfloat16):
    """name -> a call of every entry point that launches kernels; the first group takes a layer."""
    z = lambda *s, dt=dtype: torch.zeros(s, dtype=dt, device="cuda")
    i32 = lambda *s: z(*s, dt=torch.int32)
    keep = dict(k=z(B, HKV, CAP, D), v=z(B, HKV, CAP, D), len=i32(B), q=z(B, K, HQ, D), out=z(B, K, HQ, D),
                kb=z(B, K, HKV, D), vb=z(B, K, HKV, D), n=i32(B), com=i32(B, K), arg=i32(B, K), nxt=i32(B), dr=i32(B, K),
                lg=z(B, K, V), lg2=z(B, K, V), u=z(B, K, dt=torch.float32), hid=z(B, K, HID, dt=torch.bfloat16),
                head=z(V, HID, dt=torch.bfloat16), anc=i32(B, 2), mq=z(B, 2, K, HQ, D), mo=z(B, 2, K, HQ, D),
                mk=z(B, 2, K, HKV, D), mv=z(B, 2, K, HKV, D))
    t = keep
    layer = b.make_layer(t["k"], t["v"], t["len"], HQ, K, 200, 0.0, flags)
    ws = b.new_workspace(b.orthrus_multi_block_workspace_bytes(layer, 2))
    cws = b.new_workspace(max(b.orthrus_consensus_workspace_bytes(B, K, V), b.orthrus_consensus_sample_workspace_bytes(B, K, V),
                              b.orthrus_lm_head_consensus_workspace_bytes(B, K, V)))
    res = (t["n"], t["com"], t["arg"], t["nxt"])
    layered = {
        "diffusion": lambda: b.orthrus_diffusion_block_attend(layer, t["q"], t["kb"], t["vb"], t["out"], ws),
        "verify": lambda: b.orthrus_ar_verify_attend(layer, t["q"], t["kb"], t["vb"], t["out"], ws),
        "multi": lambda: b.orthrus_multi_block_attend(layer, t["anc"], t["mq"], t["mk"], t["mv"], t["mo"], ws),
        "append": lambda: b.orthrus_kv_append(layer, t["kb"], t["vb"], t["n"], True, ws),
        "append layers": lambda: b.orthrus_kv_append_layers([layer], [t["kb"]], [t["vb"]], t["n"], True, ws),
        "block write": lambda: b.orthrus_block_kv_write(layer, t["kb"], t["vb"], ws),
        "rotary write": lambda: b.orthrus_rope_block_kv_write(layer, t["q"], t["kb"], t["vb"], 1e4, t["out"], ws),
        "commit": lambda: b.orthrus_commit_len(layer, t["n"], ws)}
    others = {
        "consensus": lambda: b.orthrus_consensus_accept(t["lg"], t["dr"], *res, cws),
        "static": lambda: b.orthrus_consensus_accept_static(t["lg"], t["dr"], *res),
        "sample": lambda: b.orthrus_consensus_sample(t["lg"], t["lg2"], t["dr"], t["u"], t["u"], 1.0, t["n"], t["com"],
                                                     t["nxt"], cws),
        "lm head": lambda: b.orthrus_lm_head_consensus(t["hid"], t["head"], t["dr"], *res, cws)}
    return layered, others, (keep, ws, cws)


@pytest.mark.parametrize("path", ["auto", "mma", "simt"])
def test_early_launches(path, monkeypatch):
    b = binding()
    b.orthrus_set_path(path)
    try:
        for flags in (0, b.LAYER_NO_EARLY_LAUNCH):
            layered, others, _keep = calls(b, flags)
            for group, by_default in ((layered, flags == 0), (others, True)):
                for name, call in group.items():
                    call()                      # (first uses set function attributes, outside of the capture)
                    for env in (None, "1"):
                        monkeypatch.delenv("ORTHRUS_NO_EARLY_LAUNCH", raising=False)
                        if env:
                            monkeypatch.setenv("ORTHRUS_NO_EARLY_LAUNCH", env)
                        got = captured_launches(call)
                        assert got, name
                        assert [e for _, e in got] == [by_default and env is None] * len(got), (name, flags, env, got)
    finally:
        b.orthrus_set_path("auto")
