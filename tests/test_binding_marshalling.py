"""The package imports and works whatever Python and torch it meets: without a native marshalling module for them, or
with one that does not load, the calls go through ctypes and behave alike."""
import os
import subprocess
import sys
import textwrap

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def child(code, **env):
    r = subprocess.run([sys.executable, "-c", textwrap.dedent(code)], cwd=ROOT, env=dict(os.environ, **env),
                       capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-3000:]
    return r.stdout


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2605_12825_b200 import build
    build.build()


@pytest.mark.parametrize("content", [None, b"", b"not a shared object"])
def test_import_without_a_native_module_that_loads(content, tmp_path):
    path = tmp_path / "_native.other.so"
    if content is not None:
        path.write_bytes(content)
    out = child(f"""
        import warnings
        from paper_2605_12825_b200 import build
        build.native_path = lambda: {str(path)!r}
        with warnings.catch_warnings(record=True) as w:
            warnings.simplefilter("always")
            from paper_2605_12825_b200 import binding as b
        assert any(issubclass(x.category, RuntimeWarning) and "ctypes" in str(x.message) for x in w)
        print(b._native.__name__, b.orthrus_version())
        """)
    assert out.split()[0].endswith("._marshal")


# every entry point with arguments that the host checks refuse before anything is launched: what is raised, with the
# status, must be the same through either module (a layer with head_dim 48; a null tensor; a short workspace; ...)
REFUSALS = """
    import ctypes, torch, warnings
    warnings.simplefilter("ignore")
    from paper_2605_12825_b200 import build
    if {fallback}:
        build.native_path = lambda: "/nonexistent"
    from paper_2605_12825_b200 import binding as b
    assert b._native.__name__.endswith("._marshal" if {fallback} else "._native")
    class S: cuda_stream = 0
    z = lambda *s, dt=torch.bfloat16: torch.zeros(s, dtype=dt)
    i = lambda *s: z(*s, dt=torch.int32)
    kc = z(1, 2, 64, 64)
    L = lambda **kw: b.Layer(*[dict(dict(batch=1, n_q_heads=4, n_kv_heads=2, head_dim=64, block=4, dtype=0, capacity=64,
        k_cache=kc.data_ptr(), v_cache=kc.data_ptr(), cache_len=kc.data_ptr(), max_len_hint=32, softmax_scale=0.0, flags=0), **kw)[f[0]]
        for f in b.Layer._fields_])
    q, kb, ws, n, com = z(1, 4, 4, 64), z(1, 4, 2, 64), z(8, dt=torch.uint8), i(1), i(1, 4)
    bad, lg, u, hid, head = L(head_dim=48), z(1, 4, 100), z(1, 4, dt=torch.float32), z(1, 4, 8), z(100, 8)
    calls = [
        lambda: b.orthrus_diffusion_block_attend(bad, q, kb, kb, q, ws, S),
        lambda: b.orthrus_diffusion_block_attend(L(), q, None, kb, q, ws, S),
        lambda: b.orthrus_ar_verify_attend(L(block=65), q, kb, kb, q, ws, S),
        lambda: b.orthrus_ar_verify_attend(L(max_len_hint=63), q, kb, kb, q, ws, S),
        lambda: b.orthrus_multi_block_attend(bad, com, q, kb, kb, q, ws, S),
        lambda: b.orthrus_multi_block_attend(L(), n, q, kb, kb, q, ws, S),
        lambda: b.orthrus_consensus_accept(lg, com, n, com, com, n, ws, S),
        lambda: b.orthrus_consensus_accept(lg[0], com, n, com, com, n, ws, S),
        lambda: b.orthrus_consensus_accept(lg.half(), com, n, com, com, n, ws, S),
        lambda: b.orthrus_consensus_accept(lg, None, n, com, com, n, ws, S),
        lambda: b.orthrus_consensus_accept_static(z(1, 9000, 64), com, n, com, com, n, S),
        lambda: b.orthrus_consensus_accept_static(lg, com, n, com, com, None, S),
        lambda: b.orthrus_consensus_sample(lg, lg, com, u, u, 0.0, n, com, n, ws, S),
        lambda: b.orthrus_consensus_sample(lg, lg, com, u, u, 1.0, n, com, n, ws, S),
        lambda: b.orthrus_consensus_sample(lg, lg.float(), com, u, u, 1.0, n, com, n, ws, S),
        lambda: b.orthrus_consensus_sample(lg, lg, com, u, u.double(), 1.0, n, com, n, ws, S),
        lambda: b.orthrus_lm_head_consensus(hid.float(), head, com, n, com, com, n, ws, S),
        lambda: b.orthrus_lm_head_consensus(hid, head, com, n, com, com, n, ws, S),
        lambda: b.orthrus_lm_head_consensus(hid, head[0], com, n, com, com, n, ws, S),
        lambda: b.orthrus_kv_append(bad, kb, kb, n, True, None, S),
        lambda: b.orthrus_kv_append(L(), kb, kb, n, True, ws, S),
        lambda: b.orthrus_kv_append(L(), kb, None, n, False, None, S),
        lambda: b.orthrus_kv_append_layers([], [], [], n, True, None, S),
        lambda: b.orthrus_kv_append_layers([bad, bad], [kb, kb], [kb, kb], n, True, None, S),
        lambda: b.orthrus_kv_append_layers([L(), L(batch=2)], (kb, kb), (kb, kb), n, True, None, S),
        lambda: b.orthrus_kv_append_layers([L()], [kb, kb], [kb], n, True, None, S),
        lambda: b.orthrus_block_kv_write(bad, kb, kb, None, S),
        lambda: b.orthrus_block_kv_write(L(), kb, kb, ws, S),
        lambda: b.orthrus_commit_len(bad, n, None, S),
        lambda: b.orthrus_commit_len(L(), None, None, S),
        lambda: b.orthrus_rope_block_kv_write(bad, q, kb, kb, 1e4, q, None, S),
        lambda: b.orthrus_rope_block_kv_write(L(), q, kb, kb, 0.0, q, None, S),
        lambda: b.orthrus_rope_block_kv_write(L(), q, kb, kb, 1e4, None, None, S),
    ]
    n0 = b.orthrus_launch_count()
    for c in calls:
        try:
            c()
            print("accepted")
        except Exception as e:
            print(type(e).__name__, getattr(e, "code", None), str(e) if hasattr(e, "code") else "")
    assert b.orthrus_launch_count() == n0
"""


def test_both_modules_refuse_alike():
    native, ctypes_ = (child(REFUSALS.format(fallback=f)).splitlines() for f in (False, True))
    assert len(native) == 33 and "accepted" not in native
    assert native == ctypes_


@pytest.mark.gpu
def test_parity_through_ctypes():
    """One test file per group of calls, run on the fallback."""
    out = child("""
        import sys, warnings
        import pytest
        from paper_2605_12825_b200 import build
        build.native_path = lambda: "/nonexistent"
        warnings.simplefilter("ignore")
        from paper_2605_12825_b200 import binding as b
        assert b._native.__name__.endswith("._marshal")
        t = "tests/test_gpu_"
        sys.exit(pytest.main([t + "early_launch.py", t + "consensus_append.py", t + "truncate_commit.py", t + "multi_block.py",
                              t + "consensus_sample.py", "tests/test_zz_no_alloc.py", "-x", "-q", "-p", "no:cacheprovider",
                              "-k", "not ragged_serving and not child"]))
        """)
    assert " passed" in out
