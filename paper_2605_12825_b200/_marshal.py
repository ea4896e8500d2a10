"""The argument marshalling of csrc/native_binding.cpp through ctypes: the same functions with the same arguments,
for an interpreter or a torch that the native module was not compiled for.  A call costs the host about 8 us
here and a third of one there (plus the launch either way)."""
import ctypes

import torch

_lib = _raise = None


def bind(lib, raiser):
    """`lib`: liborthrus.so with its argument types declared; `raiser(code, name)` raises for an error code."""
    global _lib, _raise
    _lib, _raise = lib, raiser


def _ptr(t):
    return None if t is None else t.data_ptr()


def _count(t):
    return 0 if t is None else t.numel()


def _stream(stream):
    return (torch.cuda.current_stream() if stream is None else stream).cuda_stream


def _dims(t, n):
    if not isinstance(t, torch.Tensor):
        raise TypeError("expected a torch tensor")
    if t.dim() != n:
        raise ValueError(f"expected a tensor of {n} dimensions, got {t.dim()}")
    return t.shape


def _dtype(t):
    if t.dtype not in (torch.bfloat16, torch.float32):
        raise TypeError(f"unsupported dtype {t.dtype}")
    return 0 if t.dtype == torch.bfloat16 else 1


def _call(name, *args):
    code = getattr(_lib, name)(*args)
    if code != 0:
        _raise(code, name)


def _attend(name, layer, q, k, v, out, workspace, stream):
    _call(name, ctypes.byref(layer), _ptr(q), _ptr(k), _ptr(v), _ptr(out), _ptr(workspace), _count(workspace), _stream(stream))


def diffusion_block_attend(*args):
    _attend("orthrus_diffusion_block_attend", *args)


def ar_verify_attend(*args):
    _attend("orthrus_ar_verify_attend", *args)


def multi_block_attend(layer, anchors, q, k, v, out, workspace, stream):
    n_blocks = _dims(anchors, 2)[1]
    _call("orthrus_multi_block_attend", ctypes.byref(layer), n_blocks, _ptr(anchors), _ptr(q), _ptr(k), _ptr(v), _ptr(out),
          _ptr(workspace), _count(workspace), _stream(stream))


def consensus_accept(logits, draft, n_commit, committed, ar_argmax, next_anchor, workspace, stream):
    B, K, V = _dims(logits, 3)
    _call("orthrus_consensus_accept", _ptr(logits), _dtype(logits), _ptr(draft), B, K, V, _ptr(n_commit), _ptr(committed),
          _ptr(ar_argmax), _ptr(next_anchor), _ptr(workspace), _count(workspace), _stream(stream))


def consensus_accept_static(logits, draft, n_commit, committed, ar_argmax, next_anchor, stream):
    B, K, V = _dims(logits, 3)
    _call("orthrus_consensus_accept_static", _ptr(logits), _dtype(logits), _ptr(draft), B, K, V, _ptr(n_commit),
          _ptr(committed), _ptr(ar_argmax), _ptr(next_anchor), _stream(stream))


def consensus_sample(ar, diff, draft, u_accept, u_resample, temperature, n_commit, committed, next_anchor, workspace, stream):
    B, K, V = _dims(ar, 3)
    if _dims(diff, 3) != ar.shape or diff.dtype != ar.dtype:
        raise TypeError("the two logit tensors must agree in shape and dtype")
    if u_accept.dtype != torch.float32 or u_resample.dtype != torch.float32:
        raise TypeError("the uniforms must be float32")
    _call("orthrus_consensus_sample", _ptr(ar), _ptr(diff), _dtype(ar), _ptr(draft), _ptr(u_accept), _ptr(u_resample),
          float(temperature), B, K, V, _ptr(n_commit), _ptr(committed), _ptr(next_anchor), _ptr(workspace), _count(workspace),
          _stream(stream))


def lm_head_consensus(hidden, lm_head, draft, n_commit, committed, ar_argmax, next_anchor, workspace, stream):
    (B, K, H), V = _dims(hidden, 3), _dims(lm_head, 2)[0]
    _call("orthrus_lm_head_consensus", _ptr(hidden), _ptr(lm_head), _dtype(hidden), H, _ptr(draft), B, K, V, _ptr(n_commit),
          _ptr(committed), _ptr(ar_argmax), _ptr(next_anchor), _ptr(workspace), _count(workspace), _stream(stream))


def kv_append(layer, k, v, n_commit, update_len, workspace, stream):
    _call("orthrus_kv_append", ctypes.byref(layer), _ptr(k), _ptr(v), _ptr(n_commit), 1 if update_len else 0, _ptr(workspace),
          _count(workspace), _stream(stream))


def kv_append_layers(layers, ks, vs, n_commit, update_len, workspace, stream):
    layers, ks, vs = list(layers), list(ks), list(vs)
    n = len(layers)
    if len(ks) != n or len(vs) != n:
        raise ValueError("one layer, one K and one V tensor per layer")
    arr = (type(layers[0]) * n)(*layers) if n else None
    kp, vp = ((ctypes.c_void_p * n)(*[t.data_ptr() for t in x]) for x in (ks, vs))
    _call("orthrus_kv_append_layers", arr, n, kp, vp, _ptr(n_commit), 1 if update_len else 0, _ptr(workspace),
          _count(workspace), _stream(stream))


def block_kv_write(layer, k, v, workspace, stream):
    _call("orthrus_block_kv_write", ctypes.byref(layer), _ptr(k), _ptr(v), _ptr(workspace), _count(workspace), _stream(stream))


def commit_len(layer, n_commit, workspace, stream):
    _call("orthrus_commit_len", ctypes.byref(layer), _ptr(n_commit), _ptr(workspace), _count(workspace), _stream(stream))


def rope_block_kv_write(layer, q, k, v, rope_theta, q_out, workspace, stream):
    _call("orthrus_rope_block_kv_write", ctypes.byref(layer), _ptr(q), _ptr(k), _ptr(v), float(rope_theta), _ptr(q_out),
          _ptr(workspace), _count(workspace), _stream(stream))
