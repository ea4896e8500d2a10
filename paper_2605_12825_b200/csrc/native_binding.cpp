// Argument marshalling of the hot calls in native code.  A decoding loop makes dozens of these calls
// per cycle, each a kernel of a few microseconds: through ctypes a call cost the host 8 us (3 us of
// them to ask torch for the current stream, the rest pointer conversions), more than most of the
// kernels take.  Here a call costs what its launch costs plus about a third of a microsecond.
//
// Every function takes the arguments of the Python function of the same name in binding.py (tensors
// or None, the layer descriptor, scalars, and last the stream or None for the current one), hands
// the pointers to the C entry point and calls the registered raiser when that reports an error.
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>
#include <vector>
#include "orthrus.h"

namespace {

PyObject *g_raise = nullptr;      // binding._raise(code, name)

struct Failed {};                 // a Python exception is set

const at::Tensor *as_tensor(PyObject *o) { return THPVariable_Check(o) ? &THPVariable_Unpack(o) : nullptr; }

void *ptr(PyObject *o)
{
    if (o == Py_None) return nullptr;
    if (const at::Tensor *t = as_tensor(o)) return t->data_ptr();
    PyObject *r = PyObject_CallMethod(o, "data_ptr", nullptr);
    if (!r) throw Failed();
    void *p = PyLong_AsVoidPtr(r);
    Py_DECREF(r);
    if (!p && PyErr_Occurred()) throw Failed();
    return p;
}

size_t count(PyObject *o)         // elements; 0 for None
{
    if (o == Py_None) return 0;
    if (const at::Tensor *t = as_tensor(o)) return (size_t)t->numel();
    PyObject *r = PyObject_CallMethod(o, "numel", nullptr);
    if (!r) throw Failed();
    const size_t n = PyLong_AsSize_t(r);
    Py_DECREF(r);
    if (n == (size_t)-1 && PyErr_Occurred()) throw Failed();
    return n;
}

const at::Tensor &need_tensor(PyObject *o, int dims)
{
    const at::Tensor *t = as_tensor(o);
    if (!t) { PyErr_SetString(PyExc_TypeError, "expected a torch tensor"); throw Failed(); }
    if (t->dim() != dims) {
        PyErr_Format(PyExc_ValueError, "expected a tensor of %d dimensions, got %d", dims, (int)t->dim());
        throw Failed();
    }
    return *t;
}

int32_t dtype_of(const at::Tensor &t)
{
    if (t.scalar_type() == at::kBFloat16) return ORTHRUS_BF16;
    if (t.scalar_type() == at::kFloat) return ORTHRUS_FP32;
    PyErr_Format(PyExc_TypeError, "unsupported dtype %s", c10::toString(t.scalar_type()));
    throw Failed();
}

void *stream_of(PyObject *o)
{
    if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
    PyObject *r = PyObject_GetAttrString(o, "cuda_stream");
    if (!r) throw Failed();
    void *p = PyLong_AsVoidPtr(r);
    Py_DECREF(r);
    if (!p && PyErr_Occurred()) throw Failed();
    return p;
}

// the orthrus_layer_t behind a ctypes structure (a copy: 88 bytes)
orthrus_layer_t layer_of(PyObject *o)
{
    Py_buffer view;
    if (PyObject_GetBuffer(o, &view, PyBUF_SIMPLE) != 0) throw Failed();
    if (view.len != (Py_ssize_t)sizeof(orthrus_layer_t)) {
        PyBuffer_Release(&view);
        PyErr_SetString(PyExc_TypeError, "expected a Layer");
        throw Failed();
    }
    const orthrus_layer_t L = *static_cast<const orthrus_layer_t *>(view.buf);
    PyBuffer_Release(&view);
    return L;
}

double real(PyObject *o)
{
    const double x = PyFloat_AsDouble(o);
    if (x == -1.0 && PyErr_Occurred()) throw Failed();
    return x;
}

bool truth(PyObject *o)
{
    const int t = PyObject_IsTrue(o);
    if (t < 0) throw Failed();
    return t != 0;
}

// runs `call` without the interpreter lock; None, or the raiser's exception
template <class Call> PyObject *finish(const char *name, Call call)
{
    int code;
    Py_BEGIN_ALLOW_THREADS
    code = (int)call();
    Py_END_ALLOW_THREADS
    if (code == ORTHRUS_OK) Py_RETURN_NONE;
    PyObject *r = PyObject_CallFunction(g_raise, "is", code, name);
    Py_XDECREF(r);
    if (!PyErr_Occurred()) PyErr_SetString(PyExc_RuntimeError, name);
    return nullptr;
}

template <class Body> PyObject *guarded(Py_ssize_t given, Py_ssize_t wanted, const char *name, Body body)
{
    if (given != wanted) return PyErr_Format(PyExc_TypeError, "%s takes %zd arguments, got %zd", name, wanted, given);
    try {
        return body();
    } catch (const Failed &) {
        return nullptr;
    } catch (const std::exception &e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
}

template <class Fn> PyObject *attend(PyObject *const *a, Py_ssize_t n, const char *name, Fn fn)
{   // layer, q, k_blk, v_blk, out, workspace, stream
    return guarded(n, 7, name, [&]() -> PyObject * {
        const orthrus_layer_t L = layer_of(a[0]);
        void *q = ptr(a[1]), *k = ptr(a[2]), *v = ptr(a[3]), *out = ptr(a[4]), *ws = ptr(a[5]), *st = stream_of(a[6]);
        const size_t wb = count(a[5]);
        return finish(name, [&] { return fn(&L, q, k, v, out, ws, wb, st); });
    });
}

PyObject *diffusion_block_attend(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    return attend(a, n, "orthrus_diffusion_block_attend", orthrus_diffusion_block_attend);
}
PyObject *ar_verify_attend(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    return attend(a, n, "orthrus_ar_verify_attend", orthrus_ar_verify_attend);
}

PyObject *multi_block_attend(PyObject *, PyObject *const *a, Py_ssize_t n)
{   // layer, anchors, q, k_blk, v_blk, out, workspace, stream
    const char *name = "orthrus_multi_block_attend";
    return guarded(n, 8, name, [&]() -> PyObject * {
        const orthrus_layer_t L = layer_of(a[0]);
        const at::Tensor &an = need_tensor(a[1], 2);
        const int32_t nb = (int32_t)an.size(1);
        const int32_t *ap = static_cast<const int32_t *>(an.data_ptr());
        void *q = ptr(a[2]), *k = ptr(a[3]), *v = ptr(a[4]), *out = ptr(a[5]), *ws = ptr(a[6]), *st = stream_of(a[7]);
        const size_t wb = count(a[6]);
        return finish(name, [&] { return orthrus_multi_block_attend(&L, nb, ap, q, k, v, out, ws, wb, st); });
    });
}

int32_t *iptr(PyObject *o) { return static_cast<int32_t *>(ptr(o)); }

PyObject *consensus_accept(PyObject *, PyObject *const *a, Py_ssize_t n)
{   // ar_logits, draft, n_commit, committed, ar_argmax, next_anchor, workspace, stream
    const char *name = "orthrus_consensus_accept";
    return guarded(n, 8, name, [&]() -> PyObject * {
        const at::Tensor &x = need_tensor(a[0], 3);
        const int32_t B = (int32_t)x.size(0), K = (int32_t)x.size(1), V = (int32_t)x.size(2), dt = dtype_of(x);
        void *lg = x.data_ptr(), *ws = ptr(a[6]), *st = stream_of(a[7]);
        int32_t *draft = iptr(a[1]), *nc = iptr(a[2]), *com = iptr(a[3]), *arg = iptr(a[4]), *nx = iptr(a[5]);
        const size_t wb = count(a[6]);
        return finish(name, [&] { return orthrus_consensus_accept(lg, dt, draft, B, K, V, nc, com, arg, nx, ws, wb, st); });
    });
}

PyObject *consensus_accept_static(PyObject *, PyObject *const *a, Py_ssize_t n)
{   // ar_logits, draft, n_commit, committed, ar_argmax, next_anchor, stream
    const char *name = "orthrus_consensus_accept_static";
    return guarded(n, 7, name, [&]() -> PyObject * {
        const at::Tensor &x = need_tensor(a[0], 3);
        const int32_t B = (int32_t)x.size(0), K = (int32_t)x.size(1), V = (int32_t)x.size(2), dt = dtype_of(x);
        void *lg = x.data_ptr(), *st = stream_of(a[6]);
        int32_t *draft = iptr(a[1]), *nc = iptr(a[2]), *com = iptr(a[3]), *arg = iptr(a[4]), *nx = iptr(a[5]);
        return finish(name, [&] { return orthrus_consensus_accept_static(lg, dt, draft, B, K, V, nc, com, arg, nx, st); });
    });
}

PyObject *consensus_sample(PyObject *, PyObject *const *a, Py_ssize_t n)
{   // ar_logits, diff_logits, draft, u_accept, u_resample, temperature, n_commit, committed, next_anchor, workspace, stream
    const char *name = "orthrus_consensus_sample";
    return guarded(n, 11, name, [&]() -> PyObject * {
        const at::Tensor &x = need_tensor(a[0], 3), &y = need_tensor(a[1], 3);
        if (x.sizes() != y.sizes() || x.scalar_type() != y.scalar_type()) {
            PyErr_SetString(PyExc_TypeError, "the two logit tensors must agree in shape and dtype");
            throw Failed();
        }
        const at::Tensor *u[2] = {as_tensor(a[3]), as_tensor(a[4])};
        if (!u[0] || !u[1] || u[0]->scalar_type() != at::kFloat || u[1]->scalar_type() != at::kFloat) {
            PyErr_SetString(PyExc_TypeError, "the uniforms must be float32");
            throw Failed();
        }
        const int32_t B = (int32_t)x.size(0), K = (int32_t)x.size(1), V = (int32_t)x.size(2), dt = dtype_of(x);
        void *la = x.data_ptr(), *ld = y.data_ptr(), *ws = ptr(a[9]), *st = stream_of(a[10]);
        const float *u1 = static_cast<const float *>(u[0]->data_ptr()), *u2 = static_cast<const float *>(u[1]->data_ptr());
        const float temp = (float)real(a[5]);
        int32_t *draft = iptr(a[2]), *nc = iptr(a[6]), *com = iptr(a[7]), *nx = iptr(a[8]);
        const size_t wb = count(a[9]);
        return finish(name, [&] {
            return orthrus_consensus_sample(la, ld, dt, draft, u1, u2, temp, B, K, V, nc, com, nx, ws, wb, st);
        });
    });
}

PyObject *lm_head_consensus(PyObject *, PyObject *const *a, Py_ssize_t n)
{   // hidden, lm_head, draft, n_commit, committed, ar_argmax, next_anchor, workspace, stream
    const char *name = "orthrus_lm_head_consensus";
    return guarded(n, 9, name, [&]() -> PyObject * {
        const at::Tensor &x = need_tensor(a[0], 3), &w = need_tensor(a[1], 2);
        const int32_t B = (int32_t)x.size(0), K = (int32_t)x.size(1), H = (int32_t)x.size(2), V = (int32_t)w.size(0);
        const int32_t dt = dtype_of(x);
        void *hp = x.data_ptr(), *wp = w.data_ptr(), *ws = ptr(a[7]), *st = stream_of(a[8]);
        int32_t *draft = iptr(a[2]), *nc = iptr(a[3]), *com = iptr(a[4]), *arg = iptr(a[5]), *nx = iptr(a[6]);
        const size_t wb = count(a[7]);
        return finish(name, [&] {
            return orthrus_lm_head_consensus(hp, wp, dt, H, draft, B, K, V, nc, com, arg, nx, ws, wb, st);
        });
    });
}

PyObject *kv_append(PyObject *, PyObject *const *a, Py_ssize_t n)
{   // layer, k_ar_blk, v_ar_blk, n_commit, update_len, workspace, stream
    const char *name = "orthrus_kv_append";
    return guarded(n, 7, name, [&]() -> PyObject * {
        const orthrus_layer_t L = layer_of(a[0]);
        void *k = ptr(a[1]), *v = ptr(a[2]), *ws = ptr(a[5]), *st = stream_of(a[6]);
        const int32_t *nc = iptr(a[3]);
        const int upd = truth(a[4]) ? 1 : 0;
        const size_t wb = count(a[5]);
        return finish(name, [&] { return orthrus_kv_append(&L, k, v, nc, upd, ws, wb, st); });
    });
}

PyObject *kv_append_layers(PyObject *, PyObject *const *a, Py_ssize_t n)
{   // layers, k_ar_blks, v_ar_blks, n_commit, update_len, workspace, stream
    const char *name = "orthrus_kv_append_layers";
    return guarded(n, 7, name, [&]() -> PyObject * {
        PyObject *seq[3] = {nullptr, nullptr, nullptr};
        struct Release { PyObject **s; ~Release() { for (int i = 0; i < 3; ++i) Py_XDECREF(s[i]); } } release{seq};
        for (int i = 0; i < 3; ++i) {
            seq[i] = PySequence_Fast(a[i], "expected a sequence");
            if (!seq[i]) throw Failed();
        }
        const Py_ssize_t m = PySequence_Fast_GET_SIZE(seq[0]);
        if (PySequence_Fast_GET_SIZE(seq[1]) != m || PySequence_Fast_GET_SIZE(seq[2]) != m) {
            PyErr_SetString(PyExc_ValueError, "one layer, one K and one V tensor per layer");
            throw Failed();
        }
        std::vector<orthrus_layer_t> L((size_t)m);
        std::vector<const void *> kp((size_t)m), vp((size_t)m);
        for (Py_ssize_t i = 0; i < m; ++i) {
            L[(size_t)i] = layer_of(PySequence_Fast_GET_ITEM(seq[0], i));
            kp[(size_t)i] = ptr(PySequence_Fast_GET_ITEM(seq[1], i));
            vp[(size_t)i] = ptr(PySequence_Fast_GET_ITEM(seq[2], i));
        }
        const int32_t *nc = iptr(a[3]);
        const int upd = truth(a[4]) ? 1 : 0;
        void *ws = ptr(a[5]), *st = stream_of(a[6]);
        const size_t wb = count(a[5]);
        return finish(name, [&] {
            return orthrus_kv_append_layers(L.data(), (int32_t)m, kp.data(), vp.data(), nc, upd, ws, wb, st);
        });
    });
}

PyObject *block_kv_write(PyObject *, PyObject *const *a, Py_ssize_t n)
{   // layer, k_blk, v_blk, workspace, stream
    const char *name = "orthrus_block_kv_write";
    return guarded(n, 5, name, [&]() -> PyObject * {
        const orthrus_layer_t L = layer_of(a[0]);
        void *k = ptr(a[1]), *v = ptr(a[2]), *ws = ptr(a[3]), *st = stream_of(a[4]);
        const size_t wb = count(a[3]);
        return finish(name, [&] { return orthrus_block_kv_write(&L, k, v, ws, wb, st); });
    });
}

PyObject *commit_len(PyObject *, PyObject *const *a, Py_ssize_t n)
{   // layer, n_commit, workspace, stream
    const char *name = "orthrus_commit_len";
    return guarded(n, 4, name, [&]() -> PyObject * {
        const orthrus_layer_t L = layer_of(a[0]);
        const int32_t *nc = iptr(a[1]);
        void *ws = ptr(a[2]), *st = stream_of(a[3]);
        const size_t wb = count(a[2]);
        return finish(name, [&] { return orthrus_commit_len(&L, nc, ws, wb, st); });
    });
}

PyObject *rope_block_kv_write(PyObject *, PyObject *const *a, Py_ssize_t n)
{   // layer, q, k_blk, v_blk, rope_theta, q_out, workspace, stream
    const char *name = "orthrus_rope_block_kv_write";
    return guarded(n, 8, name, [&]() -> PyObject * {
        const orthrus_layer_t L = layer_of(a[0]);
        void *q = ptr(a[1]), *k = ptr(a[2]), *v = ptr(a[3]), *qo = ptr(a[5]), *ws = ptr(a[6]), *st = stream_of(a[7]);
        const float theta = (float)real(a[4]);
        const size_t wb = count(a[6]);
        return finish(name, [&] { return orthrus_rope_block_kv_write(&L, q, k, v, theta, qo, ws, wb, st); });
    });
}

PyObject *set_raiser(PyObject *, PyObject *f)
{
    Py_XINCREF(f);
    Py_XSETREF(g_raise, f);
    Py_RETURN_NONE;
}

#define FAST(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(name)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {
    FAST(diffusion_block_attend), FAST(ar_verify_attend), FAST(multi_block_attend), FAST(consensus_accept),
    FAST(consensus_accept_static), FAST(consensus_sample), FAST(lm_head_consensus), FAST(kv_append),
    FAST(kv_append_layers), FAST(block_kv_write), FAST(commit_len), FAST(rope_block_kv_write),
    {"set_raiser", set_raiser, METH_O, nullptr}, {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native(void) { return PyModule_Create(&module); }
