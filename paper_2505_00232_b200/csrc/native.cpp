// The calls of the Python binding whose host work a small layer would otherwise wait for: the arguments of a call are checked, its outputs
// allocated and the C entry point called in native code.  Bound: a layer of a few million weights takes the GPU 3 us, and the launch itself
// the host 2.3; QLinear.forward at one token took 6.7 us through Python and ctypes and takes 3.5 to 4.0 through here, by machine (other calls:
// binding.py).
//
// Every function takes the common form of its call (plain tensors of the documented types, shapes and layout) and returns None for anything
// else, whatever is wrong with it; the caller in binding.py then does the call in Python, with Python's own errors.  A status
// other than QL_OK is raised by the binding's own check.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/PythonTorchFunctionTLS.h>
#include <ATen/cuda/EmptyTensor.h>
#include <c10/core/impl/LocalDispatchKeySet.h>
#include <c10/cuda/CUDAFunctions.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <climits>

#include "../../include/qlinear.h"

namespace {

// Entry points of libqlinear.so, which the binding has loaded (init).
struct Api {
    decltype(&qlinear_forward) forward;
    decltype(&qlinear_forward_a8) forward_a8;
    decltype(&qlinear_forward_group) forward_group;
    decltype(&qlinear_forward_gated) forward_gated;
    decltype(&qlinear_residual_rmsnorm) residual_rmsnorm;
    decltype(&qlinear_rope_qkv) rope_qkv;
    decltype(&qlinear_embed) embed;
    decltype(&qlinear_kv_append_heads) kv_append_heads;
    decltype(&qlinear_kv_scores_heads) kv_scores_heads;
    decltype(&qlinear_kv_output_heads) kv_output_heads;
    decltype(&qlinear_kv_output) kv_output;
    decltype(&qlinear_kv_output_uses_tmp) kv_output_uses_tmp;
} api;
PyObject* check_status = nullptr;                                        // binding._check(status, where)

using c10::DispatchKey;

// Tracing, modes of both kinds, functionalisation and the function transforms see every operator, allocations among them: such calls are Python's.
bool modes_are_on()
{
    const auto on = c10::impl::tls_local_dispatch_key_set().included_;
    return on.has_any(c10::DispatchKeySet({DispatchKey::Python, DispatchKey::PythonTLSSnapshot, DispatchKey::FuncTorchDynamicLayerFrontMode, DispatchKey::FuncTorchDynamicLayerBackMode,
                                           DispatchKey::FuncTorchVmapMode, DispatchKey::Functionalize, DispatchKey::Tracer})) ||
           at::impl::PythonTorchFunctionTLS::stack_len() > 0;
}

// The tensor of a Python object, if it is a dense contiguous CUDA tensor of the type and no subclass or wrapper of one.
const at::Tensor* plain(PyObject* o, at::ScalarType type)
{
    if (!THPVariable_CheckExact(o)) return nullptr;
    const at::Tensor& t = THPVariable_Unpack(o);
    if (!t.defined() || !t.is_cuda() || t.scalar_type() != type || t.layout() != at::kStrided || !t.is_contiguous()) return nullptr;
    if (t.key_set().has_any(c10::DispatchKeySet({DispatchKey::Python, DispatchKey::FuncTorchBatched, DispatchKey::FuncTorchGradWrapper, DispatchKey::Functionalize, DispatchKey::Conjugate,
                                                 DispatchKey::Negative, DispatchKey::ZeroTensor}))) return nullptr;
    return &t;
}
bool is_matrix(const at::Tensor* t, int64_t rows, int64_t cols) { return t && t->dim() == 2 && t->size(0) == rows && t->size(1) == cols; }

at::Tensor half_like(const at::Tensor& x, at::IntArrayRef size) { return at::detail::empty_cuda(size, at::kHalf, x.device(), std::nullopt); }

// None: the current stream of the current device; otherwise a raw stream handle.
void* stream_of(PyObject* o) { return o == Py_None ? static_cast<void*>(c10::cuda::getCurrentCUDAStream(c10::cuda::current_device()).stream()) : PyLong_AsVoidPtr(o); }

// Runs `call`, which allocates its outputs (that may go to the driver) and calls the library, without the interpreter lock; false with the
// binding's exception set if its status is not QL_OK.
struct Unlocked {
    PyThreadState* state = PyEval_SaveThread();
    ~Unlocked() { PyEval_RestoreThread(state); }                         // (past a C++ exception as well)
};
template <typename F>
bool done(F call, const char* where)
{
    ql_status s;
    {
        Unlocked unlocked;
        s = call();
    }
    if (s == QL_OK) return true;
    PyObject* r = PyObject_CallFunction(check_status, "is", (int)s, where);
    if (r) { Py_DECREF(r); PyErr_SetString(PyExc_RuntimeError, where); }  // (the check raises)
    return false;
}

// A C++ exception (out of memory, a CUDA error of the allocator) becomes the Python exception that torch would raise.
template <typename F>
PyObject* guarded(F f)
{
    HANDLE_TH_ERRORS
    if (modes_are_on()) Py_RETURN_NONE;
    return f();
    END_HANDLE_TH_ERRORS
}

// (handle, K, N) of a layer: the `_native` attribute of the binding's QLinear
struct Layer { qlinear_t h; int64_t K, N; };
bool layer_of(PyObject* t, Layer* l)
{
    if (!PyTuple_CheckExact(t) || PyTuple_GET_SIZE(t) != 3) return false;
    l->h = static_cast<qlinear_t>(PyLong_AsVoidPtr(PyTuple_GET_ITEM(t, 0)));
    l->K = PyLong_AsLongLong(PyTuple_GET_ITEM(t, 1));
    l->N = PyLong_AsLongLong(PyTuple_GET_ITEM(t, 2));
    return l->h != nullptr;
}

template <typename Fn>
PyObject* one_layer(Fn fn, const char* where, PyObject* const* a)        // (layer, x, out, stream)
{
    Layer l;
    const at::Tensor* x = plain(a[1], at::kHalf);
    if (!layer_of(a[0], &l) || !x || x->dim() != 2 || x->size(1) != l.K || x->size(0) > INT_MAX) Py_RETURN_NONE;
    const int64_t M = x->size(0);
    const bool make = a[2] == Py_None;
    at::Tensor made;
    const at::Tensor* out = make ? &made : plain(a[2], at::kHalf);
    if (!make && !is_matrix(out, M, l.N)) Py_RETURN_NONE;
    void *xp = x->data_ptr(), *st = stream_of(a[3]);
    if (!done([&] {
            if (make) made = half_like(*x, {M, l.N});
            return fn(l.h, xp, out->data_ptr(), (int32_t)M, st);
        }, where)) return nullptr;
    return make ? THPVariable_Wrap(std::move(made)) : Py_NewRef(a[2]);
}
PyObject* forward(PyObject*, PyObject* const* a, Py_ssize_t) { return guarded([&] { return one_layer(api.forward, "qlinear_forward", a); }); }
PyObject* kv_scores_one(PyObject*, PyObject* const* a, Py_ssize_t) { return guarded([&] { return one_layer(api.forward, "qlinear_kv_scores", a); }); }
PyObject* forward_a8(PyObject*, PyObject* const* a, Py_ssize_t) { return guarded([&] { return one_layer(api.forward_a8, "qlinear_forward_a8", a); }); }

PyObject* forward_group(PyObject*, PyObject* const* a, Py_ssize_t)       // (list of layers, x, stream)
{
    return guarded([&]() -> PyObject* {
        constexpr int kMost = 4;
        if (!PyList_CheckExact(a[0])) Py_RETURN_NONE;
        const Py_ssize_t n = PyList_GET_SIZE(a[0]);
        const at::Tensor* x = plain(a[1], at::kHalf);
        if (n < 1 || n > kMost || !x || x->dim() != 2 || x->size(0) > INT_MAX) Py_RETURN_NONE;
        qlinear_t hs[kMost];
        void* ys[kMost];
        int64_t N[kMost];
        for (Py_ssize_t i = 0; i < n; ++i) {
            PyObject* t = PyObject_GetAttrString(PyList_GET_ITEM(a[0], i), "_native");
            Layer l{};
            const bool ok = t && layer_of(t, &l);
            Py_XDECREF(t);
            if (!ok) { PyErr_Clear(); Py_RETURN_NONE; }
            if (i == 0 && x->size(1) != l.K) Py_RETURN_NONE;
            hs[i] = l.h; N[i] = l.N;
        }
        const int64_t M = x->size(0);
        at::Tensor outs[kMost];
        void *xp = x->data_ptr(), *st = stream_of(a[2]);
        if (!done([&] {
                for (Py_ssize_t i = 0; i < n; ++i) { outs[i] = half_like(*x, {M, N[i]}); ys[i] = outs[i].data_ptr(); }
                return api.forward_group(hs, (int32_t)n, xp, ys, (int32_t)M, st);
            }, "qlinear_forward_group")) return nullptr;
        PyObject* r = PyList_New(n);
        for (Py_ssize_t i = 0; r && i < n; ++i) PyList_SET_ITEM(r, i, THPVariable_Wrap(std::move(outs[i])));
        return r;
    });
}

PyObject* forward_gated(PyObject*, PyObject* const* a, Py_ssize_t)       // (gate, up, x, act, out, stream)
{
    return guarded([&]() -> PyObject* {
        Layer g, u;
        const at::Tensor* x = plain(a[2], at::kHalf);
        if (!layer_of(a[0], &g) || !layer_of(a[1], &u) || !x || x->dim() != 2 || x->size(1) != g.K || x->size(0) > INT_MAX) Py_RETURN_NONE;
        const int64_t M = x->size(0);
        const int act = (int)PyLong_AsLong(a[3]);
        const bool make = a[4] == Py_None;
        at::Tensor made;
        const at::Tensor* out = make ? &made : plain(a[4], at::kHalf);
        if (!make && !is_matrix(out, M, g.N)) Py_RETURN_NONE;
        void *xp = x->data_ptr(), *st = stream_of(a[5]);
        if (!done([&] {
                if (make) made = half_like(*x, {M, g.N});
                return api.forward_gated(g.h, u.h, xp, out->data_ptr(), (int32_t)M, act, st);
            }, "qlinear_forward_gated")) return nullptr;
        return make ? THPVariable_Wrap(std::move(made)) : Py_NewRef(a[4]);
    });
}

PyObject* residual_rmsnorm(PyObject*, PyObject* const* a, Py_ssize_t)    // (x, residual, gamma, eps, gamma_offset, h_out, y_out, want_h, stream)
{
    return guarded([&]() -> PyObject* {
        const at::Tensor *x = plain(a[0], at::kHalf), *g = plain(a[2], at::kHalf), *r = a[1] == Py_None ? nullptr : plain(a[1], at::kHalf);
        if (!x || x->dim() != 2 || x->size(0) > INT_MAX || x->size(1) > INT_MAX || x->size(1) % 8 || x->size(1) < 8) Py_RETURN_NONE;
        const int64_t M = x->size(0), K = x->size(1);
        const auto same = [&](const at::Tensor* t) { return t->get_device() == x->get_device(); };
        if (!g || g->dim() != 1 || g->size(0) != K || !same(g)) Py_RETURN_NONE;
        if (a[1] != Py_None && (!is_matrix(r, M, K) || !same(r))) Py_RETURN_NONE;
        const double eps = PyFloat_AsDouble(a[3]), offset = PyFloat_AsDouble(a[4]);
        if (PyErr_Occurred()) { PyErr_Clear(); Py_RETURN_NONE; }
        at::Tensor made_h, made_y;
        const at::Tensor *h = nullptr, *y = &made_y;
        if (a[5] != Py_None) { if (!is_matrix(h = plain(a[5], at::kHalf), M, K) || !same(h)) Py_RETURN_NONE; }
        if (a[6] != Py_None) { if (!is_matrix(y = plain(a[6], at::kHalf), M, K) || !same(y)) Py_RETURN_NONE; }
        const int want_h = a[5] == Py_None ? PyObject_IsTrue(a[7]) : 0;
        if (want_h < 0) return nullptr;
        if (want_h) h = &made_h;
        void *xp = x->data_ptr(), *rp = r ? r->data_ptr() : nullptr, *gp = g->data_ptr(), *st = stream_of(a[8]);
        const int dev = x->get_device();
        if (!done([&] {
                if (y == &made_y) made_y = half_like(*x, {M, K});
                if (want_h) made_h = half_like(*x, {M, K});
                return api.residual_rmsnorm(xp, rp, gp, (float)eps, (float)offset, h ? h->data_ptr() : nullptr, y->data_ptr(), (int32_t)M, (int32_t)K, dev, st);
            }, "qlinear_residual_rmsnorm")) return nullptr;
        PyObject* pair = PyTuple_New(2);
        if (!pair) return nullptr;
        PyTuple_SET_ITEM(pair, 0, want_h ? THPVariable_Wrap(std::move(made_h)) : Py_NewRef(a[5]));
        PyTuple_SET_ITEM(pair, 1, a[6] == Py_None ? THPVariable_Wrap(std::move(made_y)) : Py_NewRef(a[6]));
        return pair;
    });
}

PyObject* rope_qkv(PyObject*, PyObject* const* a, Py_ssize_t)            // (q, k, v, pos, cos, sin, B, S, h_q, h_kv, d_h, stream)
{
    return guarded([&]() -> PyObject* {
        const at::Tensor *q = plain(a[0], at::kHalf), *k = plain(a[1], at::kHalf), *v = plain(a[2], at::kHalf), *pos = plain(a[3], at::kInt);
        const at::Tensor *cos = plain(a[4], at::kFloat), *sin = plain(a[5], at::kFloat);
        if (!q || !k || !v || !pos || !cos || !sin) Py_RETURN_NONE;
        int64_t n[5];
        for (int i = 0; i < 5; ++i) {
            if (!PyLong_CheckExact(a[6 + i])) Py_RETURN_NONE;
            n[i] = PyLong_AsLongLong(a[6 + i]);
            if (n[i] < 1 || n[i] > INT_MAX) { PyErr_Clear(); Py_RETURN_NONE; }
        }
        const int64_t B = n[0], S = n[1], hq = n[2], hkv = n[3], d = n[4], T = B * S;
        const auto same = [&](const at::Tensor* t) { return t->get_device() == q->get_device(); };
        if (hq % hkv || d % 16 || T > INT_MAX || hq * d > INT_MAX || !is_matrix(q, T, hq * d) || !is_matrix(k, T, hkv * d) || !is_matrix(v, T, hkv * d) || pos->dim() != 1 || pos->size(0) != T ||
            cos->dim() != 2 || cos->size(0) > INT_MAX || cos->size(1) != d / 2 || !is_matrix(sin, cos->size(0), d / 2) || !same(k) || !same(v) || !same(pos) || !same(cos) || !same(sin)) Py_RETURN_NONE;
        at::Tensor qo, ko, vo;
        const void* in[6] = {q->data_ptr(), k->data_ptr(), v->data_ptr(), pos->data_ptr(), cos->data_ptr(), sin->data_ptr()};
        void* st = stream_of(a[11]);
        const int dev = q->get_device();
        const int32_t n_pos = (int32_t)cos->size(0);
        if (!done([&] {
                qo = half_like(*q, {B * hkv, S * (hq / hkv), d}); ko = half_like(*q, {B * hkv, S, d}); vo = half_like(*q, {B * hkv, S, d});
                return api.rope_qkv(in[0], in[1], in[2], static_cast<const int32_t*>(in[3]), static_cast<const float*>(in[4]), static_cast<const float*>(in[5]), n_pos,
                                    qo.data_ptr(), ko.data_ptr(), vo.data_ptr(), (int32_t)B, (int32_t)S, (int32_t)hq, (int32_t)hkv, (int32_t)d, dev, st);
            }, "qlinear_rope_qkv")) return nullptr;
        PyObject* r = PyTuple_New(3);
        if (!r) return nullptr;
        PyTuple_SET_ITEM(r, 0, THPVariable_Wrap(std::move(qo)));
        PyTuple_SET_ITEM(r, 1, THPVariable_Wrap(std::move(ko)));
        PyTuple_SET_ITEM(r, 2, THPVariable_Wrap(std::move(vo)));
        return r;
    });
}

PyObject* embed(PyObject*, PyObject* const* a, Py_ssize_t)               // (layer, ids, out, stream)
{
    return guarded([&]() -> PyObject* {
        Layer l;
        const at::Tensor* ids = plain(a[1], at::kInt);
        if (!layer_of(a[0], &l) || !ids || ids->dim() != 1 || ids->size(0) > INT_MAX || a[2] != Py_None) Py_RETURN_NONE;
        const int64_t n = ids->size(0);
        at::Tensor out;
        const auto* ip = static_cast<const int32_t*>(ids->data_ptr());
        void* st = stream_of(a[3]);
        if (!done([&] {
                out = half_like(*ids, {n, l.K});
                return api.embed(l.h, ip, (int32_t)n, out.data_ptr(), st);
            }, "qlinear_embed")) return nullptr;
        return THPVariable_Wrap(std::move(out));
    });
}

// The caches of a layer's heads: (n_heads, cache size, d_h, addresses of the arrays of K handles, V handles and V scales): `_native` of KVHeads
struct Heads { int32_t n; int64_t T, d; const qlinear_t *hk, *hv; void* const* vs; };
bool heads_of(PyObject* t, Heads* h)
{
    if (!PyTuple_CheckExact(t) || PyTuple_GET_SIZE(t) != 6) return false;
    h->n = (int32_t)PyLong_AsLong(PyTuple_GET_ITEM(t, 0));
    h->T = PyLong_AsLongLong(PyTuple_GET_ITEM(t, 1));
    h->d = PyLong_AsLongLong(PyTuple_GET_ITEM(t, 2));
    h->hk = static_cast<const qlinear_t*>(PyLong_AsVoidPtr(PyTuple_GET_ITEM(t, 3)));
    h->hv = static_cast<const qlinear_t*>(PyLong_AsVoidPtr(PyTuple_GET_ITEM(t, 4)));
    h->vs = static_cast<void* const*>(PyLong_AsVoidPtr(PyTuple_GET_ITEM(t, 5)));
    return true;
}
bool is_of_heads(const at::Tensor* t, const Heads& h, int64_t cols) { return t && t->dim() == 3 && t->size(0) == h.n && t->size(2) == cols && t->size(1) <= INT_MAX; }

PyObject* kv_append(PyObject*, PyObject* const* a, Py_ssize_t)           // (heads, length, k_new, v_new, stream) -> number of new tokens
{
    return guarded([&]() -> PyObject* {
        Heads h;
        const at::Tensor *k = plain(a[2], at::kHalf), *v = plain(a[3], at::kHalf);
        if (!heads_of(a[0], &h) || !is_of_heads(k, h, h.d) || !is_of_heads(v, h, h.d) || k->size(1) != v->size(1)) Py_RETURN_NONE;
        const int64_t n_new = k->size(1), pos = PyLong_AsLongLong(a[1]);
        if (pos < 0 || pos > INT_MAX) { PyErr_Clear(); Py_RETURN_NONE; }
        void *kp = k->data_ptr(), *vp = v->data_ptr(), *st = stream_of(a[4]);
        if (!done([&] { return api.kv_append_heads(h.hk, h.hv, h.n, kp, vp, n_new * h.d, h.d, h.vs, (int32_t)pos, (int32_t)n_new, st); }, "qlinear_kv_append_heads")) return nullptr;
        return PyLong_FromLongLong(n_new);
    });
}

PyObject* kv_scores(PyObject*, PyObject* const* a, Py_ssize_t)           // (heads, q_rows, stream)
{
    return guarded([&]() -> PyObject* {
        Heads h;
        const at::Tensor* q = plain(a[1], at::kHalf);
        if (!heads_of(a[0], &h) || !is_of_heads(q, h, h.d)) Py_RETURN_NONE;
        const int64_t R = q->size(1);
        at::Tensor out;
        void *qp = q->data_ptr(), *st = stream_of(a[2]);
        if (!done([&] {
                out = half_like(*q, {h.n, R, h.T});
                return api.kv_scores_heads(h.hk, h.n, qp, out.data_ptr(), (int32_t)R, st);
            }, "qlinear_kv_scores_heads")) return nullptr;
        return THPVariable_Wrap(std::move(out));
    });
}

PyObject* kv_output_heads(PyObject*, PyObject* const* a, Py_ssize_t)     // (heads, prob, stream)
{
    return guarded([&]() -> PyObject* {
        Heads h;
        const at::Tensor* p = plain(a[1], at::kHalf);
        if (!heads_of(a[0], &h) || !is_of_heads(p, h, h.T)) Py_RETURN_NONE;
        const int64_t R = p->size(1);
        at::Tensor out;
        void *pp = p->data_ptr(), *st = stream_of(a[2]);
        const auto* vs = reinterpret_cast<const void* const*>(h.vs);
        if (!done([&] {
                out = half_like(*p, {h.n, R, h.d});
                return api.kv_output_heads(h.hv, h.n, pp, vs, out.data_ptr(), (int32_t)R, st);
            }, "qlinear_kv_output_heads")) return nullptr;
        return THPVariable_Wrap(std::move(out));
    });
}

PyObject* kv_output(PyObject*, PyObject* const* a, Py_ssize_t)           // (V layer, V scales, prob, stream)
{
    return guarded([&]() -> PyObject* {
        Layer l;
        const at::Tensor *p = plain(a[2], at::kHalf), *scales = plain(a[1], at::kHalf);
        if (!layer_of(a[0], &l) || !p || !scales || p->dim() != 2 || p->size(1) != l.K || p->size(0) > INT_MAX) Py_RETURN_NONE;
        const int64_t R = p->size(0);
        at::Tensor out, tmp;
        void *vs = scales->data_ptr(), *pp = p->data_ptr(), *st = stream_of(a[3]);
        const bool uses_tmp = R < 1 || api.kv_output_uses_tmp(l.h, pp, vs, (int32_t)R);
        if (!done([&] {
                out = half_like(*p, {R, l.N});
                if (uses_tmp) tmp = half_like(*p, {R, l.K});
                return api.kv_output(l.h, pp, vs, (uses_tmp ? tmp : out).data_ptr(), out.data_ptr(), (int32_t)R, st);
            }, "qlinear_kv_output")) return nullptr;
        return THPVariable_Wrap(std::move(out));
    });
}

// (check, addresses of the entry points in the order of Api)
PyObject* init(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    void** to = reinterpret_cast<void**>(&api);
    if (n != 1 + (Py_ssize_t)(sizeof(Api) / sizeof(void*))) { PyErr_SetString(PyExc_TypeError, "native.init: one check and the entry points"); return nullptr; }
    for (Py_ssize_t i = 1; i < n; ++i) to[i - 1] = PyLong_AsVoidPtr(a[i]);
    Py_XSETREF(check_status, Py_NewRef(a[0]));
    Py_RETURN_NONE;
}

#define FAST(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(name)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {FAST(init), FAST(forward), FAST(forward_a8), FAST(forward_group), FAST(forward_gated), FAST(residual_rmsnorm), FAST(rope_qkv), FAST(embed),
                         FAST(kv_append), FAST(kv_scores), FAST(kv_scores_one), FAST(kv_output_heads), FAST(kv_output), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native(void)
{
    PyObject* m = PyModule_Create(&module);
    if (m && PyModule_AddStringConstant(m, "built_for", QL_BUILT_FOR)) Py_CLEAR(m);   // (the versions of torch and Python; see build.py)
    return m;
}
