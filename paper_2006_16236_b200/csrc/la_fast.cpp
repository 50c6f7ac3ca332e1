// The successful call of the Python binding, in native code.
//
// binding.py checks every tensor it is given and marshals it through ctypes: 15 to 35 us of interpreter work per
// call, more than the kernels of a decode step (2.3 us) or of a short prompt take.  The functions here do the same
// checks on the C++ tensors and call the library (1 to 3 us).  They only ever take the ordinary case: plain CUDA
// tensors of the current device with the right shapes and types.  Anything else - a wrong argument, another device, a
// tensor subclass, a wrapper of a transform, an active function mode - returns NotImplemented before anything is
// allocated or enqueued, and binding.py goes its own way, which also raises its own errors.  A library status other
// than LA_OK is returned as an int.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/ATen.h>
#include <ATen/PythonTorchFunctionTLS.h>
#include <c10/cuda/CUDAFunctions.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include "la.h"

namespace {

enum Kind { kQK, kV, kRow, kS, kZ, kQ1, kV1, kBytes, kLengths };

struct Call {
    la_problem p = {};
    at::ScalarType io = at::kFloat;
    c10::DeviceIndex device = -1;
    bool fits = true;               // so far nothing asks for the general path

    // the plain CUDA tensor behind a Python object, or null
    const at::Tensor* plain(PyObject* o) {
        if (!THPVariable_CheckExact(o)) return nullptr;
        const at::Tensor& t = THPVariable_Unpack(o);
        const auto keys = t.key_set();
        if (!t.is_cuda() || !t.has_storage() || keys.has(c10::DispatchKey::FuncTorchBatched) ||
            keys.has(c10::DispatchKey::FuncTorchGradWrapper) || keys.has(c10::DispatchKey::Functionalize) ||
            keys.has(c10::DispatchKey::Python) || t.layout() != at::kStrided || !t.is_contiguous())
            return nullptr;
        if (device < 0) device = t.device().index();
        return t.device().index() == device ? &t : nullptr;
    }

    bool start(PyObject* q, PyObject* v, int dims, PyObject* phi, PyObject* eps) {
        const at::Tensor *tq = plain(q), *tv = plain(v);
        if (!tq || !tv || tq->dim() != dims || tv->dim() != dims) return fits = false;
        io = tq->scalar_type();
        if (io != at::kFloat && io != at::kBFloat16) return fits = false;
        const auto s = tq->sizes();
        p.B = s[0]; p.H = s[1];
        p.N = dims == 4 ? s[2] : 1;
        p.D = s[dims - 1];
        p.M = tv->size(dims - 1);
        p.dtype = io == at::kFloat ? LA_F32 : LA_BF16;
        return options(phi, eps);
    }
    bool options(PyObject* phi, PyObject* eps) {
        if (device != c10::cuda::current_device() || at::impl::torch_function_mode_enabled()) return fits = false;
        if (PyUnicode_Check(phi)) {
            if (!PyUnicode_CompareWithASCIIString(phi, "elu1")) p.phi = LA_PHI_ELU1;
            else if (!PyUnicode_CompareWithASCIIString(phi, "identity")) p.phi = LA_PHI_IDENTITY;
            else return fits = false;
        } else if (PyLong_CheckExact(phi)) {
            const long x = PyLong_AsLong(phi);
            if (x == -1 && PyErr_Occurred()) { PyErr_Clear(); return fits = false; }
            if (x != LA_PHI_ELU1 && x != LA_PHI_IDENTITY) return fits = false;
            p.phi = (int32_t)x;
        } else {
            return fits = false;
        }
        if (!PyFloat_CheckExact(eps) && !PyLong_CheckExact(eps)) return fits = false;
        const double e = PyFloat_AsDouble(eps);
        if (e == -1.0 && PyErr_Occurred()) { PyErr_Clear(); return fits = false; }
        p.eps = (float)e;
        return true;
    }

    // an argument of the given kind: its tensor, or null for None (fits becomes false if it is neither)
    const at::Tensor* arg(PyObject* o, Kind kind) {
        if (!fits || o == Py_None) return nullptr;
        const at::Tensor* t = plain(o);
        if (!t) { fits = false; return nullptr; }
        const auto s = t->sizes();
        const size_t n = s.size();
        bool ok = false;
        at::ScalarType type = at::kFloat;
        switch (kind) {
            case kQK: ok = n == 4 && s[0] == p.B && s[1] == p.H && s[2] == p.N && s[3] == p.D; type = io; break;
            case kV: ok = n == 4 && s[0] == p.B && s[1] == p.H && s[2] == p.N && s[3] == p.M; type = io; break;
            case kRow: ok = n == 3 && s[0] == p.B && s[1] == p.H && s[2] == p.N; break;
            case kS: ok = n == 4 && s[0] == p.B && s[1] == p.H && s[2] == p.D && s[3] == p.M; break;
            case kZ: ok = n == 3 && s[0] == p.B && s[1] == p.H && s[2] == p.D; break;
            case kQ1: ok = n == 3 && s[0] == p.B && s[1] == p.H && s[2] == p.D; type = io; break;
            case kV1: ok = n == 3 && s[0] == p.B && s[1] == p.H && s[2] == p.M; type = io; break;
            case kBytes: ok = n == 1; type = at::kByte; break;
            case kLengths: ok = n == 1 && s[0] == p.B; type = at::kInt; break;
        }
        if (!ok || t->scalar_type() != type) { fits = false; return nullptr; }
        return t;
    }
    const at::Tensor* need(PyObject* o, Kind kind) {
        const at::Tensor* t = arg(o, kind);
        if (!t) fits = false;
        return t;
    }
    // a two-dimensional tensor of the I/O type
    const at::Tensor* matrix(PyObject* o, int64_t rows, int64_t cols) {
        if (!fits || o == Py_None) return nullptr;
        const at::Tensor* t = plain(o);
        if (!t || t->dim() != 2 || t->size(0) != rows || t->size(1) != cols || t->scalar_type() != io) { fits = false; return nullptr; }
        return t;
    }
    void* stream() const { return c10::cuda::getCurrentCUDAStream(device).stream(); }
    at::Tensor bytes(size_t n) const {
        return at::empty({(int64_t)n}, at::TensorOptions().dtype(at::kByte).device(at::Device(at::kCUDA, device)));
    }
};

void* ptr(const at::Tensor* t) { return t ? t->data_ptr() : nullptr; }
size_t size_of(const at::Tensor* t) { return t ? (size_t)t->numel() : 0; }        // of a byte tensor

// the tensor given, or a new one like `like`
struct Out {
    at::Tensor t;
    PyObject* given;
    Out(PyObject* o, const at::Tensor* g, const at::Tensor& like) : t(g ? *g : at::empty_like(like)), given(g ? o : nullptr) {}
    void* data() const { return t.data_ptr(); }
    PyObject* release() {
        if (given) { Py_INCREF(given); return given; }
        return THPVariable_Wrap(std::move(t));
    }
};

// binding.py's scratch buffers: one per (operation, device), grown on demand, in the dictionary it passes
bool scratch(PyObject* cache, const Call& c, int op, at::Tensor* ws) {
    const size_t need = la_workspace_bytes(&c.p, op);
    if (!need) return true;
    PyObject* key = PyLong_FromLong((long)op * 1024 + c.device);
    if (!key) return false;
    PyObject* held = PyDict_GetItemWithError(cache, key);
    if (held && THPVariable_Check(held) && (size_t)THPVariable_Unpack(held).numel() >= need) {
        *ws = THPVariable_Unpack(held);
    } else {
        *ws = c.bytes(need);
        PyObject* w = THPVariable_Wrap(*ws);
        if (!w || PyDict_SetItem(cache, key, w)) { Py_XDECREF(w); Py_DECREF(key); return false; }
        Py_DECREF(w);
    }
    Py_DECREF(key);
    return true;
}

PyObject* not_here() { Py_RETURN_NOTIMPLEMENTED; }

template <typename F> int unlocked(F f) {
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = f();
    Py_END_ALLOW_THREADS
    return rc;
}

// No C++ exception leaves this file: it becomes the Python exception that torch's own functions raise (an allocation that
// fails is a torch.OutOfMemoryError, which programs catch to go on with a smaller batch).
template <typename F> PyObject* guarded(F f) {
    HANDLE_TH_ERRORS
    return f();
    END_HANDLE_TH_ERRORS
}

PyObject* three(Out& a, Out& b, Out& c) {
    PyObject* r = PyTuple_New(3);
    if (!r) return nullptr;
    Out* o[3] = {&a, &b, &c};
    for (int i = 0; i < 3; ++i) {
        PyObject* x = o[i]->release();
        if (!x) { Py_DECREF(r); return nullptr; }
        PyTuple_SET_ITEM(r, i, x);
    }
    return r;
}

#define LA_NARGS(n)                                                                          \
    if (nargs != (n)) { PyErr_SetString(PyExc_TypeError, "wrong number of arguments"); return nullptr; }

// (q, k, v, S, Z, phi, eps, out)
PyObject* recurrent_step(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
    LA_NARGS(8)
    return guarded([&]() -> PyObject* {
        Call c;
        if (!c.start(a[0], a[2], 3, a[5], a[6])) return not_here();
        const at::Tensor *q = c.need(a[0], kQ1), *k = c.need(a[1], kQ1), *v = c.need(a[2], kV1), *S = c.need(a[3], kS), *Z = c.need(a[4], kZ);
        const at::Tensor* o = c.arg(a[7], kV1);
        if (!c.fits) return not_here();
        Out out(a[7], o, *v);
        void* st = c.stream();
        const int rc = unlocked([&] {
            return la_recurrent_step(&c.p, ptr(q), ptr(k), ptr(v), (float*)ptr(S), (float*)ptr(Z), out.data(), st);
        });
        return rc ? PyLong_FromLong(rc) : out.release();
    });
}

// (x, Wqkv, Wo, S, Z, phi, eps, out, ws, cache)
PyObject* decode_layer_step(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
    LA_NARGS(10)
    return guarded([&]() -> PyObject* {
        Call c;
        const at::Tensor *S = c.plain(a[3]), *x = S ? c.plain(a[0]) : nullptr;
        if (!S || !x || S->dim() != 4 || x->dim() != 2) return not_here();
        c.io = x->scalar_type();
        if (c.io != at::kFloat && c.io != at::kBFloat16) return not_here();
        c.p.B = S->size(0); c.p.H = S->size(1); c.p.N = 1; c.p.D = S->size(2); c.p.M = S->size(3);
        c.p.dtype = c.io == at::kFloat ? LA_F32 : LA_BF16;
        if (!c.options(a[5], a[6])) return not_here();
        const int64_t B = c.p.B, F = c.p.H * c.p.D;
        c.need(a[3], kS);
        x = c.matrix(a[0], B, F);
        const at::Tensor *Wqkv = c.matrix(a[1], 3 * F, F), *Wo = c.matrix(a[2], F, F), *Z = c.need(a[4], kZ);
        const at::Tensor *o = c.matrix(a[7], B, F), *given = c.arg(a[8], kBytes);
        if (!c.fits || !x || !Wqkv || !Wo) return not_here();
        at::Tensor ws;
        if (!given && !scratch(a[9], c, LA_OP_DECODE_LAYER, &ws)) return nullptr;
        if (given) ws = *given;
        Out out(a[7], o, *x);
        void* st = c.stream();
        const int rc = unlocked([&] {
            return la_decode_layer_step(&c.p, ptr(x), ptr(Wqkv), ptr(Wo), (float*)ptr(S), (float*)ptr(Z), out.data(),
                                        ws.defined() ? ws.data_ptr() : nullptr, ws.defined() ? (size_t)ws.numel() : 0, st);
        });
        return rc ? PyLong_FromLong(rc) : out.release();
    });
}

// (Q, K, V, phi, eps, O, den, S_out, Z_out, saved, ws, S_in, Z_in, lengths, cache)
PyObject* causal_forward(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
    LA_NARGS(15)
    return guarded([&]() -> PyObject* {
        Call c;
        if (!c.start(a[0], a[2], 4, a[3], a[4])) return not_here();
        const at::Tensor *Q = c.need(a[0], kQK), *K = c.need(a[1], kQK), *V = c.need(a[2], kV), *o = c.arg(a[5], kV), *den = c.arg(a[6], kRow);
        const at::Tensor *S1 = c.arg(a[7], kS), *Z1 = c.arg(a[8], kZ), *saved = c.arg(a[9], kBytes), *given = c.arg(a[10], kBytes);
        const at::Tensor *S0 = c.arg(a[11], kS), *Z0 = c.arg(a[12], kZ), *len = c.arg(a[13], kLengths);
        if (!c.fits) return not_here();
        const int op = len ? LA_OP_CAUSAL_VARLEN_FORWARD : LA_OP_CAUSAL_FORWARD;
        at::Tensor ws;
        if (given) {
            ws = *given;
        } else if (c.p.dtype == LA_BF16 && c.p.D == c.p.M && (c.p.D == 32 || c.p.D == 64)) {
            if (!scratch(a[14], c, op, &ws)) return nullptr;
        } else if (const size_t n = la_workspace_bytes(&c.p, op)) {        // see _forward_scratch() in binding.py
            ws = c.bytes(n);
        }
        Out O(a[5], o, *V);
        void* st = c.stream();
        void* w = ws.defined() ? ws.data_ptr() : nullptr;
        const size_t wn = ws.defined() ? (size_t)ws.numel() : 0;
        const int rc = unlocked([&] {
            if (len)
                return la_causal_forward_varlen(&c.p, ptr(Q), ptr(K), ptr(V), (const int32_t*)ptr(len), (float*)ptr(S0), (float*)ptr(Z0),
                                                O.data(), (float*)ptr(den), (float*)ptr(S1), (float*)ptr(Z1), ptr(saved), size_of(saved), w, wn, st);
            return la_causal_forward_from(&c.p, ptr(Q), ptr(K), ptr(V), (float*)ptr(S0), (float*)ptr(Z0), O.data(), (float*)ptr(den),
                                          (float*)ptr(S1), (float*)ptr(Z1), ptr(saved), size_of(saved), w, wn, st);
        });
        return rc ? PyLong_FromLong(rc) : O.release();
    });
}

// (Q, K, V, G, phi, eps, O, den, saved, dQ, dK, dV, ws, S_in, Z_in, dS_out, dZ_out, dS_in, dZ_in, lengths, cache)
PyObject* causal_backward(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
    LA_NARGS(21)
    return guarded([&]() -> PyObject* {
        Call c;
        if (!c.start(a[0], a[2], 4, a[4], a[5])) return not_here();
        const at::Tensor *Q = c.need(a[0], kQK), *K = c.need(a[1], kQK), *V = c.need(a[2], kV), *G = c.need(a[3], kV);
        const at::Tensor *O = c.arg(a[6], kV), *den = c.arg(a[7], kRow), *saved = c.arg(a[8], kBytes);
        const at::Tensor *q = c.arg(a[9], kQK), *k = c.arg(a[10], kQK), *v = c.arg(a[11], kV), *given = c.arg(a[12], kBytes);
        const at::Tensor *S0 = c.arg(a[13], kS), *Z0 = c.arg(a[14], kZ), *dS1 = c.arg(a[15], kS), *dZ1 = c.arg(a[16], kZ);
        const at::Tensor *dS0 = c.arg(a[17], kS), *dZ0 = c.arg(a[18], kZ), *len = c.arg(a[19], kLengths);
        if (!c.fits) return not_here();
        at::Tensor ws;
        if (given) ws = *given;
        else if (!scratch(a[20], c, len ? LA_OP_CAUSAL_VARLEN_BACKWARD : LA_OP_CAUSAL_BACKWARD, &ws)) return nullptr;
        Out dQ(a[9], q, *Q), dK(a[10], k, *K), dV(a[11], v, *V);
        void* st = c.stream();
        void* w = ws.defined() ? ws.data_ptr() : nullptr;
        const size_t wn = ws.defined() ? (size_t)ws.numel() : 0;
        const int rc = unlocked([&] {
            if (len)
                return la_causal_backward_varlen(&c.p, ptr(Q), ptr(K), ptr(V), (const int32_t*)ptr(len), (float*)ptr(S0), (float*)ptr(Z0), ptr(O),
                                                 (float*)ptr(den), ptr(G), (float*)ptr(dS1), (float*)ptr(dZ1), ptr(saved), size_of(saved),
                                                 dQ.data(), dK.data(), dV.data(), (float*)ptr(dS0), (float*)ptr(dZ0), w, wn, st);
            return la_causal_backward_from(&c.p, ptr(Q), ptr(K), ptr(V), (float*)ptr(S0), (float*)ptr(Z0), ptr(O), (float*)ptr(den), ptr(G),
                                           (float*)ptr(dS1), (float*)ptr(dZ1), ptr(saved), size_of(saved), dQ.data(), dK.data(), dV.data(),
                                           (float*)ptr(dS0), (float*)ptr(dZ0), w, wn, st);
        });
        return rc ? PyLong_FromLong(rc) : three(dQ, dK, dV);
    });
}

// (Q, K, V, phi, eps, O, den, KV, Zs, ws, saved, lengths, cache)
PyObject* linear_forward(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
    LA_NARGS(13)
    return guarded([&]() -> PyObject* {
        Call c;
        if (!c.start(a[0], a[2], 4, a[3], a[4])) return not_here();
        const at::Tensor *Q = c.need(a[0], kQK), *K = c.need(a[1], kQK), *V = c.need(a[2], kV), *o = c.arg(a[5], kV), *den = c.arg(a[6], kRow);
        const at::Tensor *KV = c.arg(a[7], kS), *Zs = c.arg(a[8], kZ), *given = c.arg(a[9], kBytes), *saved = c.arg(a[10], kBytes);
        const at::Tensor* len = c.arg(a[11], kLengths);
        if (!c.fits) return not_here();
        at::Tensor ws;
        if (given) ws = *given;
        else if (!saved && !scratch(a[12], c, len ? LA_OP_LINEAR_VARLEN_FORWARD : LA_OP_LINEAR_FORWARD, &ws)) return nullptr;
        Out O(a[5], o, *V);
        void* st = c.stream();
        const int rc = unlocked([&] {
            return la_linear_attention_keep(&c.p, ptr(Q), ptr(K), ptr(V), (const int32_t*)ptr(len), O.data(), (float*)ptr(den), (float*)ptr(KV),
                                            (float*)ptr(Zs), ptr(saved), size_of(saved), ws.defined() ? ws.data_ptr() : nullptr,
                                            ws.defined() ? (size_t)ws.numel() : 0, st);
        });
        return rc ? PyLong_FromLong(rc) : O.release();
    });
}

// (Q, K, V, G, phi, eps, O, den, dQ, dK, dV, ws, saved, lengths, cache)
PyObject* linear_backward(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
    LA_NARGS(15)
    return guarded([&]() -> PyObject* {
        Call c;
        if (!c.start(a[0], a[2], 4, a[4], a[5])) return not_here();
        const at::Tensor *Q = c.need(a[0], kQK), *K = c.need(a[1], kQK), *V = c.need(a[2], kV), *G = c.need(a[3], kV);
        const at::Tensor *O = c.arg(a[6], kV), *den = c.arg(a[7], kRow), *q = c.arg(a[8], kQK), *k = c.arg(a[9], kQK), *v = c.arg(a[10], kV);
        const at::Tensor *given = c.arg(a[11], kBytes), *saved = c.arg(a[12], kBytes), *len = c.arg(a[13], kLengths);
        if (!c.fits) return not_here();
        at::Tensor ws;
        // (with a saved buffer binding.py sizes the scratch for whole sequences, ragged or not)
        if (given) ws = *given;
        else if (!scratch(a[14], c, len && !saved ? LA_OP_LINEAR_VARLEN_BACKWARD : LA_OP_LINEAR_BACKWARD, &ws)) return nullptr;
        Out dQ(a[8], q, *Q), dK(a[9], k, *K), dV(a[10], v, *V);
        void* st = c.stream();
        const int rc = unlocked([&] {
            return la_linear_attention_backward_kept(&c.p, ptr(Q), ptr(K), ptr(V), (const int32_t*)ptr(len), ptr(saved), size_of(saved), ptr(O),
                                                     (float*)ptr(den), ptr(G), dQ.data(), dK.data(), dV.data(),
                                                     ws.defined() ? ws.data_ptr() : nullptr, ws.defined() ? (size_t)ws.numel() : 0, st);
        });
        return rc ? PyLong_FromLong(rc) : three(dQ, dK, dV);
    });
}

// (Q, V, phi, eps, op): a new buffer of la_workspace_bytes(op) bytes, None if that is 0
PyObject* new_buffer(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
    LA_NARGS(5)
    return guarded([&]() -> PyObject* {
        Call c;
        if (!c.start(a[0], a[1], 4, a[2], a[3])) return not_here();
        const long op = PyLong_AsLong(a[4]);
        if (op == -1 && PyErr_Occurred()) return nullptr;
        const size_t n = la_workspace_bytes(&c.p, (int32_t)op);
        if (!n) Py_RETURN_NONE;
        return THPVariable_Wrap(c.bytes(n));
    });
}

#define LA_METHOD(f) {#f, (PyCFunction)(void (*)(void))f, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {LA_METHOD(recurrent_step), LA_METHOD(decode_layer_step), LA_METHOD(causal_forward), LA_METHOD(causal_backward),
                         LA_METHOD(linear_forward), LA_METHOD(linear_backward), LA_METHOD(new_buffer), {nullptr, nullptr, 0, nullptr}};
// (build.py looks for this string in the file: built against another torch or Python it is built again)
PyModuleDef module_def = {PyModuleDef_HEAD_INIT, "_la_fast", LA_BUILT_FOR, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__la_fast(void) { return PyModule_Create(&module_def); }
