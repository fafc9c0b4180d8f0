// Argument marshalling of the calls a program makes once per layer or per generated token, as a CPython
// module: the same checks as binding.py's, on the tensors themselves.  Looked at from Python each tensor
// costs four attribute reads and a ctypes conversion, 7 us for the fused prefill call, more than its host
// side takes to enqueue two kernels; here 0.5 us.
//
// Every function returns None, with nothing done, when an argument is not exactly what it expects;
// binding.py then takes its own path, which converts what can be converted and names what cannot.
#include <Python.h>
#include <c10/cuda/CUDAStream.h>

#include <optional>
#include <utility>

#include <torch/csrc/autograd/python_variable.h>

#include "../../include/shotkv.h"

namespace {

PyTypeObject *g_dims, *g_policy, *g_state;      // the ctypes structures of binding.py
decltype(&shotkv_prefill_score) g_prefill_score;
decltype(&shotkv_select_shots) g_select_shots;
decltype(&shotkv_compact_kv) g_compact_kv;
decltype(&shotkv_prefill_compress) g_prefill_compress;
decltype(&shotkv_decode_step) g_decode_step;
decltype(&shotkv_decode_step_attend) g_decode_step_attend;

// Reads one argument after the other; `ok` falls when one is not as expected, and the rest is not read.
struct Args {
    PyObject* const* a;
    Py_ssize_t n, i = 0;
    bool ok = true;

    PyObject* next() {
        if (i >= n) ok = false;
        return ok ? a[i++] : nullptr;
    }
    // memory of an object that offers its buffer; it stays where it is while the caller holds the object
    void* memory(PyObject* o, Py_ssize_t bytes) {
        Py_buffer b;
        if (!ok || PyObject_GetBuffer(o, &b, PyBUF_SIMPLE) != 0) {
            PyErr_Clear();
            ok = false;
            return nullptr;
        }
        void* p = b.buf;
        if (b.len != bytes) ok = false;
        PyBuffer_Release(&b);
        return p;
    }
    template <class T>
    T* structure(PyTypeObject* type) {
        PyObject* o = next();
        if (!ok || Py_TYPE(o) != type) {
            ok = false;
            return nullptr;
        }
        return static_cast<T*>(memory(o, sizeof(T)));
    }
    shotkv_ctx* context() {                     // a ctypes.c_void_p
        PyObject* o = next();
        void* p = memory(o, sizeof(void*));
        return ok ? *static_cast<shotkv_ctx**>(p) : nullptr;
    }
    const at::Tensor* cuda_tensor() {
        PyObject* o = next();
        if (!ok || !THPVariable_CheckExact(o)) {
            ok = false;
            return nullptr;
        }
        const at::Tensor& t = THPVariable_Unpack(o);
        if (!t.is_cuda() || t.layout() != at::kStrided || !t.is_contiguous()) ok = false;
        return ok ? &t : nullptr;
    }
    template <class T>
    T* tensor(at::ScalarType type) {
        if (ok && i < n && a[i] == Py_None) {
            ++i;
            return nullptr;
        }
        const at::Tensor* t = cuda_tensor();
        if (ok && t->scalar_type() != type) ok = false;
        return ok ? static_cast<T*>(t->data_ptr()) : nullptr;
    }
    shotkv_bf16* bf16() { return tensor<shotkv_bf16>(at::kBFloat16); }
    float* f32() { return tensor<float>(at::kFloat); }
    int32_t* i32() { return tensor<int32_t>(at::kInt); }
    uint8_t* u8() { return tensor<uint8_t>(at::kByte); }
    void* raw(size_t& bytes) {
        const at::Tensor* t = cuda_tensor();
        if (!ok) return nullptr;
        bytes = t->nbytes();
        return t->data_ptr();
    }
    // a C-contiguous int32 array of B * (S + 1) numbers
    const int32_t* offsets(const shotkv_dims* d) {
        PyObject* o = next();
        Py_buffer b;
        if (!ok || !d || PyObject_GetBuffer(o, &b, PyBUF_C_CONTIGUOUS | PyBUF_FORMAT) != 0) {
            PyErr_Clear();
            ok = false;
            return nullptr;
        }
        const int32_t* p = static_cast<const int32_t*>(b.buf);
        if (b.itemsize != 4 || !b.format || b.format[0] != 'i' || b.format[1] || b.len != 4LL * d->B * (d->S + 1LL)) ok = false;
        PyBuffer_Release(&b);
        return p;
    }
    long long integer(long long lo, long long hi) {
        PyObject* o = next();
        if (!ok || !PyLong_CheckExact(o)) {
            ok = false;
            return 0;
        }
        int over = 0;
        const long long v = PyLong_AsLongLongAndOverflow(o, &over);
        if (over || v < lo || v > hi) ok = false;
        return v;
    }
    // None: torch's current stream of the current device
    void* stream() {
        PyObject* o = next();
        if (!ok || o != Py_None || i != n) {
            ok = false;
            return nullptr;
        }
        return c10::cuda::getCurrentCUDAStream().stream();
    }
};

// `body` reads its arguments and, when all were as expected, returns a call to make without the
// interpreter's lock.  Only the reading may throw (a tensor that cannot say where it lies): an exception out of
// the call would be caught without the lock.
template <class Body>
PyObject* guarded(PyObject* const* a, Py_ssize_t n, Body&& body) {
    using Call = decltype(body(std::declval<Args&>()));
    std::optional<Call> call;
    Args g{a, n};
    try {
        call.emplace(body(g));
    } catch (...) {
        Py_RETURN_NONE;
    }
    if (!g.ok) Py_RETURN_NONE;
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = (*call)();
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

PyObject* prefill_score(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(a, n, [](Args& g) {
        auto* c = g.context();
        auto* d = g.structure<shotkv_dims>(g_dims);
        auto *Q = g.bf16(), *K = g.bf16();
        auto* imp = g.f32();
        size_t wsb = 0;
        void* ws = g.raw(wsb);
        void* st = g.stream();
        return [=] { return g_prefill_score(c, d, Q, K, imp, ws, wsb, st); };
    });
}
PyObject* select_shots(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(a, n, [](Args& g) {
        auto* c = g.context();
        auto* d = g.structure<shotkv_dims>(g_dims);
        auto* p = g.structure<shotkv_policy>(g_policy);
        auto* imp = g.f32();
        auto* off = g.offsets(d);
        auto* score = g.f32();
        auto* keep = g.u8();
        auto *idx = g.i32(), *count = g.i32();
        const int32_t mcap = (int32_t)g.integer(INT32_MIN, INT32_MAX);
        size_t wsb = 0;
        void* ws = g.raw(wsb);
        void* st = g.stream();
        return [=] { return g_select_shots(c, d, p, imp, off, score, keep, idx, count, mcap, ws, wsb, st); };
    });
}
PyObject* compact_kv(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(a, n, [](Args& g) {
        auto* c = g.context();
        auto* d = g.structure<shotkv_dims>(g_dims);
        auto *K = g.bf16(), *V = g.bf16();
        auto *idx = g.i32(), *count = g.i32();
        const int32_t mcap = (int32_t)g.integer(INT32_MIN, INT32_MAX);
        auto *Kc = g.bf16(), *Vc = g.bf16();
        void* st = g.stream();
        return [=] { return g_compact_kv(c, d, K, V, idx, count, mcap, Kc, Vc, st); };
    });
}
PyObject* prefill_compress(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(a, n, [](Args& g) {
        auto* c = g.context();
        auto* d = g.structure<shotkv_dims>(g_dims);
        auto* p = g.structure<shotkv_policy>(g_policy);
        auto *Q = g.bf16(), *K = g.bf16(), *V = g.bf16();
        auto* off = g.offsets(d);
        auto* score = g.f32();
        auto* keep = g.u8();
        auto *idx = g.i32(), *count = g.i32();
        const int32_t mcap = (int32_t)g.integer(INT32_MIN, INT32_MAX);
        auto *Kc = g.bf16(), *Vc = g.bf16();
        auto* imp = g.f32();
        const uint32_t flags = (uint32_t)g.integer(0, UINT32_MAX);
        size_t wsb = 0;
        void* ws = g.raw(wsb);
        void* st = g.stream();
        return [=] { return g_prefill_compress(c, d, p, Q, K, V, off, score, keep, idx, count, mcap, Kc, Vc, imp, flags, ws, wsb, st); };
    });
}
PyObject* decode_step(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(a, n, [](Args& g) {
        auto* c = g.context();
        auto* s = g.structure<shotkv_decode_state>(g_state);
        auto *q = g.bf16(), *k = g.bf16(), *v = g.bf16(), *Kc = g.bf16();
        auto* count = g.i32();
        void* st = g.stream();
        return [=] { return g_decode_step(c, s, q, k, v, Kc, count, st); };
    });
}
PyObject* decode_step_attend(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(a, n, [](Args& g) {
        auto* c = g.context();
        auto* s = g.structure<shotkv_decode_state>(g_state);
        auto *q = g.bf16(), *k = g.bf16(), *v = g.bf16(), *Kc = g.bf16(), *Vc = g.bf16();
        auto* count = g.i32();
        auto* out = g.f32();
        void* st = g.stream();
        return [=] { return g_decode_step_attend(c, s, q, k, v, Kc, Vc, count, out, st); };
    });
}

// init(Dims, Policy, DecodeState, addresses of the six functions in the order above)
PyObject* init(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (n != 9 || !PyType_Check(a[0]) || !PyType_Check(a[1]) || !PyType_Check(a[2])) {
        PyErr_SetString(PyExc_TypeError, "init(Dims, Policy, DecodeState, six addresses)");
        return nullptr;
    }
    void* f[6];
    for (int k = 0; k < 6; ++k) {
        f[k] = PyLong_AsVoidPtr(a[3 + k]);
        if (PyErr_Occurred()) return nullptr;
    }
    PyTypeObject** types[3] = {&g_dims, &g_policy, &g_state};
    for (int k = 0; k < 3; ++k) {
        Py_INCREF(a[k]);
        Py_XDECREF(reinterpret_cast<PyObject*>(*types[k]));
        *types[k] = reinterpret_cast<PyTypeObject*>(a[k]);
    }
    g_prefill_score = reinterpret_cast<decltype(g_prefill_score)>(f[0]);
    g_select_shots = reinterpret_cast<decltype(g_select_shots)>(f[1]);
    g_compact_kv = reinterpret_cast<decltype(g_compact_kv)>(f[2]);
    g_prefill_compress = reinterpret_cast<decltype(g_prefill_compress)>(f[3]);
    g_decode_step = reinterpret_cast<decltype(g_decode_step)>(f[4]);
    g_decode_step_attend = reinterpret_cast<decltype(g_decode_step_attend)>(f[5]);
    Py_RETURN_NONE;
}

#define FAST(name) {#name, (PyCFunction)(void (*)(void))name, METH_FASTCALL, nullptr}
PyMethodDef g_methods[] = {FAST(init), FAST(prefill_score), FAST(select_shots), FAST(compact_kv), FAST(prefill_compress),
                           FAST(decode_step), FAST(decode_step_attend), {nullptr, nullptr, 0, nullptr}};
PyModuleDef g_module = {PyModuleDef_HEAD_INIT, "_marshal", nullptr, -1, g_methods};

}  // namespace

PyMODINIT_FUNC PyInit__marshal() { return PyModule_Create(&g_module); }
