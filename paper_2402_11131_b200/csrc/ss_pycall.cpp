// CPython side of the binding: takes tensors apart and calls the C entry points (ss_msa.h) of the library that api.py has
// loaded, whose addresses it is given: it is not linked to one.
//
// A decode step of a small model is a handful of calls of 3 to 8 us of GPU time each, so the host has to spend less than that
// on a call.  Through ctypes, with the pointers collected in Python, a verification call took 5.6 us, of which the launch is
// 2.6; here it takes 3.5 us.  Only the CPython API is used: a tensor is any object with `data_ptr()`, `shape` and
// `nbytes`.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include "ss_msa.h"

namespace {

PyObject *s_data_ptr, *s_shape, *s_nbytes, *s_cuda_stream;      // interned attribute names
PyObject *g_error, *g_raw_stream, *g_device;                    // SsError; torch's raw current stream and current device
PyObject *g_attn_params, *g_cache_layout;                       // the ctypes structures of ss_attn_params and ss_cache_layout
// the entry points, in the order in which setup() takes them
#define SS_FUNCTIONS(F)                                                                                                 \
    F(ss_msa_attention) F(ss_tree_verify) F(ss_tree_verify_soft) F(ss_tree_verify_sampled) F(ss_tree_prune)             \
    F(ss_next_draft) F(ss_kv_compact) F(ss_stream_insert) F(ss_value_rotate)
struct Functions {
#define SS_MEMBER(name) decltype(&::name) name;
    SS_FUNCTIONS(SS_MEMBER)
} g_lib;
PyObject *g_byref, *g_argument_error;                           // ctypes.byref and ctypes.ArgumentError

// One call's arguments.  After the first Python error everything reads as zero and `ok` stays false.
struct Args {
    PyObject* const* a;
    bool ok;
    void* ptr(int i) {
        if (!ok || a[i] == Py_None) return nullptr;
        PyObject* r = PyObject_CallMethodNoArgs(a[i], s_data_ptr);
        void* p = r ? reinterpret_cast<void*>(PyLong_AsUnsignedLongLong(r)) : nullptr;
        if (!r || PyErr_Occurred()) ok = false;
        Py_XDECREF(r);
        return p;
    }
    template <typename T>
    T* as(int i) { return static_cast<T*>(ptr(i)); }
    // the first n sizes of argument i, which has to have exactly (or at least) n dimensions
    void sizes(int i, int n, long long* out, bool exact = true) {
        for (int k = 0; k < n; ++k) out[k] = 0;
        if (!ok) return;
        PyObject* s = PyObject_GetAttr(a[i], s_shape);
        if (!s || !PyTuple_Check(s) || PyTuple_GET_SIZE(s) < n || (exact && PyTuple_GET_SIZE(s) != n)) {
            if (s && !PyErr_Occurred()) PyErr_Format(PyExc_ValueError, "expected a tensor of %d dimensions", n);
            ok = false;
        } else {
            for (int k = 0; k < n; ++k) out[k] = PyLong_AsLongLong(PyTuple_GET_ITEM(s, k));
        }
        Py_XDECREF(s);
    }
    size_t nbytes(int i) {
        if (!ok) return 0;
        PyObject* r = PyObject_GetAttr(a[i], s_nbytes);
        const size_t n = r ? static_cast<size_t>(PyLong_AsUnsignedLongLong(r)) : 0;
        if (!r || PyErr_Occurred()) ok = false;
        Py_XDECREF(r);
        return n;
    }
    int32_t i32(int i) {
        const long v = ok ? PyLong_AsLong(a[i]) : 0;
        if (v == -1 && PyErr_Occurred()) ok = false;
        return static_cast<int32_t>(v);
    }
    float f32(int i) {
        const double v = ok ? PyFloat_AsDouble(a[i]) : 0.0;
        if (v == -1.0 && PyErr_Occurred()) ok = false;
        return static_cast<float>(v);
    }
    // a torch.cuda.Stream, or None for the current stream of the current device
    void* stream(int i) {
        if (!ok) return nullptr;
        PyObject* r;
        if (a[i] != Py_None) {
            r = PyObject_GetAttr(a[i], s_cuda_stream);
        } else {
            PyObject* dev = PyObject_CallNoArgs(g_device);
            r = dev ? PyObject_CallOneArg(g_raw_stream, dev) : nullptr;
            Py_XDECREF(dev);
        }
        void* p = r ? reinterpret_cast<void*>(PyLong_AsUnsignedLongLong(r)) : nullptr;
        if (!r || PyErr_Occurred()) ok = false;
        Py_XDECREF(r);
        return p;
    }
    // The memory of a ctypes structure of class `type`.  Anything else is refused as ctypes refuses it: a TypeError for what is
    // no ctypes object, an ArgumentError for another one.
    template <typename T>
    const T* structure(int i, PyObject* type, Py_buffer* view) {
        view->obj = nullptr;
        if (!ok) return nullptr;
        ok = false;
        const int is = PyObject_IsInstance(a[i], type);
        if (is < 0) return nullptr;
        if (!is) {
            PyObject* r = PyObject_CallOneArg(g_byref, a[i]);
            if (r) PyErr_Format(g_argument_error, "expected an instance of %R instead of %R", type, reinterpret_cast<PyObject*>(Py_TYPE(a[i])));
            Py_XDECREF(r);
            return nullptr;
        }
        if (PyObject_GetBuffer(a[i], view, PyBUF_SIMPLE) != 0) return nullptr;
        ok = view->len >= static_cast<Py_ssize_t>(sizeof(T));
        if (ok) return static_cast<const T*>(view->buf);
        PyBuffer_Release(view);
        PyErr_Format(g_argument_error, "%R is smaller than the structure", type);
        return nullptr;
    }
};

PyObject* done(const char* what, int32_t status) {
    if (status == SS_OK) Py_RETURN_NONE;
    PyObject* e = PyObject_CallFunction(g_error, "si", what, static_cast<int>(status));
    if (e) PyErr_SetObject(g_error, e);
    Py_XDECREF(e);
    return nullptr;
}

#define SS_ENTRY(name, count)                                                                    \
    PyObject* name(PyObject*, PyObject* const* argv, Py_ssize_t argc) {                          \
        if (argc != count) return PyErr_Format(PyExc_TypeError, #name ": %d arguments", count);  \
        Args a{argv, true};                                                                      \
        int32_t st = SS_OK;
// (the GIL is free while the call runs, as under ctypes)
#define SS_CALL(expr)                                                                            \
        if (!a.ok) return nullptr;                                                               \
        Py_BEGIN_ALLOW_THREADS st = expr;                                                        \
        Py_END_ALLOW_THREADS

SS_ENTRY(msa_attention, 2)
    Py_buffer view;
    void* const s = a.stream(1);
    const ss_attn_params* const p = a.structure<ss_attn_params>(0, g_attn_params, &view);
    SS_CALL(g_lib.ss_msa_attention(p, s))
    PyBuffer_Release(&view);
    return done("ss_msa_attention", st);
}

SS_ENTRY(tree_verify, 10)
    long long n[3];
    a.sizes(0, 3, n);
    const float* lg = a.as<float>(0);
    const int32_t* tok = a.as<int32_t>(1);
    const ss_tree_desc* tr = a.as<ss_tree_desc>(2);
    int32_t *al = a.as<int32_t>(3), *ap = a.as<int32_t>(4), *ln = a.as<int32_t>(5), *bt = a.as<int32_t>(6), *am = a.as<int32_t>(7);
    void* const ws = a.ptr(8);
    const size_t wb = a.nbytes(8);
    void* const s = a.stream(9);
    SS_CALL(g_lib.ss_tree_verify(lg, tok, tr, static_cast<int32_t>(n[0]), static_cast<int32_t>(n[1]), static_cast<int32_t>(n[2]), al, ap, ln, bt, am, ws, wb, s))
    return done("ss_tree_verify", st);
}

SS_ENTRY(tree_verify_soft, 13)
    long long n[3];
    a.sizes(0, 3, n);
    const float* lg = a.as<float>(0);
    const int32_t* tok = a.as<int32_t>(1);
    const ss_tree_desc* tr = a.as<ss_tree_desc>(2);
    const float eps = a.f32(3), delta = a.f32(4);
    int32_t *al = a.as<int32_t>(5), *ap = a.as<int32_t>(6), *ln = a.as<int32_t>(7), *bt = a.as<int32_t>(8);
    float *ep = a.as<float>(9), *en = a.as<float>(10);
    void* const ws = a.ptr(11);
    const size_t wb = a.nbytes(11);
    void* const s = a.stream(12);
    SS_CALL(g_lib.ss_tree_verify_soft(lg, tok, tr, static_cast<int32_t>(n[0]), static_cast<int32_t>(n[1]), static_cast<int32_t>(n[2]), eps, delta, al, ap, ln, bt,
                                ep, en, ws, wb, s))
    return done("ss_tree_verify_soft", st);
}

SS_ENTRY(tree_verify_sampled, 12)
    long long n[3];
    a.sizes(0, 3, n);
    const float* lg = a.as<float>(0);
    const int32_t* tok = a.as<int32_t>(1);
    const ss_tree_desc* tr = a.as<ss_tree_desc>(2);
    const float* un = a.as<float>(3);
    const int32_t k = a.i32(4);
    int32_t *al = a.as<int32_t>(5), *ap = a.as<int32_t>(6), *ln = a.as<int32_t>(7), *bt = a.as<int32_t>(8), *nt = a.as<int32_t>(9);
    void* const ws = a.ptr(10);
    const size_t wb = a.nbytes(10);
    void* const s = a.stream(11);
    SS_CALL(g_lib.ss_tree_verify_sampled(lg, tok, tr, un, static_cast<int32_t>(n[0]), static_cast<int32_t>(n[1]), static_cast<int32_t>(n[2]), k, al, ap, ln, bt, nt,
                                   ws, wb, s))
    return done("ss_tree_verify_sampled", st);
}

SS_ENTRY(tree_prune, 11)
    long long n[3];
    a.sizes(0, 3, n);
    const float* lg = a.as<float>(0);
    const int32_t* tok = a.as<int32_t>(1);
    const ss_tree_desc* tr = a.as<ss_tree_desc>(2);
    const float threshold = a.f32(3);
    float* ep = a.as<float>(4);
    int32_t *ni = a.as<int32_t>(5), *kn = a.as<int32_t>(6), *kt = a.as<int32_t>(7);
    ss_tree_desc* pt = a.as<ss_tree_desc>(8);
    void* const ws = a.ptr(9);
    const size_t wb = a.nbytes(9);
    void* const s = a.stream(10);
    SS_CALL(g_lib.ss_tree_prune(lg, tok, tr, static_cast<int32_t>(n[0]), static_cast<int32_t>(n[1]), static_cast<int32_t>(n[2]), threshold, ep, ni, kn, kt, pt, ws, wb, s))
    return done("ss_tree_prune", st);
}

SS_ENTRY(next_draft, 9)
    long long n[4];
    a.sizes(0, 4, n);
    const float* lg = a.as<float>(0);
    const int32_t *ri = a.as<int32_t>(1), *bt = a.as<int32_t>(2);
    const int32_t k = a.i32(3), nodes = a.i32(4);
    int32_t* tok = a.as<int32_t>(5);
    ss_tree_desc* tr = a.as<ss_tree_desc>(6);
    void* const ws = a.ptr(7);
    const size_t wb = a.nbytes(7);
    void* const s = a.stream(8);
    SS_CALL(g_lib.ss_next_draft(lg, static_cast<int32_t>(n[1]), ri, bt, static_cast<int32_t>(n[0]), static_cast<int32_t>(n[2]), static_cast<int32_t>(n[3]), k, nodes, tok,
                          tr, ws, wb, s))
    return done("ss_next_draft", st);
}

SS_ENTRY(kv_compact, 9)
    long long n[1];
    Py_buffer view;
    void *k = a.ptr(0), *v = a.ptr(1);
    a.sizes(3, 1, n, false);
    const int64_t* ks = a.as<int64_t>(3);
    const int32_t *kl = a.as<int32_t>(4), *al = a.as<int32_t>(5), *ap = a.as<int32_t>(6);
    int32_t* ko = a.as<int32_t>(7);
    void* const s = a.stream(8);
    const ss_cache_layout* const lo = a.structure<ss_cache_layout>(2, g_cache_layout, &view);
    SS_CALL(g_lib.ss_kv_compact(k, v, lo, static_cast<int32_t>(n[0]), ks, kl, al, ap, ko, s))
    PyBuffer_Release(&view);
    return done("ss_kv_compact", st);
}

SS_ENTRY(stream_insert, 4)
    long long n[2], g[1];
    a.sizes(0, 2, n);
    a.sizes(1, 1, g, false);
    void *m = a.ptr(0), *e = a.ptr(1), *o = a.ptr(2);
    void* const s = a.stream(3);
    SS_CALL(g_lib.ss_stream_insert(m, e, o, n[0], static_cast<int32_t>(g[0]), static_cast<int32_t>(n[1]), s))
    return done("ss_stream_insert", st);
}

SS_ENTRY(value_rotate, 4)
    long long n[2], g[2];
    a.sizes(0, 2, n);
    a.sizes(1, 2, g, false);
    void *v = a.ptr(0), *o = a.ptr(1);
    const float epsilon = a.f32(2);
    void* const s = a.stream(3);
    SS_CALL(g_lib.ss_value_rotate(v, o, n[0], static_cast<int32_t>(g[1]), static_cast<int32_t>(n[1]), epsilon, s))
    return done("ss_value_rotate", st);
}

// setup(SsError, raw_stream(device) -> int, device() -> int, AttnParams, CacheLayout, ctypes.byref, ctypes.ArgumentError,
//       addresses of SS_FUNCTIONS: a tuple of int)
SS_ENTRY(setup, 8)
    (void)a; (void)st;
    PyObject* const at = argv[7];
    Py_ssize_t n = 0;
    Functions lib = {};
#define SS_TAKE(name)                                                                                                   \
    if (PyTuple_Check(at) && n < PyTuple_GET_SIZE(at)) lib.name = reinterpret_cast<decltype(lib.name)>(PyLong_AsVoidPtr(PyTuple_GET_ITEM(at, n))); \
    if (!lib.name) return PyErr_Occurred() ? nullptr : PyErr_Format(PyExc_ValueError, "setup: no address of %s", #name);  \
    ++n;
    SS_FUNCTIONS(SS_TAKE)
    g_lib = lib;
    PyObject** const kept[7] = {&g_error, &g_raw_stream, &g_device, &g_attn_params, &g_cache_layout, &g_byref, &g_argument_error};
    for (int i = 0; i < 7; ++i) Py_XSETREF(*kept[i], Py_NewRef(argv[i]));
    Py_RETURN_NONE;
}

#define SS_METHOD(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(name)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {SS_METHOD(setup), SS_METHOD(msa_attention), SS_METHOD(tree_verify), SS_METHOD(tree_verify_soft),
                         SS_METHOD(tree_verify_sampled), SS_METHOD(tree_prune), SS_METHOD(next_draft), SS_METHOD(kv_compact),
                         SS_METHOD(stream_insert), SS_METHOD(value_rotate), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_pycall", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__pycall() {
    s_data_ptr = PyUnicode_InternFromString("data_ptr");
    s_shape = PyUnicode_InternFromString("shape");
    s_nbytes = PyUnicode_InternFromString("nbytes");
    s_cuda_stream = PyUnicode_InternFromString("cuda_stream");
    return PyModule_Create(&module);
}
