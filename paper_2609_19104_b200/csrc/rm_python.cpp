// CPython side of the binding: the calls of a control loop, from Python objects straight to the C ABI.
//
// A call of this library can be shorter on the GPU than its marshalling through ctypes was on the host (a mask compaction:
// 8 us of Python and ctypes for ~5 us of kernel; 18 layer pointers alone: 7 us).  These functions take the tensors
// themselves, read their data pointers, and release the interpreter lock around the call.  Integer arguments may be
// anything int() accepts, within the range of the C argument; a tensor argument may be None (NULL).
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <climits>
#include <new>
#include <vector>

#include "rmuscle.h"

namespace {

PyObject* g_data_ptr = nullptr;            // "data_ptr"
PyObject* g_get_device = nullptr;          // torch._C._cuda_getDevice
PyObject* g_raw_stream = nullptr;          // torch._C._cuda_getCurrentRawStream

struct Args {                              // positional arguments, converted one after the other; `bad` once one failed
    PyObject* const* a;
    Py_ssize_t n, i = 0;
    bool bad = false;
    PyObject* next() {
        if (i >= n) {
            if (!bad) PyErr_SetString(PyExc_TypeError, "missing argument");
            bad = true;
            return nullptr;
        }
        return a[i++];
    }
    long long integer() {
        PyObject* o = next();
        if (bad) return 0;
        long long v;
        if (PyLong_Check(o)) {
            v = PyLong_AsLongLong(o);
        } else {
            PyObject* l = PyNumber_Long(o);
            if (!l) { bad = true; return 0; }
            v = PyLong_AsLongLong(l);
            Py_DECREF(l);
        }
        if (v == -1 && PyErr_Occurred()) bad = true;
        return v;
    }
    int i32() {
        const long long v = integer();
        if (!bad && (v < INT_MIN || v > INT_MAX)) {
            PyErr_Format(PyExc_OverflowError, "argument %zd is outside the range of a 32-bit integer", i - 1);
            bad = true;
        }
        return bad ? 0 : (int)v;
    }
    bool truth() {
        PyObject* o = next();
        const int v = bad ? 0 : PyObject_IsTrue(o);
        if (v < 0) bad = true;
        return v > 0;
    }
    double real() {
        PyObject* o = next();
        if (bad) return 0.0;
        PyObject* f = PyNumber_Float(o);
        if (!f) { bad = true; return 0.0; }
        const double v = PyFloat_AS_DOUBLE(f);
        Py_DECREF(f);
        return v;
    }
    static void* pointer_of(PyObject* o, bool& bad) {
        if (bad || o == Py_None) return nullptr;
        PyObject* r = PyObject_VectorcallMethod(g_data_ptr, &o, 1 | PY_VECTORCALL_ARGUMENTS_OFFSET, nullptr);
        if (!r) { bad = true; return nullptr; }
        void* p = PyLong_AsVoidPtr(r);
        Py_DECREF(r);
        if (!p && PyErr_Occurred()) bad = true;
        return p;
    }
    template <class T = void>
    T* pointer() {
        PyObject* o = next();
        return bad ? nullptr : static_cast<T*>(pointer_of(o, bad));
    }
    void pointers(std::vector<void*>& out) {   // a sequence of tensors
        PyObject* o = next();
        if (bad) return;
        PyObject* s = PySequence_Fast(o, "a sequence of tensors is expected");
        if (!s) { bad = true; return; }
        const Py_ssize_t m = PySequence_Fast_GET_SIZE(s);
        try {
            out.resize((size_t)m);
        } catch (const std::bad_alloc&) {
            PyErr_NoMemory();
            bad = true;
        }
        for (Py_ssize_t k = 0; k < m && !bad; ++k) out[(size_t)k] = pointer_of(PySequence_Fast_GET_ITEM(s, k), bad);
        Py_DECREF(s);
    }
    void layers(std::vector<void*>& out) { // a sequence of a step's packed layers, then their number: the call reads that many
        pointers(out);
        const int L = i32();
        if (!bad && (long long)out.size() < L) {
            PyErr_Format(PyExc_ValueError, "%zd packed layers for a model of %d", (Py_ssize_t)out.size(), L);
            bad = true;
        }
    }
    bool done() {                          // every argument has been read
        if (!bad && i != n) {
            PyErr_Format(PyExc_TypeError, "%zd arguments where %zd are expected", n, i);
            bad = true;
        }
        return !bad;
    }
    rm_ctx* context() { return reinterpret_cast<rm_ctx*>((uintptr_t)integer()); }
};

// torch's current stream of the current device
void* current_stream(bool& bad) {
    if (bad) return nullptr;
    PyObject* dev = PyObject_CallNoArgs(g_get_device);
    PyObject* st = dev ? PyObject_CallOneArg(g_raw_stream, dev) : nullptr;
    Py_XDECREF(dev);
    if (!st) { bad = true; return nullptr; }
    void* p = PyLong_AsVoidPtr(st);
    Py_DECREF(st);
    if (!p && PyErr_Occurred()) bad = true;
    return p;
}

template <class F>
PyObject* call(const Args& in, F f) {
    if (in.bad) return nullptr;
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = f();
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

#define RM_FN(name) PyObject* name(PyObject*, PyObject* const* args, Py_ssize_t n_args)

// (ctx, records, kind, reduce, threshold, k, min_votes, scale, scale_per_list, n_lists, I, idx_out, count_out, stride)
RM_FN(mask_compact) {
    Args in{args, n_args};
    rm_ctx* ctx = in.context();
    std::vector<void*> rec;
    in.pointers(rec);
    rm_mask_src s{};
    s.kind = in.i32();
    s.reduce = in.i32();
    s.threshold = (float)in.real();
    s.k = in.i32();
    s.min_votes = in.i32();
    s.scale = in.pointer<const float>();
    s.scale_per_list = in.truth();
    s.n_lists = in.i32();
    s.I = in.i32();
    int32_t* idx = in.pointer<int32_t>();
    int32_t* cnt = in.pointer<int32_t>();
    const int64_t stride = in.integer();
    void* st = in.done() ? current_stream(in.bad) : nullptr;
    s.n_records = (int32_t)rec.size();
    if (rec.empty()) rec.push_back(nullptr);
    s.records = rec.data();
    return call(in, [&] { return rm_mask_compact(ctx, &s, idx, cnt, stride, st); });
}

// (ctx, packed, x, residual, idx, count, y, record_out, record_scale, T, ws, ws_bytes)
RM_FN(sparse_mlp) {
    Args in{args, n_args};
    rm_ctx* ctx = in.context();
    void *packed = in.pointer(), *x = in.pointer();
    float* r = in.pointer<float>();
    int32_t *idx = in.pointer<int32_t>(), *cnt = in.pointer<int32_t>();
    float *y = in.pointer<float>(), *rec = in.pointer<float>(), *sc = in.pointer<float>();
    const int T = in.i32();
    void* ws = in.pointer();
    const size_t nws = (size_t)in.integer();
    void* st = in.done() ? current_stream(in.bad) : nullptr;
    return call(in, [&] { return rm_sparse_mlp(ctx, packed, x, r, idx, cnt, y, rec, sc, T, ws, nws, st); });
}

// (packed, x, residual, idx, count, y, T, H, I)
RM_FN(sparse_mlp_static) {
    Args in{args, n_args};
    void *packed = in.pointer(), *x = in.pointer();
    float* r = in.pointer<float>();
    int32_t *idx = in.pointer<int32_t>(), *cnt = in.pointer<int32_t>();
    float* y = in.pointer<float>();
    const int T = in.i32(), H = in.i32(), I = in.i32();
    void* st = in.done() ? current_stream(in.bad) : nullptr;
    return call(in, [&] { return rm_sparse_mlp_static(packed, x, r, idx, cnt, y, T, H, I, st); });
}

// (ctx, layers, L, r_in, idx, count, stride, r_out, records_out, record_scale, B, T, ws, ws_bytes)
RM_FN(step) {
    Args in{args, n_args};
    rm_ctx* ctx = in.context();
    std::vector<void*> layers;
    in.layers(layers);
    float* r_in = in.pointer<float>();
    int32_t *idx = in.pointer<int32_t>(), *cnt = in.pointer<int32_t>();
    const int64_t stride = in.integer();
    float *r_out = in.pointer<float>(), *rec = in.pointer<float>(), *sc = in.pointer<float>();
    const int B = in.i32(), T = in.i32();
    void* ws = in.pointer();
    const size_t nws = (size_t)in.integer();
    void* st = in.done() ? current_stream(in.bad) : nullptr;
    return call(in, [&] { return rm_action_expert_step(ctx, layers.data(), r_in, idx, cnt, stride, r_out, rec, sc, B, T, ws, nws, st); });
}

// (ctx, layers, L, r_in, idx, count, stride, r_out, records_out, record_scale, B, T, anchor_mode, y_anchor, h_anchor, h_stride,
//  out_gate, ws, ws_bytes)
RM_FN(step_ex) {
    Args in{args, n_args};
    rm_ctx* ctx = in.context();
    std::vector<void*> layers;
    in.layers(layers);
    float* r_in = in.pointer<float>();
    int32_t *idx = in.pointer<int32_t>(), *cnt = in.pointer<int32_t>();
    const int64_t stride = in.integer();
    float *r_out = in.pointer<float>(), *rec = in.pointer<float>(), *sc = in.pointer<float>();
    const int B = in.i32(), T = in.i32(), mode = in.i32();
    float *ya = in.pointer<float>(), *ha = in.pointer<float>();
    const int64_t hs = in.integer();
    float* gate = in.pointer<float>();
    void* ws = in.pointer();
    const size_t nws = (size_t)in.integer();
    void* st = in.done() ? current_stream(in.bad) : nullptr;
    return call(in, [&] {
        return rm_action_expert_step_ex(ctx, layers.data(), r_in, idx, cnt, stride, r_out, rec, sc, B, T, mode, ya, ha, hs, gate,
                                        ws, nws, st);
    });
}

// (ctx, layers, L, r_in_host, idx, count, stride, r_out_host, B, T, ws, ws_bytes)
RM_FN(step_host) {
    Args in{args, n_args};
    rm_ctx* ctx = in.context();
    std::vector<void*> layers;
    in.layers(layers);
    float* r_in = in.pointer<float>();
    int32_t *idx = in.pointer<int32_t>(), *cnt = in.pointer<int32_t>();
    const int64_t stride = in.integer();
    float* r_out = in.pointer<float>();
    const int B = in.i32(), T = in.i32();
    void* ws = in.pointer();
    const size_t nws = (size_t)in.integer();
    void* st = in.done() ? current_stream(in.bad) : nullptr;
    return call(in, [&] { return rm_action_expert_step_host(ctx, layers.data(), r_in, idx, cnt, stride, r_out, B, T, ws, nws, st); });
}

// (ctx, x, x_ref, P, score_out)
RM_FN(context_drift) {
    Args in{args, n_args};
    rm_ctx* ctx = in.context();
    void *x = in.pointer(), *xr = in.pointer();
    const int P = in.i32();
    float* score = in.pointer<float>();
    void* st = in.done() ? current_stream(in.bad) : nullptr;
    return call(in, [&] { return rm_context_drift(ctx, x, xr, P, score, st); });
}

// (ctx, Wg, Wu, Wd, x, rows, count, P, S, R_max, y_ref, y_out, ws, ws_bytes)
RM_FN(context_ffn) {
    Args in{args, n_args};
    rm_ctx* ctx = in.context();
    void *wg = in.pointer(), *wu = in.pointer(), *wd = in.pointer(), *x = in.pointer();
    int32_t *rows = in.pointer<int32_t>(), *cnt = in.pointer<int32_t>();
    const int P = in.i32(), S = in.i32(), R = in.i32();
    float *yr = in.pointer<float>(), *yo = in.pointer<float>();
    void* ws = in.pointer();
    const size_t nws = (size_t)in.integer();
    void* st = in.done() ? current_stream(in.bad) : nullptr;
    return call(in, [&] { return rm_context_ffn(ctx, wg, wu, wd, x, rows, cnt, P, S, R, yr, yo, ws, nws, st); });
}

PyObject* init(PyObject*, PyObject* const* args, Py_ssize_t n_args) {   // (torch._C._cuda_getDevice, torch._C._cuda_getCurrentRawStream)
    if (n_args != 2) {
        PyErr_SetString(PyExc_TypeError, "init takes two callables");
        return nullptr;
    }
    Py_XSETREF(g_get_device, Py_NewRef(args[0]));
    Py_XSETREF(g_raw_stream, Py_NewRef(args[1]));
    Py_RETURN_NONE;
}

#define RM_DEF(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)(void)>(name)), METH_FASTCALL, nullptr}
PyMethodDef g_methods[] = {RM_DEF(init), RM_DEF(mask_compact), RM_DEF(sparse_mlp), RM_DEF(sparse_mlp_static), RM_DEF(step),
                           RM_DEF(step_ex), RM_DEF(step_host), RM_DEF(context_drift), RM_DEF(context_ffn),
                           {nullptr, nullptr, 0, nullptr}};
PyModuleDef g_module = {PyModuleDef_HEAD_INIT, "_rmuscle", nullptr, -1, g_methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__rmuscle(void) {
    g_data_ptr = PyUnicode_InternFromString("data_ptr");
    return g_data_ptr ? PyModule_Create(&g_module) : nullptr;
}
