// The calls of binding.py that enqueue work on device tensors, as a Python extension module: argument marshalling only.
//
// Why native.  A decode-sized call is ~20 us of GPU time behind three launches; through ctypes its host side took 24 us
// (stream lookup 3.4, three output tensors 7, argument conversion 4, the C call 8.5), which then was what a caller waited
// for.  Here the marshalling is ~1 us and the outputs ~1 us each.
//
// The module does not link the library: bind() is given the addresses of its functions, so that whichever build of it
// binding.py has loaded is the one called.  The GIL is released around every call, as ctypes does.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/ops/empty.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include <stdint.h>

#include "../../include/more_route.h"

namespace {

decltype(&more_route_ex) g_route_ex;
decltype(&more_route_psum) g_psum;
decltype(&more_dispatch) g_dispatch;
decltype(&more_route_full) g_full;
decltype(&more_merge_shards) g_merge;

struct Error {};                    // a Python exception is set

const at::Tensor& tensor(PyObject* o)
{
    if (!THPVariable_Check(o)) {
        PyErr_Format(PyExc_TypeError, "expected a tensor, got %s", Py_TYPE(o)->tp_name);
        throw Error();
    }
    return THPVariable_Unpack(o);
}
void* ptr(PyObject* o) { return o == Py_None ? nullptr : const_cast<void*>(tensor(o).const_data_ptr()); }

int integer(PyObject* o)
{
    const long v = PyLong_AsLong(o);
    if (v == -1 && PyErr_Occurred()) throw Error();
    if (v < INT32_MIN || v > INT32_MAX) {
        PyErr_SetString(PyExc_OverflowError, "argument does not fit in 32 bits");
        throw Error();
    }
    return (int)v;
}
int size(const at::Tensor& t, int dims, int d)
{
    if (t.dim() != dims) {
        PyErr_Format(PyExc_ValueError, "expected a tensor of %d dimensions, got %d", dims, (int)t.dim());
        throw Error();
    }
    return (int)t.size(d);
}
// None: torch's current stream of the current device
void* stream(PyObject* o)
{
    if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
    PyObject* v = PyObject_GetAttrString(o, "cuda_stream");
    if (!v) throw Error();
    void* s = PyLong_AsVoidPtr(v);
    Py_DECREF(v);
    if (!s && PyErr_Occurred()) throw Error();
    return s;
}
void expect(Py_ssize_t n, Py_ssize_t want)
{
    if (n != want) {
        PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, n);
        throw Error();
    }
}

template <class F>
PyObject* guarded(F body)
{
    HANDLE_TH_ERRORS
    try {
        return body();
    } catch (const Error&) {
        return nullptr;
    }
    END_HANDLE_TH_ERRORS
}

template <class F>
int released(F call)
{
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = call();
    Py_END_ALLOW_THREADS
    return rc;
}

int route_ex(PyObject* const* a, int k, int mode, void* idx, void* gate, void* counts, void* topval, void* lse, int path, int msplit,
             void* st)
{
    const at::Tensor &X = tensor(a[0]), &R2 = tensor(a[2]);
    void* r1 = ptr(a[1]);
    const int T = size(X, 2, 0), h = size(X, 2, 1), r = size(R2, 2, 0), M = size(R2, 2, 1);
    const void *x = X.const_data_ptr(), *r2 = R2.const_data_ptr();
    return released([&] {
        return g_route_ex(x, r1, r2, T, h, r, M, k, mode, static_cast<int32_t*>(idx), static_cast<float*>(gate),
                          static_cast<int32_t*>(counts), static_cast<float*>(topval), static_cast<float*>(lse), path, msplit, st);
    });
}

// bind(route_ex, psum, dispatch, full, merge): addresses of the library's functions
PyObject* py_bind(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    return guarded([&]() -> PyObject* {
        expect(n, 5);
        void* f[5];
        for (int i = 0; i < 5; ++i)
            if (!(f[i] = PyLong_AsVoidPtr(a[i]))) {
                if (!PyErr_Occurred()) PyErr_SetString(PyExc_ValueError, "null function address");
                throw Error();
            }
        g_route_ex = reinterpret_cast<decltype(g_route_ex)>(f[0]);
        g_psum = reinterpret_cast<decltype(g_psum)>(f[1]);
        g_dispatch = reinterpret_cast<decltype(g_dispatch)>(f[2]);
        g_full = reinterpret_cast<decltype(g_full)>(f[3]);
        g_merge = reinterpret_cast<decltype(g_merge)>(f[4]);
        Py_RETURN_NONE;
    });
}

// route_ex(X, R1, R2, k, gate_mode, idx, gate, counts, topval, lse, path, msplit, stream) -> rc
PyObject* py_route_ex(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    return guarded([&]() -> PyObject* {
        expect(n, 13);
        return PyLong_FromLong(route_ex(a, integer(a[3]), integer(a[4]), ptr(a[5]), ptr(a[6]), ptr(a[7]), ptr(a[8]), ptr(a[9]),
                                        integer(a[10]), integer(a[11]), stream(a[12])));
    });
}

// route(X, R1, R2, k, gate_mode, want_topval, want_lse, path, msplit, stream) -> (rc, idx, gate, counts, topval, lse)
PyObject* py_route(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    return guarded([&]() -> PyObject* {
        expect(n, 10);
        const at::Tensor &X = tensor(a[0]), &R2 = tensor(a[2]);
        const int64_t T = size(X, 2, 0), M = size(R2, 2, 1);
        const int k = integer(a[3]);
        const bool want_topval = PyObject_IsTrue(a[5]) == 1, want_lse = PyObject_IsTrue(a[6]) == 1;
        const auto f32 = at::TensorOptions().device(X.device()).dtype(at::kFloat), i32 = f32.dtype(at::kInt);
        at::Tensor idx = at::empty({T, k}, i32), gate = at::empty({T, k}, f32), counts = at::empty({M}, i32), topval, lse;
        if (want_topval) topval = at::empty({T, k}, f32);
        if (want_lse) lse = at::empty({T}, f32);
        const int rc = route_ex(a, k, integer(a[4]), idx.data_ptr(), gate.data_ptr(), counts.data_ptr(),
                                want_topval ? topval.data_ptr() : nullptr, want_lse ? lse.data_ptr() : nullptr, integer(a[7]),
                                integer(a[8]), stream(a[9]));
        // (an undefined tensor is wrapped as None)
        return Py_BuildValue("(iNNNNN)", rc, THPVariable_Wrap(idx), THPVariable_Wrap(gate), THPVariable_Wrap(counts),
                             THPVariable_Wrap(topval), THPVariable_Wrap(lse));
    });
}

// psum(X, R1, R2, lse, out, path, stream) -> rc
PyObject* py_psum(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    return guarded([&]() -> PyObject* {
        expect(n, 7);
        const at::Tensor &X = tensor(a[0]), &R2 = tensor(a[2]);
        const int T = size(X, 2, 0), h = size(X, 2, 1), r = size(R2, 2, 0), M = size(R2, 2, 1), path = integer(a[5]);
        void *r1 = ptr(a[1]), *lse = ptr(a[3]), *out = ptr(a[4]), *st = stream(a[6]);
        return PyLong_FromLong(released([&] {
            return g_psum(X.const_data_ptr(), r1, R2.const_data_ptr(), T, h, r, M, static_cast<const float*>(lse),
                          static_cast<float*>(out), path, st);
        }));
    });
}

// dispatch(idx, counts, offsets, pairs, stream) -> rc
PyObject* py_dispatch(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    return guarded([&]() -> PyObject* {
        expect(n, 5);
        const at::Tensor &idx = tensor(a[0]), &counts = tensor(a[1]);
        const int T = size(idx, 2, 0), k = size(idx, 2, 1), M = counts.dim() > 0 ? (int)counts.size(0) : size(counts, 1, 0);
        void *off = ptr(a[2]), *pairs = ptr(a[3]), *st = stream(a[4]);
        return PyLong_FromLong(released([&] {
            return g_dispatch(static_cast<const int32_t*>(idx.const_data_ptr()), static_cast<const int32_t*>(counts.const_data_ptr()), T,
                              k, M, static_cast<int32_t*>(off), static_cast<int32_t*>(pairs), st);
        }));
    });
}

// full(X, W, k, gate_mode, idx, gate, counts, topval, lse, msplit, stream) -> rc
PyObject* py_full(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    return guarded([&]() -> PyObject* {
        expect(n, 11);
        const at::Tensor &X = tensor(a[0]), &Wt = tensor(a[1]);
        const int T = size(X, 2, 0), h = size(X, 2, 1), M = size(Wt, 2, 1), k = integer(a[2]), mode = integer(a[3]);
        void *idx = ptr(a[4]), *gate = ptr(a[5]), *counts = ptr(a[6]), *topval = ptr(a[7]), *lse = ptr(a[8]);
        const int msplit = integer(a[9]);
        void* st = stream(a[10]);
        return PyLong_FromLong(released([&] {
            return g_full(X.const_data_ptr(), Wt.const_data_ptr(), T, h, M, k, mode, static_cast<int32_t*>(idx), static_cast<float*>(gate),
                          static_cast<int32_t*>(counts), static_cast<float*>(topval), static_cast<float*>(lse), msplit, st);
        }));
    });
}

// merge(idx, topval, lse, shard_base, M, gate_mode, out_idx, out_gate, counts, out_topval, out_lse, stream) -> rc
PyObject* py_merge(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    return guarded([&]() -> PyObject* {
        expect(n, 12);
        const at::Tensor& idx = tensor(a[0]);
        const int S = size(idx, 3, 0), T = size(idx, 3, 1), k = size(idx, 3, 2);
        int32_t base[MORE_MERGE_MAX_SHARDS];
        const bool based = a[3] != Py_None;
        if (based && S <= MORE_MERGE_MAX_SHARDS) {           // (more shards than that: the library refuses the call)
            PyObject* seq = PySequence_Fast(a[3], "shard_base is a sequence of integers");
            if (!seq) throw Error();
            const Py_ssize_t count = PySequence_Fast_GET_SIZE(seq);
            if (count != S) {
                Py_DECREF(seq);
                PyErr_Format(PyExc_IndexError, "shard_base has %zd entries for %d shards", count, S);
                throw Error();
            }
            for (int s = 0; s < S; ++s) {
                PyObject* v = PyNumber_Long(PySequence_Fast_GET_ITEM(seq, s));
                const long b = v ? PyLong_AsLong(v) : -1;
                Py_XDECREF(v);
                if (b == -1 && PyErr_Occurred()) {
                    Py_DECREF(seq);
                    throw Error();
                }
                base[s] = (int32_t)b;
            }
            Py_DECREF(seq);
        }
        const int M = integer(a[4]), mode = integer(a[5]);
        void *val = ptr(a[1]), *lse = ptr(a[2]), *oi = ptr(a[6]), *og = ptr(a[7]), *oc = ptr(a[8]), *ov = ptr(a[9]), *ol = ptr(a[10]);
        void* st = stream(a[11]);
        return PyLong_FromLong(released([&] {
            return g_merge(static_cast<const int32_t*>(idx.const_data_ptr()), static_cast<const float*>(val), static_cast<const float*>(lse),
                           based ? base : nullptr, S, T, k, M, mode, static_cast<int32_t*>(oi), static_cast<float*>(og),
                           static_cast<float*>(ov), static_cast<float*>(ol), static_cast<int32_t*>(oc), st);
        }));
    });
}

#define MORE_FAST(name, f) {name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(f)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {
    MORE_FAST("bind", py_bind), MORE_FAST("route", py_route), MORE_FAST("route_ex", py_route_ex), MORE_FAST("psum", py_psum),
    MORE_FAST("dispatch", py_dispatch), MORE_FAST("full", py_full), MORE_FAST("merge", py_merge), {nullptr, nullptr, 0, nullptr}};
// (the text by which build.py tells whether the module fits the torch and the Python that are installed)
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_more_binding", "built for " MORE_BUILT_FOR ";", -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__more_binding() { return PyModule_Create(&module); }
