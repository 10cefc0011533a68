// Native argument marshalling of the Python binding: the calls that a program makes every step.  A
// decode step of a small batch is a few microseconds on the GPU, and turning eight tensors and six
// numbers into C arguments through ctypes took 9 us of Python per call; here it is well under one.
//
// Every function takes the arguments of the api.py function of the same name, in order.  It returns
// the status of the C entry point, or None when an argument is not of the plain expected kind (wrong
// type, device, layout; an explicit stream): api.py then takes its own path, which raises the error.
// The entry points are reached through the addresses that api.py took from the loaded library.
#include <Python.h>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "kda.h"

namespace {

decltype(&kda_decode_step) p_decode_step;
decltype(&kda_decode_multi) p_decode_multi;
decltype(&kda_layer_decode_step) p_layer_decode_step;
decltype(&kda_chunk_fwd) p_chunk_fwd;
decltype(&kda_layer_fwd) p_layer_fwd;
decltype(&kda_chunk_bwd) p_chunk_bwd;

// Takes the arguments one by one; ok turns false at the first that is not plain.
struct Args {
    PyObject* const* a;
    bool ok = true;

    void* tensor(at::ScalarType dtype, bool cuda = true, bool any = false) {
        PyObject* o = *a++;
        if (!ok || o == Py_None) return nullptr;
        if (THPVariable_Check(o)) {
            try {   // (a tensor without storage throws)
                const at::Tensor& t = THPVariable_Unpack(o);
                if (t.defined() && t.layout() == at::kStrided && t.is_cuda() == cuda && t.is_contiguous() &&
                    (any || t.scalar_type() == dtype))
                    return t.data_ptr();
            } catch (...) {
            }
        }
        ok = false;
        return nullptr;
    }
    float* f32() { return static_cast<float*>(tensor(at::kFloat)); }
    void* bf16() { return tensor(at::kBFloat16); }
    int32_t* i32(bool cuda = true) { return static_cast<int32_t*>(tensor(at::kInt, cuda)); }
    int64_t i64() {
        PyObject* o = *a++;
        if (!ok || !PyLong_CheckExact(o)) { ok = false; return 0; }
        int over = 0;
        const long long v = PyLong_AsLongLongAndOverflow(o, &over);
        if (over) ok = false;
        return v;
    }
    int i() {
        const int64_t v = i64();
        if (v != (int)v) ok = false;
        return (int)v;
    }
    float f() {
        PyObject* o = *a++;
        if (!ok || !PyFloat_CheckExact(o)) { ok = false; return 0.f; }
        return (float)PyFloat_AS_DOUBLE(o);
    }
    // workspace and workspace_bytes (None = the tensor's size)
    void* workspace(size_t& bytes) {
        PyObject* o = *a;
        void* p = tensor(at::kByte, true, true);
        if (!ok || !p) { ok = false; return nullptr; }
        if (*a == Py_None) {
            const at::Tensor& t = THPVariable_Unpack(o);
            bytes = (size_t)t.numel() * t.element_size();
            ++a;
        } else {
            bytes = (size_t)i64();
        }
        return p;
    }
    void* stream() {
        if (*a++ != Py_None) ok = false;
        if (!ok) return nullptr;
        try {   // (a machine without a GPU throws)
            return c10::cuda::getCurrentCUDAStream().stream();
        } catch (...) {
            ok = false;
            return nullptr;
        }
    }
};

// the element type that an argument `dt` further on names
at::ScalarType elem(PyObject* dt, bool& ok) {
    int over = 0;
    const long v = PyLong_CheckExact(dt) ? PyLong_AsLongAndOverflow(dt, &over) : -1;
    if (v != KDA_BF16 && v != KDA_F32) ok = false;
    return v == KDA_BF16 ? at::kBFloat16 : at::kFloat;
}

template <typename F>
PyObject* call(Args& A, F f) {
    if (!A.ok) Py_RETURN_NONE;
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = (int)f();
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}
#define EXPECT(n) if (nargs != (n)) Py_RETURN_NONE

PyObject* decode_step(PyObject*, PyObject* const* args, Py_ssize_t nargs) {
    EXPECT(15);
    Args A{args};
    const auto et = elem(args[13], A.ok);
    void* q = A.tensor(et); void* k = A.tensor(et); void* v = A.tensor(et);
    float* g = A.f32(); float* b = A.f32(); float* S = A.f32();
    int32_t* slot = A.i32();
    void* o = A.tensor(et);
    const int n = A.i(), H = A.i(), dk = A.i(), dv = A.i();
    const float scale = A.f();
    const int dt = A.i();
    void* st = A.stream();
    return call(A, [&] { return p_decode_step(q, k, v, g, b, S, slot, o, n, H, dk, dv, scale, (kda_dtype_t)dt, st); });
}

PyObject* decode_multi(PyObject*, PyObject* const* args, Py_ssize_t nargs) {
    EXPECT(16);
    Args A{args};
    const auto et = elem(args[14], A.ok);
    void* q = A.tensor(et); void* k = A.tensor(et); void* v = A.tensor(et);
    float* g = A.f32(); float* b = A.f32(); float* S = A.f32();
    int32_t* slot = A.i32();
    void* o = A.tensor(et);
    const int n = A.i(), tok = A.i(), H = A.i(), dk = A.i(), dv = A.i();
    const float scale = A.f();
    const int dt = A.i();
    void* st = A.stream();
    return call(A, [&] { return p_decode_multi(q, k, v, g, b, S, slot, o, n, tok, H, dk, dv, scale, (kda_dtype_t)dt, st); });
}

PyObject* layer_decode_step(PyObject*, PyObject* const* args, Py_ssize_t nargs) {
    EXPECT(20);
    Args A{args};
    void* q = A.bf16(); void* k = A.bf16(); void* v = A.bf16(); void* ga = A.bf16();
    float* b = A.f32();
    void* go = A.bf16();
    float* al = A.f32(); float* bias = A.f32(); float* w = A.f32();
    const float e1 = A.f(), e2 = A.f();
    float* S = A.f32();
    int32_t* slot = A.i32();
    void* y = A.bf16();
    const int n = A.i(), H = A.i(), dk = A.i(), dv = A.i();
    const float scale = A.f();
    void* st = A.stream();
    return call(A, [&] { return p_layer_decode_step(q, k, v, ga, b, go, al, bias, w, e1, e2, S, slot, y, n, H, dk, dv, scale, st); });
}

PyObject* chunk_fwd(PyObject*, PyObject* const* args, Py_ssize_t nargs) {
    EXPECT(21);
    Args A{args};
    const auto et = elem(args[17], A.ok);
    void* q = A.tensor(et); void* k = A.tensor(et); void* v = A.tensor(et);
    float* g = A.f32(); float* b = A.f32(); float* S0 = A.f32();
    void* o = A.tensor(et);
    float* S_T = A.f32();
    int32_t* cu = A.i32(); int32_t* cuh = A.i32(false);
    const int n = A.i();
    const int64_t T = A.i64();
    const int H = A.i(), dk = A.i(), dv = A.i(), chunk = A.i();
    const float scale = A.f();
    const int dt = A.i();
    size_t bytes = 0;
    void* ws = A.workspace(bytes);
    void* st = A.stream();
    return call(A, [&] {
        return p_chunk_fwd(q, k, v, g, b, S0, o, S_T, cu, cuh, n, T, H, dk, dv, chunk, scale, (kda_dtype_t)dt, ws, bytes, st);
    });
}

PyObject* layer_fwd(PyObject*, PyObject* const* args, Py_ssize_t nargs) {
    EXPECT(26);
    Args A{args};
    void* q = A.bf16(); void* k = A.bf16(); void* v = A.bf16(); void* ga = A.bf16();
    float* b = A.f32();
    void* go = A.bf16();
    float* al = A.f32(); float* bias = A.f32(); float* w = A.f32();
    const float e1 = A.f(), e2 = A.f();
    float* S0 = A.f32();
    void* y = A.bf16();
    float* S_T = A.f32();
    int32_t* cu = A.i32(); int32_t* cuh = A.i32(false);
    const int n = A.i();
    const int64_t T = A.i64();
    const int H = A.i(), dk = A.i(), dv = A.i(), chunk = A.i();
    const float scale = A.f();
    size_t bytes = 0;
    void* ws = A.workspace(bytes);
    void* st = A.stream();
    return call(A, [&] {
        return p_layer_fwd(q, k, v, ga, b, go, al, bias, w, e1, e2, S0, y, S_T, cu, cuh, n, T, H, dk, dv, chunk, scale, ws, bytes, st);
    });
}

PyObject* chunk_bwd(PyObject*, PyObject* const* args, Py_ssize_t nargs) {
    EXPECT(27);
    Args A{args};
    const auto et = elem(args[23], A.ok);
    void* q = A.tensor(et); void* k = A.tensor(et); void* v = A.tensor(et);
    float* g = A.f32(); float* b = A.f32(); float* S0 = A.f32();
    void* d_o = A.tensor(et);
    float* dST = A.f32();
    float* dq = A.f32(); float* dkk = A.f32(); float* dvv = A.f32(); float* dg = A.f32(); float* db = A.f32(); float* dS0 = A.f32();
    int32_t* cu = A.i32(); int32_t* cuh = A.i32(false);
    const int n = A.i();
    const int64_t T = A.i64();
    const int H = A.i(), dk = A.i(), dv = A.i(), chunk = A.i();
    const float scale = A.f();
    const int dt = A.i();
    size_t bytes = 0;
    void* ws = A.workspace(bytes);
    void* st = A.stream();
    return call(A, [&] {
        return p_chunk_bwd(q, k, v, g, b, S0, d_o, dST, dq, dkk, dvv, dg, db, dS0, cu, cuh, n, T, H, dk, dv, chunk, scale,
                           (kda_dtype_t)dt, ws, bytes, st);
    });
}

// bind(kda_decode_step, kda_decode_multi, kda_layer_decode_step, kda_chunk_fwd, kda_layer_fwd, kda_chunk_bwd): addresses
PyObject* bind(PyObject*, PyObject* const* args, Py_ssize_t nargs) {
    void* p[6];
    if (nargs != 6) { PyErr_SetString(PyExc_TypeError, "bind takes six addresses"); return nullptr; }
    for (int i = 0; i < 6; ++i) {
        p[i] = PyLong_AsVoidPtr(args[i]);
        if (!p[i]) {
            if (!PyErr_Occurred()) PyErr_SetString(PyExc_ValueError, "NULL address");
            return nullptr;
        }
    }
    p_decode_step = reinterpret_cast<decltype(p_decode_step)>(p[0]);
    p_decode_multi = reinterpret_cast<decltype(p_decode_multi)>(p[1]);
    p_layer_decode_step = reinterpret_cast<decltype(p_layer_decode_step)>(p[2]);
    p_chunk_fwd = reinterpret_cast<decltype(p_chunk_fwd)>(p[3]);
    p_layer_fwd = reinterpret_cast<decltype(p_layer_fwd)>(p[4]);
    p_chunk_bwd = reinterpret_cast<decltype(p_chunk_bwd)>(p[5]);
    Py_RETURN_NONE;
}

#define FN(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(name)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {FN(bind), FN(decode_step), FN(decode_multi), FN(layer_decode_step), FN(chunk_fwd), FN(layer_fwd),
                         FN(chunk_bwd), {nullptr, nullptr, 0, nullptr}};
// (build.py and api.py look for this text in the file: torch's C++ interface changes from version to version)
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_marshal", KDA_BUILT_FOR, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__marshal() { return PyModule_Create(&module); }
