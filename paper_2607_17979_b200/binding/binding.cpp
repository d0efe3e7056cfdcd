// Native side of the Python binding for the calls of a serving loop: checks the tensors, reads
// sizes, device pointers and the current stream, and calls the C entry point of the same name.
//
// What bounds a small decode step or a short prompt is the host: marshalled in Python (dtype,
// contiguity and device checks, ctypes conversions, current_stream()), a decode call took 11.9 us
// while its kernel takes 2.0 us.  Here the checks are a few loads from the tensor objects.
// Errors are the same types and texts the Python marshalling raises (api.py).
#include <Python.h>

#include <array>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/gdn.h"

namespace {

// A failed check: the Python error is already set.
struct Failed {};

const at::Tensor* tensor(PyObject* obj) {
    return THPVariable_Check(obj) ? &THPVariable_Unpack(obj) : nullptr;
}

// Device pointer of a contiguous CUDA tensor of the given type; null for an optional None.
template <class T> T* dev(PyObject* obj, at::ScalarType type, const char* name, bool optional = false) {
    if (obj == Py_None) {
        if (optional) return nullptr;
        PyErr_Format(PyExc_TypeError, "%s is required", name);
        throw Failed();
    }
    const at::Tensor* t = tensor(obj);
    if (!t || !t->is_cuda() || t->scalar_type() != type || !t->is_contiguous()) {
        PyErr_Format(PyExc_TypeError, "%s must be a contiguous CUDA tensor of dtype torch.%s", name,
                     type == at::kBFloat16 ? "bfloat16" : type == at::kFloat ? "float32"
                     : type == at::kInt    ? "int32"
                                           : "uint8");
        throw Failed();
    }
    return static_cast<T*>(t->data_ptr());
}
void* bf16(PyObject* o, const char* name) { return dev<void>(o, at::kBFloat16, name); }
float* f32(PyObject* o, const char* name, bool opt = false) { return dev<float>(o, at::kFloat, name, opt); }
int32_t* i32(PyObject* o, const char* name, bool opt = false) { return dev<int32_t>(o, at::kInt, name, opt); }

// `obj.shape` of a tensor that must have N dimensions (as unpacking it into N names would check).  A copy:
// the tensor's own array may be changed by another thread while the call runs without the interpreter lock.
template <int N> std::array<int32_t, N> shape(PyObject* obj) {
    const at::Tensor* t = tensor(obj);
    if (!t) {
        PyObject* s = PyObject_GetAttrString(obj, "shape");       // AttributeError for what has none
        if (s) {
            Py_DECREF(s);
            PyErr_SetString(PyExc_TypeError, "arguments must be torch tensors");
        }
        throw Failed();
    }
    const int64_t d = t->dim();
    if (d < N)
        PyErr_Format(PyExc_ValueError, "not enough values to unpack (expected %d, got %lld)", N, (long long)d);
    if (d > N) PyErr_Format(PyExc_ValueError, "too many values to unpack (expected %d)", N);
    if (d != N) throw Failed();
    const at::IntArrayRef now = t->sizes();
    std::array<int32_t, N> sizes;
    for (int i = 0; i < N; ++i) sizes[i] = static_cast<int32_t>(now[i]);
    return sizes;
}
int64_t rows(PyObject* obj) {
    const at::Tensor* t = tensor(obj);
    if (!t) shape<1>(obj);
    if (t->dim() == 0) {
        PyErr_SetString(PyExc_IndexError, "tuple index out of range");
        throw Failed();
    }
    return t->size(0);
}

float as_float(PyObject* o) {
    if (PyFloat_CheckExact(o)) return static_cast<float>(PyFloat_AS_DOUBLE(o));
    PyObject* f = PyNumber_Float(o);
    if (!f) throw Failed();
    const double v = PyFloat_AS_DOUBLE(f);
    Py_DECREF(f);
    return static_cast<float>(v);
}
int32_t as_int(PyObject* o) {
    PyObject* i = PyLong_CheckExact(o) ? Py_NewRef(o) : PyNumber_Long(o);
    if (!i) throw Failed();
    const long long v = PyLong_AsLongLong(i);
    Py_DECREF(i);
    if (v == -1 && PyErr_Occurred()) throw Failed();
    return static_cast<int32_t>(v);
}

void* stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

// The body of every function below: C++ exceptions become Python errors, the status code is the
// result, and other Python threads run while the call is made.
template <class F> PyObject* guarded(Py_ssize_t n, Py_ssize_t want, F body) {
    if (n != want) {
        PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, n);
        return nullptr;
    }
    try {
        return PyLong_FromLong(body());
    } catch (const Failed&) {
    } catch (const std::exception& e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
    }
    return nullptr;
}
template <class F> int unlocked(F call) {
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = call();
    Py_END_ALLOW_THREADS
    return rc;
}

// decode(q, k, v, g, beta, state_pool, slot_idx, o, scale, dev_status)
PyObject* decode(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(n, 10, [&] {
        const auto qs = shape<3>(a[0]), vs = shape<3>(a[2]);
        const void *q = bf16(a[0], "q"), *k = bf16(a[1], "k"), *v = bf16(a[2], "v");
        const float *g = f32(a[3], "g"), *beta = f32(a[4], "beta");
        float* pool = f32(a[5], "state_pool");
        const int32_t* slot = i32(a[6], "slot_idx", true);
        void* o = bf16(a[7], "o");
        const int32_t slots = rows(a[5]);
        const float scale = as_float(a[8]);
        int32_t* status = i32(a[9], "dev_status", true);
        void* st = stream();
        return unlocked([&] {
            return gdn_decode(q, k, v, g, beta, pool, slot, o, qs[0], qs[1], vs[1], qs[2], vs[2], slots, scale,
                              status, st);
        });
    });
}

// decode_multi(q, k, v, g, beta, state_pool, slot_idx, o, scale, state_layout, dev_status)
PyObject* decode_multi(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(n, 11, [&] {
        const auto qs = shape<4>(a[0]), vs = shape<4>(a[2]);
        const void *q = bf16(a[0], "q"), *k = bf16(a[1], "k"), *v = bf16(a[2], "v");
        const float *g = f32(a[3], "g"), *beta = f32(a[4], "beta");
        float* pool = f32(a[5], "state_pool");
        const int32_t* slot = i32(a[6], "slot_idx", true);
        void* o = bf16(a[7], "o");
        const int32_t slots = rows(a[5]);
        const float scale = as_float(a[8]);
        const int32_t layout = as_int(a[9]);
        int32_t* status = i32(a[10], "dev_status", true);
        void* st = stream();
        return unlocked([&] {
            return gdn_decode_multi(q, k, v, g, beta, pool, slot, o, qs[0], qs[1], qs[2], vs[2], qs[3], vs[3],
                                    slots, scale, layout, status, st);
        });
    });
}

// gate(a, b, A_log, dt_bias, g, beta)
PyObject* gate(PyObject*, PyObject* const* x, Py_ssize_t n) {
    return guarded(n, 6, [&] {
        const auto s = shape<2>(x[0]);
        const void *a = bf16(x[0], "a"), *b = bf16(x[1], "b");
        const float *A_log = f32(x[2], "A_log"), *dt_bias = f32(x[3], "dt_bias");
        float *g = f32(x[4], "g"), *beta = f32(x[5], "beta");
        void* st = stream();
        return unlocked([&] { return gdn_gate(a, b, A_log, dt_bias, g, beta, s[0], s[1], st); });
    });
}

// prefill(route, q, k, v, g, beta, cu_seqlens, init_state, final_state, slot_idx, o, scale, workspace,
//         max_seqlen_hint, chunk, dev_status, split_permille); route as GDN_ROUTE_*, 0 = gdn_prefill
PyObject* prefill(PyObject*, PyObject* const* args, Py_ssize_t n) {
    return guarded(n, 17, [&] {
        const int32_t route = as_int(args[0]);
        PyObject* const* a = args + 1;
        const auto qs = shape<3>(a[0]), vs = shape<3>(a[2]);
        const int32_t N = static_cast<int32_t>(rows(a[5])) - 1;
        const int32_t split = route == GDN_ROUTE_OVERLAP ? as_int(a[15]) : 0;
        const void *q = bf16(a[0], "q"), *k = bf16(a[1], "k"), *v = bf16(a[2], "v");
        const float *g = f32(a[3], "g"), *beta = f32(a[4], "beta");
        const int32_t* cu = i32(a[5], "cu_seqlens");
        const float* init = f32(a[6], "init_state", true);
        float* final_state = f32(a[7], "final_state");
        const int32_t* slot = i32(a[8], "slot_idx", true);
        void* o = bf16(a[9], "o");
        const int32_t hint = as_int(a[12]), chunk = as_int(a[13]);
        const int32_t slots = rows(a[7]);
        const float scale = as_float(a[10]);
        void* ws = dev<void>(a[11], at::kByte, "workspace");
        const size_t ws_bytes = static_cast<size_t>(tensor(a[11])->numel());
        int32_t* status = i32(a[14], "dev_status", true);
        void* st = stream();
        return unlocked([&] {
            if (route == GDN_ROUTE_OVERLAP)
                return gdn_prefill_overlap(q, k, v, g, beta, cu, init, final_state, slot, o, qs[0], N, hint, qs[1],
                                           vs[1], qs[2], vs[2], chunk, slots, scale, ws, ws_bytes, status, st, split);
            const auto fn = route == GDN_ROUTE_CHUNKED  ? gdn_prefill_chunked
                            : route == GDN_ROUTE_FUSED  ? gdn_prefill_fused
                            : route == GDN_ROUTE_STREAM ? gdn_prefill_stream
                                                        : gdn_prefill;
            return fn(q, k, v, g, beta, cu, init, final_state, slot, o, qs[0], N, hint, qs[1], vs[1], qs[2], vs[2],
                      chunk, slots, scale, ws, ws_bytes, status, st);
        });
    });
}

#define GDN_FASTCALL(f) reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)(void)>(f)), METH_FASTCALL
PyMethodDef methods[] = {
    {"decode", GDN_FASTCALL(decode), "gdn_decode"},
    {"decode_multi", GDN_FASTCALL(decode_multi), "gdn_decode_multi"},
    {"gate", GDN_FASTCALL(gate), "gdn_gate"},
    {"prefill", GDN_FASTCALL(prefill), "gdn_prefill and its routes"},
    {nullptr, nullptr, 0, nullptr},
};
#ifndef GDN_BINDING_KEY
#define GDN_BINDING_KEY ""
#endif
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_binding", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__binding(void) {
    PyObject* m = PyModule_Create(&module);
    // what it was built for, which build.py also looks for in the file
    if (m && PyModule_AddStringConstant(m, "built_for", GDN_BINDING_KEY) < 0) {
        Py_DECREF(m);
        return nullptr;
    }
    return m;
}
