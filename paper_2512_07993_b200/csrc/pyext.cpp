// Python entry points of the C ABI as a CPython extension: argument marshalling only.
//
// A decode step of a small cache takes the GPU a few microseconds, and the program that issues it is a Python loop over
// layers.  Marshalling 25 tensor arguments through ctypes (four attribute reads and one pointer object each) took 14.7 us
// per skipkv_decode_step call and bounded that loop; here a call is one vectorcall that unpacks the tensors in place.
// Every function is generated from the prototype in skipkv.h: the parameter's C type decides what is accepted
//   const skipkv_shape* / const skipkv_params*   the ctypes structures of binding.py (read through the buffer protocol)
//   int32_t*, float*, uint8_t*, uint32_t*        contiguous device tensor of that type (uint32_t: int32), or None
//   void*                                        contiguous bfloat16 device tensor, or None
//   int32_t, float                               numbers
// and the trailing void* parameters are the workspace (any type) and the stream (None: the current stream).
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/core/Tensor.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <tuple>
#include <type_traits>
#include <utility>

#include "skipkv.h"

namespace {

bool fail_value(const char* msg) {
    PyErr_SetString(PyExc_ValueError, msg);
    return false;
}

// device pointer of a tensor argument; want == Undefined accepts every type
bool tensor_ptr(PyObject* o, at::ScalarType want, void** out) {
    if (o == Py_None) { *out = nullptr; return true; }
    if (!THPVariable_Check(o)) {
        PyErr_Format(PyExc_TypeError, "device-resident contiguous tensor expected, got %.80s", Py_TYPE(o)->tp_name);
        return false;
    }
    const at::Tensor& t = THPVariable_Unpack(o);
    if (!t.is_cuda() || !t.is_contiguous()) return fail_value("device-resident contiguous tensor expected");
    if (want != at::ScalarType::Undefined && t.scalar_type() != want) {
        PyErr_Format(PyExc_ValueError, "expected torch.%s, got torch.%s", c10::toString(want), c10::toString(t.scalar_type()));
        return false;
    }
    *out = t.data_ptr();
    return true;
}

template <typename T> struct ScalarOf { static constexpr at::ScalarType value = at::ScalarType::BFloat16; };   // void*
template <> struct ScalarOf<int32_t> { static constexpr at::ScalarType value = at::ScalarType::Int; };
template <> struct ScalarOf<uint32_t> { static constexpr at::ScalarType value = at::ScalarType::Int; };
template <> struct ScalarOf<float> { static constexpr at::ScalarType value = at::ScalarType::Float; };
template <> struct ScalarOf<uint8_t> { static constexpr at::ScalarType value = at::ScalarType::Byte; };

template <typename S>
bool struct_ptr(PyObject* o, const S** out) {
    Py_buffer view;
    if (PyObject_GetBuffer(o, &view, PyBUF_SIMPLE) != 0) return false;
    *out = static_cast<const S*>(view.buf);
    const bool ok = view.len == Py_ssize_t(sizeof(S));
    PyBuffer_Release(&view);                              // the caller's structure outlives the call
    return ok || fail_value("structure of another size");
}

template <typename T, bool kRaw>
bool convert(PyObject* o, T& out) {
    if constexpr (std::is_same_v<T, const skipkv_shape*> || std::is_same_v<T, const skipkv_params*>) {
        return struct_ptr(o, &out);
    } else if constexpr (std::is_pointer_v<T>) {
        using E = std::remove_const_t<std::remove_pointer_t<T>>;
        void* p = nullptr;
        if (!tensor_ptr(o, kRaw ? at::ScalarType::Undefined : ScalarOf<E>::value, &p)) return false;
        out = static_cast<T>(p);
        return true;
    } else if constexpr (std::is_same_v<T, float>) {
        const double v = PyFloat_AsDouble(o);
        out = float(v);
        return !(v == -1.0 && PyErr_Occurred());
    } else {
        static_assert(std::is_same_v<T, int32_t>, "unknown parameter type");
        const unsigned long long v = PyLong_AsUnsignedLongLongMask(o);
        out = int32_t(uint32_t(v));
        return !(v == ~0ull && PyErr_Occurred());
    }
}

bool stream_ptr(PyObject* o, void** out) {
    if (o == Py_None) {
        *out = c10::cuda::getCurrentCUDAStream().stream();
        return true;
    }
    PyObject* h = PyObject_GetAttrString(o, "cuda_stream");
    if (!h) return false;
    const unsigned long long v = PyLong_AsUnsignedLongLongMask(h);
    Py_DECREF(h);
    if (v == ~0ull && PyErr_Occurred()) return false;
    *out = reinterpret_cast<void*>(v);
    return true;
}

template <auto kFn, bool kWs, typename... A, size_t... I>
PyObject* invoke(int (*)(A...), std::index_sequence<I...>, PyObject* const* args, Py_ssize_t nargs) {
    constexpr size_t n = sizeof...(A);                    // the stream is the last parameter, the workspace (if any) the one before
    if (nargs != Py_ssize_t(n)) {
        PyErr_Format(PyExc_TypeError, "%zd arguments expected, got %zd", Py_ssize_t(n), nargs);
        return nullptr;
    }
    std::tuple<std::remove_cv_t<A>...> v{};
    void* stream = nullptr;
    const bool ok = ([&] {
        if constexpr (I + 1 == n) {
            return stream_ptr(args[I], &stream);
        } else {
            return convert<std::tuple_element_t<I, decltype(v)>, kWs && I + 2 == n>(args[I], std::get<I>(v));
        }
    }() && ...);
    if (!ok) return nullptr;
    std::get<n - 1>(v) = stream;
    return PyLong_FromLong(kFn(std::get<I>(v)...));
}

template <typename F> struct Arity;
template <typename... A> struct Arity<int (*)(A...)> { static constexpr size_t value = sizeof...(A); };

template <auto kFn, bool kWs = true>
PyObject* entry(PyObject*, PyObject* const* args, Py_ssize_t nargs) {
    try {
        return invoke<kFn, kWs>(kFn, std::make_index_sequence<Arity<decltype(kFn)>::value>{}, args, nargs);
    } catch (const std::exception& e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
}

#define ENTRY(name, ...) {#name, reinterpret_cast<PyCFunction>(&entry<&name, ##__VA_ARGS__>), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {
    ENTRY(skipkv_score), ENTRY(skipkv_score_table), ENTRY(skipkv_score_paged), ENTRY(skipkv_select), ENTRY(skipkv_select_fill),
    ENTRY(skipkv_select_fill_red), ENTRY(skipkv_compact), ENTRY(skipkv_compact_fill), ENTRY(skipkv_compact_paged),
    ENTRY(skipkv_token_redundancy), ENTRY(skipkv_decode_attn), ENTRY(skipkv_decode_attn_paged), ENTRY(skipkv_decode_step),
    ENTRY(skipkv_decode_step_paged), ENTRY(skipkv_append), ENTRY(skipkv_append_step), ENTRY(skipkv_decode_attn_static, false),
    ENTRY(skipkv_table_step, false), ENTRY(skipkv_steer, false),
    {nullptr, nullptr, 0, nullptr}};
#undef ENTRY

PyModuleDef module_def = {PyModuleDef_HEAD_INIT, "_native", "Marshalling of the SkipKV C ABI.", -1, methods,
                          nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native(void) {
    PyObject* m = PyModule_Create(&module_def);
    if (m && PyModule_AddStringConstant(m, "built_for", SKIPKV_BUILT_FOR) < 0) Py_CLEAR(m);      // the caller compares it with what runs
    return m;
}
