// CPython entry points of the library: argument conversion and the call, nothing else.
//
// One function template turns any function of sdverify.h into a Python callable by its C signature:
//   pointers   a CUDA tensor (contiguous), an address as int, or None (null; as the last argument, the
//              stream: the current stream of the current device)
//   size_t     a tensor (its size in bytes) or an int
// The same conversions through ctypes and torch's Python properties cost 5 us of an attention call's 12 and
// 10 us of the tail call's 16 (half of it torch.cuda.current_stream()): as long as the kernels of small
// problems run.  Here they take about 0.3 us.
#include <Python.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>
#include <utility>
#include "sdverify.h"

namespace {

struct Arg { PyObject* obj; bool is_stream; };

// address behind an argument; sets a Python error and returns false where it has none
bool address(const Arg& a, void** out) {
    if (THPVariable_Check(a.obj)) {
        const at::Tensor& t = THPVariable_Unpack(a.obj);
        if (!t.is_cuda() || !t.is_contiguous()) {
            PyErr_SetString(PyExc_AssertionError, "device tensors must be contiguous CUDA tensors");
            return false;
        }
        *out = t.data_ptr();
        return true;
    }
    if (a.obj == Py_None) {
        *out = a.is_stream ? static_cast<void*>(c10::cuda::getCurrentCUDAStream().stream()) : nullptr;
        return true;
    }
    PyObject* obj = a.obj;
    Py_INCREF(obj);
    if (!PyLong_Check(obj)) {                              // a torch stream, or anything else that has an address
        PyObject* got = a.is_stream ? PyObject_GetAttrString(obj, "cuda_stream") : PyObject_CallMethod(obj, "data_ptr", nullptr);
        Py_DECREF(obj);
        if (!got) return false;
        obj = got;
    }
    *out = PyLong_AsVoidPtr(obj);
    Py_DECREF(obj);
    return !(*out == nullptr && PyErr_Occurred());
}

template <typename T> struct Convert {                     // pointers
    static bool get(const Arg& a, T* out) {
        void* p = nullptr;
        if (!address(a, &p)) return false;
        *out = reinterpret_cast<T>(p);
        return true;
    }
};
template <> struct Convert<int32_t> {
    static bool get(const Arg& a, int32_t* out) {
        *out = static_cast<int32_t>(PyLong_AsLong(a.obj));
        return !PyErr_Occurred();
    }
};
template <> struct Convert<float> {
    static bool get(const Arg& a, float* out) {
        *out = static_cast<float>(PyFloat_AsDouble(a.obj));
        return !PyErr_Occurred();
    }
};
template <> struct Convert<size_t> {
    static bool get(const Arg& a, size_t* out) {
        if (THPVariable_Check(a.obj)) { *out = THPVariable_Unpack(a.obj).nbytes(); return true; }
        *out = PyLong_AsSize_t(a.obj);
        return !PyErr_Occurred();
    }
};

template <typename... A, size_t... I>
PyObject* invoke(sd_status (*fn)(A...), PyObject* const* args, std::index_sequence<I...>) {
    std::tuple<A...> v;
    if (!(Convert<A>::get(Arg{args[I], I + 1 == sizeof...(A)}, &std::get<I>(v)) && ...)) return nullptr;
    sd_status s;
    Py_BEGIN_ALLOW_THREADS
    s = fn(std::get<I>(v)...);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(s);
}

template <typename... A>
constexpr size_t arity(sd_status (*)(A...)) { return sizeof...(A); }
template <typename... A>
PyObject* dispatch(sd_status (*fn)(A...), PyObject* const* args) { return invoke(fn, args, std::index_sequence_for<A...>{}); }

template <auto Fn>
PyObject* call(PyObject*, PyObject* const* args, Py_ssize_t n) {
    if (n != static_cast<Py_ssize_t>(arity(Fn))) {
        PyErr_Format(PyExc_TypeError, "%zd arguments, %zu expected", n, arity(Fn));
        return nullptr;
    }
    try {
        return dispatch(Fn, args);
    } catch (const std::exception& e) {
        if (!PyErr_Occurred()) PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
}

#define SD_METHOD(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(&call<&name>)), METH_FASTCALL, nullptr}
PyMethodDef kMethods[] = {
    SD_METHOD(sd_tree_prepare), SD_METHOD(sd_verify_attention), SD_METHOD(sd_verify_attention_layers),
    SD_METHOD(sd_lmhead_argmax), SD_METHOD(sd_lmhead_argmax_static), SD_METHOD(sd_accept_tree), SD_METHOD(sd_compact_kv),
    SD_METHOD(sd_lmhead_accept_compact), SD_METHOD(sd_lmhead_stats), SD_METHOD(sd_lmhead_stats_logits),
    SD_METHOD(sd_accept_tree_sampled), SD_METHOD(sd_accept_chain_sampled), SD_METHOD(sd_accept_tree_sampled_q),
    SD_METHOD(sd_lmhead_accept_sampled_compact), SD_METHOD(sd_draft_feature_attention), {nullptr, nullptr, 0, nullptr}};

PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "_sdnative", nullptr, -1, kMethods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__sdnative(void) { return PyModule_Create(&kModule); }
