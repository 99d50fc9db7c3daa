// Argument marshalling of the stream-ordered entry points for Python: tensors to pointers, numbers to C numbers, the
// current stream appended, nothing else.  A whole model's verification pass is 66 calls; through ctypes, with every argument
// wrapped by Python code, a call took 13 us of host time, more than its kernels (measured at 32 heads and 1.5k keys).
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>
#include <ATen/core/Tensor.h>
#include <c10/cuda/CUDAStream.h>

#include <tuple>
#include <type_traits>
#include <utility>

#include "goose.h"

namespace {

template <typename T>
bool convert(PyObject* o, T& v) {
    if constexpr (std::is_same_v<T, goose_ctx*>) {
        v = o == Py_None ? nullptr : static_cast<T>(PyLong_AsVoidPtr(o));
    } else if constexpr (std::is_pointer_v<T>) {
        if (o == Py_None) v = nullptr;
        else if (THPVariable_Check(o)) {
            // what the library writes is asked for as such: a copy-on-write tensor gets memory of its own then
            const at::Tensor& t = THPVariable_Unpack(o);
            if constexpr (std::is_const_v<std::remove_pointer_t<T>>) v = static_cast<T>(t.const_data_ptr());
            else v = static_cast<T>(t.mutable_data_ptr());
        } else {
            // any other object has to say itself where its memory is (a number is not an address)
            PyObject* at = PyObject_CallMethod(o, "data_ptr", nullptr);
            if (!at) return false;
            v = static_cast<T>(PyLong_AsVoidPtr(at));
            Py_DECREF(at);
        }
    } else if constexpr (std::is_floating_point_v<T>) {
        v = static_cast<T>(PyFloat_AsDouble(o));
    } else {
        v = static_cast<T>(PyLong_AsLongLong(o));
    }
    return !PyErr_Occurred();
}

// f(), its C++ exceptions as Python ones: none may leave an entry (a tensor subclass answers in Python, and may raise)
template <typename Fn>
PyObject* guarded(Fn f) {
    try {
        return f();
    } catch (python_error& e) {
        e.restore();
    } catch (const c10::Error& e) {
        PyErr_SetString(PyExc_RuntimeError, e.what_without_backtrace());
    } catch (const std::exception& e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
    }
    return nullptr;
}

// int f(args..., void* stream) as a Python function of args...
template <auto F>
struct Entry;
template <typename... A, int (*F)(A...)>
struct Entry<F> {
    template <size_t... I>
    static PyObject* run(PyObject* const* args, std::index_sequence<I...>) {
        return guarded([&]() -> PyObject* {
            std::tuple<A...> v{};
            if (!(convert(args[I], std::get<I>(v)) && ...)) return nullptr;
            std::get<sizeof...(A) - 1>(v) = c10::cuda::getCurrentCUDAStream().stream();
            int rc;
            Py_BEGIN_ALLOW_THREADS
            rc = std::apply(F, v);
            Py_END_ALLOW_THREADS
            return PyLong_FromLong(rc);
        });
    }
    static PyObject* call(PyObject*, PyObject* const* args, Py_ssize_t n) {
        constexpr Py_ssize_t want = sizeof...(A) - 1;
        if (n != want) return PyErr_Format(PyExc_TypeError, "%zd arguments expected, %zd given", want, n);
        return run(args, std::make_index_sequence<want>{});
    }
};

// check(kinds, tensors...): the index of the first one that is not a contiguous CUDA tensor of its kind, -1 if there is none
PyObject* check(PyObject*, PyObject* const* args, Py_ssize_t n) {
    Py_ssize_t len = 0;
    const char* kinds = n > 0 ? PyUnicode_AsUTF8AndSize(args[0], &len) : nullptr;
    if (!kinds) return nullptr;
    if (len != n - 1) return PyErr_Format(PyExc_TypeError, "%zd kinds, %zd tensors", len, n - 1);
    return guarded([&]() -> PyObject* {
        for (Py_ssize_t i = 0; i < len; ++i) {
            if (!THPVariable_Check(args[i + 1])) return PyLong_FromSsize_t(i);
            const at::Tensor& t = THPVariable_Unpack(args[i + 1]);
            const at::ScalarType want = kinds[i] == 'b' ? at::kBFloat16 : kinds[i] == 'l' ? at::kLong : kinds[i] == 'i' ? at::kInt : at::kFloat;
            if (!t.is_cuda() || t.scalar_type() != want || !t.is_contiguous()) return PyLong_FromSsize_t(i);
        }
        return PyLong_FromLong(-1);
    });
}

template <auto F>
constexpr PyMethodDef entry(const char* name) {
    return {name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(&Entry<F>::call)), METH_FASTCALL, nullptr};
}

PyMethodDef methods[] = {
    entry<&goose_tree_attn>("tree_attn"),
    entry<&goose_tree_attn_gqa>("tree_attn_gqa"),
    entry<&goose_node_topk>("node_topk"),
    entry<&goose_harvest>("harvest"),
    entry<&goose_accept>("accept"),
    entry<&goose_kv_compact>("kv_compact"),
    entry<&goose_verify_step>("verify_step"),
    entry<&goose_verify_step_gqa>("verify_step_gqa"),
    entry<&goose_verify_step_harvest>("verify_step_harvest"),
    {"check", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(&check)), METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};

PyModuleDef module = {PyModuleDef_HEAD_INIT, "_marshal", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__marshal() {
    PyObject* m = PyModule_Create(&module);
    if (m && PyModule_AddStringConstant(m, "built_for", GOOSE_BUILT_FOR) < 0) Py_CLEAR(m);
    return m;
}
