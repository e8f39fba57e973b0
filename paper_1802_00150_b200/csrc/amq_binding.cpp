// CPython binding of the C ABI in include/amq.h: argument marshalling only, in native code.
//
// A call through ctypes costs some 9 us of interpreter time (argument conversion, data_ptr per tensor, current_stream), twice a
// short kernel's duration; here it costs about one.  Every entry point of the header is a Python function of the same name without the trailing
// stream argument (the calling thread's current stream is used): pointers take None, a tensor (checked: CUDA, contiguous, the element
// type of the pointer) or an integer address (unchecked: strided views, host memory), sizes take integers.  The library is opened
// by path, so that an instrumented build can take its place.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <dlfcn.h>

#include <tuple>
#include <type_traits>
#include <utility>

#include <ATen/ATen.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "amq.h"

namespace {

template <typename T> struct Element;
template <> struct Element<float> { static constexpr at::ScalarType type = at::kFloat; static constexpr const char* name = "float32"; };
template <> struct Element<uint32_t> { static constexpr at::ScalarType type = at::kInt; static constexpr const char* name = "int32"; };
template <> struct Element<int32_t> { static constexpr at::ScalarType type = at::kInt; static constexpr const char* name = "int32"; };
template <> struct Element<void> { static constexpr at::ScalarType type = at::kByte; static constexpr const char* name = "uint8"; };    // (any)

// one argument; on a mismatch sets a Python error
template <typename T, typename = void> struct Arg;

template <typename T>
struct Arg<T*> {
    static T* get(PyObject* o, Py_ssize_t index)
    {
        using E = Element<std::remove_const_t<T>>;
        if (o == Py_None) return nullptr;
        if (THPVariable_Check(o)) {
            const at::Tensor& t = THPVariable_Unpack(o);
            if (t.is_cuda() && (std::is_void_v<std::remove_const_t<T>> || t.scalar_type() == E::type) && t.is_contiguous()) return static_cast<T*>(t.data_ptr());
            PyErr_Format(PyExc_TypeError, "argument %zd must be a contiguous CUDA tensor of dtype %s", index, E::name);
            return nullptr;
        }
        void* p = PyLong_AsVoidPtr(o);
        return static_cast<T*>(p);
    }
};

template <typename T>
struct Arg<T, std::enable_if_t<std::is_integral_v<T>>> {
    static T get(PyObject* o, Py_ssize_t index)
    {
        const long long v = PyLong_AsLongLong(o);
        const T r = static_cast<T>(v);
        if (static_cast<long long>(r) != v && !PyErr_Occurred())
            PyErr_Format(PyExc_OverflowError, "argument %zd is out of range", index);
        return r;
    }
};

template <typename... A, size_t... I>
PyObject* call_checked(amq_status (*f)(A...), PyObject* const* args, std::index_sequence<I...>)
{
    using Tuple = std::tuple<A...>;
    // all arguments but the last, which is the stream
    std::tuple<std::tuple_element_t<I, Tuple>...> v{Arg<std::tuple_element_t<I, Tuple>>::get(args[I], (Py_ssize_t)I)...};
    if (PyErr_Occurred()) return nullptr;
    void* stream = c10::cuda::getCurrentCUDAStream().stream();
    amq_status s;
    Py_BEGIN_ALLOW_THREADS
    s = f(std::get<I>(v)..., stream);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(s);
}

template <typename... A>
PyObject* call(amq_status (*f)(A...), PyObject* const* args, Py_ssize_t nargs)
{
    constexpr size_t N = sizeof...(A) - 1;
    if (!f) { PyErr_SetString(PyExc_RuntimeError, "the library has not been opened"); return nullptr; }
    if (nargs != (Py_ssize_t)N) {
        PyErr_Format(PyExc_TypeError, "expected %zu arguments, got %zd", N, nargs);
        return nullptr;
    }
    try {
        return call_checked(f, args, std::make_index_sequence<N>{});
    } catch (const std::exception& e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
}

#define AMQ_ENTRIES(X)                                                                                                          \
    X(amq_quantize) X(amq_pack) X(amq_unpack) X(amq_binary_dots) X(amq_binary_gemm) X(amq_quantized_gemv) X(amq_lstm_step)      \
    X(amq_lstm_step_static) X(amq_gru_step) X(amq_lstm_sequence) X(amq_gru_sequence) X(amq_lstm_sequence_host)                  \
    X(amq_gru_sequence_host) X(amq_selftest_sequence_give_up) X(amq_selftest_batched_sequence) X(amq_selftest_decode_give_up) X(amq_selftest_binary_gemm) \
    X(amq_gru_step_original) X(amq_quantize_variant) X(amq_lm_greedy_decode) X(amq_log_softmax_argmax) X(amq_embedding_rows) X(amq_lstm_step_paper) X(amq_lstm_sequence_paper)

#define AMQ_WRAP(name)                                                                          \
    decltype(&::name) p_##name = nullptr;                                                       \
    PyObject* py_##name(PyObject*, PyObject* const* args, Py_ssize_t nargs) { return call(p_##name, args, nargs); }
AMQ_ENTRIES(AMQ_WRAP)

// open(path): the library whose entry points the functions call
PyObject* py_open(PyObject*, PyObject* path)
{
    const char* p = PyUnicode_AsUTF8(path);
    if (!p) return nullptr;
    void* lib = dlopen(p, RTLD_NOW | RTLD_LOCAL);
    if (!lib) { PyErr_SetString(PyExc_ImportError, dlerror()); return nullptr; }
#define AMQ_LOOKUP(name)                                                                        \
    p_##name = reinterpret_cast<decltype(&::name)>(dlsym(lib, #name));                          \
    if (!p_##name) { PyErr_SetString(PyExc_ImportError, "missing entry point " #name); return nullptr; }
    AMQ_ENTRIES(AMQ_LOOKUP)
    Py_RETURN_NONE;
}

// empty(like, kind, d0, d1, ..): an uninitialised contiguous tensor on the device of `like`; kind 0 float32, 1 int32
PyObject* py_empty(PyObject*, PyObject* const* args, Py_ssize_t nargs)
{
    if (nargs < 2 || nargs > 8 || !THPVariable_Check(args[0])) {
        PyErr_SetString(PyExc_TypeError, "empty(like, kind, sizes..)");
        return nullptr;
    }
    int64_t size[6];
    const long kind = PyLong_AsLong(args[1]);
    for (Py_ssize_t i = 2; i < nargs; ++i) size[i - 2] = PyLong_AsLongLong(args[i]);
    if (PyErr_Occurred()) return nullptr;
    try {
        const at::Tensor& like = THPVariable_Unpack(args[0]);
        return THPVariable_Wrap(at::empty(at::IntArrayRef(size, nargs - 2),
                                          at::TensorOptions().dtype(kind ? at::kInt : at::kFloat).device(like.device())));
    } catch (const std::exception& e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
}

#define AMQ_METHOD(name) {#name, (PyCFunction)(void (*)(void))py_##name, METH_FASTCALL, nullptr},
PyMethodDef methods[] = {
    AMQ_ENTRIES(AMQ_METHOD)
    {"open", py_open, METH_O, nullptr},
    {"empty", (PyCFunction)(void (*)(void))py_empty, METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr},
};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_amq_binding", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__amq_binding() { return PyModule_Create(&module); }
