// Call path from Python into the C ABI of include/rvq.h.
//
// Every kernel call of the package goes through here: the arguments come as a vectorcall array in
// the C function's own order and are converted by the type of the C parameter they meet (tensors to
// their device address, None to NULL, the config by its buffer).  The last parameter of every entry
// point is its stream; None there is PyTorch's current stream.
//
// Why native: what bounds a call on a few head vectors is the host.  Marshalled through ctypes a call
// cost 5.9-6.6 us before the CUDA runtime was reached (data_ptr(), the current stream's Python object
// and ctypes' conversions), twice what the launch itself costs.
#include <Python.h>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <tuple>
#include <type_traits>
#include <utility>

#include "rvq.h"
#include "rvq_selftest.h"

namespace {

// Converts one argument; false with a Python error set when it cannot.
template <typename T>
bool from_python(PyObject *o, T *out)
{
    if constexpr (std::is_same_v<T, const rvq_config *>) {
        return false;                                        // (configs are taken by config_of below)
    } else if constexpr (std::is_pointer_v<T>) {
        if (o == Py_None) {
            *out = nullptr;
        } else if (THPVariable_Check(o)) {
            // (a buffer that the call writes is asked for as such: a tensor that shares its storage until the
            // first write gets storage of its own)
            if constexpr (std::is_const_v<std::remove_pointer_t<T>>) *out = reinterpret_cast<T>(THPVariable_Unpack(o).const_data_ptr());
            else *out = reinterpret_cast<T>(THPVariable_Unpack(o).mutable_data_ptr());
        } else if (PyLong_Check(o)) {
            *out = reinterpret_cast<T>(PyLong_AsVoidPtr(o));
        } else {
            PyObject *p = PyObject_CallMethod(o, "data_ptr", nullptr);
            if (!p) return false;
            *out = reinterpret_cast<T>(PyLong_AsVoidPtr(p));
            Py_DECREF(p);
        }
    } else if constexpr (std::is_floating_point_v<T>) {
        *out = (T)PyFloat_AsDouble(o);
    } else if constexpr (std::is_unsigned_v<T>) {
        *out = (T)PyLong_AsUnsignedLongLong(o);
    } else {
        *out = (T)PyLong_AsLongLong(o);
    }
    return !PyErr_Occurred();
}

bool config_of(PyObject *o, rvq_config *out)
{
    Py_buffer view;
    if (PyObject_GetBuffer(o, &view, PyBUF_SIMPLE) != 0) return false;
    const bool fits = view.len == (Py_ssize_t)sizeof(rvq_config);
    if (fits) memcpy(out, view.buf, sizeof(rvq_config));
    PyBuffer_Release(&view);
    if (!fits) PyErr_SetString(PyExc_TypeError, "expected an rvq_config");
    return fits;
}

bool stream_of(PyObject *o, void **out)
{
    if (o == Py_None) {
        *out = c10::cuda::getCurrentCUDAStream().stream();
        return true;
    }
    if (!PyLong_Check(o) && PyObject_HasAttrString(o, "cuda_stream")) {
        PyObject *h = PyObject_GetAttrString(o, "cuda_stream");
        if (!h) return false;
        *out = PyLong_AsVoidPtr(h);
        Py_DECREF(h);
    } else {
        PyObject *h = PyNumber_Long(o);
        if (!h) return false;
        *out = PyLong_AsVoidPtr(h);
        Py_DECREF(h);
    }
    return !PyErr_Occurred();
}

template <typename... A, size_t... I>
PyObject *invoke(int (*fn)(A...), PyObject *const *args, Py_ssize_t nargs, std::index_sequence<I...>)
{
    constexpr size_t N = sizeof...(A);
    if (nargs != (Py_ssize_t)N) {
        PyErr_Format(PyExc_TypeError, "expected %zu arguments, got %zd", N, nargs);
        return nullptr;
    }
    std::tuple<A...> v;
    rvq_config configs[2];                                    // (at most two, in the first places)
    auto take = [&](auto index) -> bool {
        constexpr size_t i = decltype(index)::value;
        using T = std::tuple_element_t<i, std::tuple<A...>>;
        if constexpr (std::is_same_v<T, const rvq_config *>) {
            static_assert(i < 2, "configs come first");
            std::get<i>(v) = &configs[i];
            return config_of(args[i], &configs[i]);
        } else if constexpr (i == N - 1) {
            static_assert(std::is_same_v<T, void *>, "the stream comes last");
            return stream_of(args[i], &std::get<i>(v));
        } else {
            return from_python(args[i], &std::get<i>(v));
        }
    };
    try {
        if (!(take(std::integral_constant<size_t, I>()) && ...)) return nullptr;
    } catch (const std::exception &e) {                       // c10: no device, no storage
        PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = std::apply(fn, v);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

template <typename F> struct Entry;
template <typename... A>
struct Entry<int (*)(A...)> {
    template <int (*fn)(A...)>
    static PyObject *call(PyObject *, PyObject *const *args, Py_ssize_t nargs)
    {
        return invoke(fn, args, nargs, std::index_sequence_for<A...>());
    }
};

#define RVQ_METHOD(name)                                                                            \
    {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(&Entry<decltype(&name)>::call<&name>)), \
     METH_FASTCALL, nullptr}

PyMethodDef methods[] = {
    RVQ_METHOD(rvq_prepare_codebooks), RVQ_METHOD(rvq_encode),      RVQ_METHOD(rvq_encode_stats),
    RVQ_METHOD(rvq_encode_exact),      RVQ_METHOD(rvq_decode),      RVQ_METHOD(rvq_rope_table),
    RVQ_METHOD(rvq_decode_rope),       RVQ_METHOD(rvq_attention_decode),
    RVQ_METHOD(rvq_ema_update),        RVQ_METHOD(rvq_ema_stats),   RVQ_METHOD(rvq_ema_apply),
    RVQ_METHOD(rvq_learn_step),        RVQ_METHOD(rvq_kmeans_init), RVQ_METHOD(rvq_ema_update_static),
    RVQ_METHOD(rvq_selftest_encode_timeout),
    {nullptr, nullptr, 0, nullptr}};

PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native() { return PyModule_Create(&module); }
