// CPython entry to the C ABI: one vectorcall per library call, arguments converted by the types of the C prototype.
//
// Through ctypes a call cost 5 to 8 us of interpreter time before its first launch (argument objects, and 3.2 us for
// torch.cuda.current_stream()), more than most small conversions and products take on the device.  Here a tensor is its
// data_ptr(), the stream is the current one unless the caller names another, and the interpreter lock is released around
// the library call as ctypes does.  Arguments that do not convert make the call return None without having called the
// library; the caller then goes through ctypes, which reports them.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <cstddef>
#include <cstdint>
#include <tuple>
#include <type_traits>
#include <utility>

#include "hif8.h"

namespace {

PyObject* g_get_device = nullptr;      // () -> current device ordinal
PyObject* g_get_raw_stream = nullptr;  // device ordinal -> its current stream
PyObject* g_data_ptr = nullptr;        // the two attribute names
PyObject* g_cuda_stream = nullptr;
bool g_cuda_ready = false;             // CUDA is initialised in this process

bool to_address(PyObject* o, void** out)
{
    if (o == Py_None) { *out = nullptr; return true; }
    if (PyLong_Check(o)) { *out = reinterpret_cast<void*>(static_cast<uintptr_t>(PyLong_AsUnsignedLongLongMask(o))); return !PyErr_Occurred(); }
    PyObject* v = PyObject_CallMethodNoArgs(o, g_data_ptr);
    if (!v) return false;
    const bool ok = PyLong_Check(v);
    if (ok) *out = reinterpret_cast<void*>(static_cast<uintptr_t>(PyLong_AsUnsignedLongLongMask(v)));
    Py_DECREF(v);
    return ok && !PyErr_Occurred();
}

bool to_stream(PyObject* o, void** out)
{
    PyObject* v;
    if (o == Py_None) {
        if (!g_cuda_ready) return false;
        PyObject* dev = PyObject_CallNoArgs(g_get_device);
        if (!dev) return false;
        v = PyObject_CallOneArg(g_get_raw_stream, dev);
        Py_DECREF(dev);
    } else if (PyLong_Check(o)) {
        Py_INCREF(o);
        v = o;
    } else v = PyObject_GetAttr(o, g_cuda_stream);
    if (!v) return false;
    const bool ok = PyLong_Check(v);
    if (ok) *out = reinterpret_cast<void*>(static_cast<uintptr_t>(PyLong_AsUnsignedLongLongMask(v)));
    Py_DECREF(v);
    return ok && !PyErr_Occurred();
}

template <class T>
bool convert(PyObject* o, T* out)
{
    if constexpr (std::is_same_v<T, hif8_stream_t>) return to_stream(o, reinterpret_cast<void**>(out));
    else if constexpr (std::is_pointer_v<T>) {
        void* p = nullptr;
        if (!to_address(o, &p)) return false;
        *out = static_cast<T>(p);
        return true;
    } else {
        if (PyFloat_Check(o)) return false;
        const unsigned long long v = PyLong_AsUnsignedLongLongMask(o);  // (wraps, as a ctypes integer argument does)
        if (v == static_cast<unsigned long long>(-1) && PyErr_Occurred()) return false;
        *out = static_cast<T>(v);
        return true;
    }
}

template <auto F> struct Entry;
template <class... A, int (*F)(A...)>
struct Entry<F> {
    template <size_t... I>
    static PyObject* run(PyObject* const* args, std::index_sequence<I...>)
    {
        std::tuple<A...> a{};
        if (!(convert<A>(args[I], &std::get<I>(a)) && ...)) { PyErr_Clear(); Py_RETURN_NONE; }
        int rc;
        Py_BEGIN_ALLOW_THREADS
        rc = F(std::get<I>(a)...);
        Py_END_ALLOW_THREADS
        return PyLong_FromLong(rc);
    }
    static PyObject* call(PyObject*, PyObject* const* args, Py_ssize_t n)
    {
        if (n != static_cast<Py_ssize_t>(sizeof...(A))) Py_RETURN_NONE;
        return run(args, std::index_sequence_for<A...>{});
    }
};

PyObject* set_up(PyObject*, PyObject* const* args, Py_ssize_t n)
{
    if (n != 2) { PyErr_SetString(PyExc_TypeError, "set_up(get_device, get_raw_stream)"); return nullptr; }
    Py_INCREF(args[0]); Py_INCREF(args[1]);
    Py_XSETREF(g_get_device, args[0]);
    Py_XSETREF(g_get_raw_stream, args[1]);
    Py_RETURN_NONE;
}

PyObject* set_cuda_ready(PyObject*, PyObject* o)
{
    const int v = PyObject_IsTrue(o);
    if (v < 0) return nullptr;
    g_cuda_ready = v != 0;
    Py_RETURN_NONE;
}

#define HIF8_ENTRY(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(&Entry<&name>::call)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {
    HIF8_ENTRY(hif8_encode), HIF8_ENTRY(hif8_decode), HIF8_ENTRY(hif8_amax), HIF8_ENTRY(hif8_amax_scale_encode),
    HIF8_ENTRY(hif8_amax_scale_encode_static), HIF8_ENTRY(hif8_fake_quant), HIF8_ENTRY(hif8_gemm), HIF8_ENTRY(hif8_gemm_ex),
    HIF8_ENTRY(hif8_gemm_channel_scaled), HIF8_ENTRY(hif8_channel_amax_scale_encode), HIF8_ENTRY(hif8_delayed_scale_encode),
    HIF8_ENTRY(hif8_encode_transpose), HIF8_ENTRY(hif8_encode_from_amax), HIF8_ENTRY(hif8_als_update), HIF8_ENTRY(hif8_check_finite),
    {"set_up", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(&set_up)), METH_FASTCALL, nullptr},
    {"set_cuda_ready", &set_cuda_ready, METH_O, nullptr},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module_def = {PyModuleDef_HEAD_INIT, "_hif8_call", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__hif8_call()
{
    g_data_ptr = PyUnicode_InternFromString("data_ptr");
    g_cuda_stream = PyUnicode_InternFromString("cuda_stream");
    if (!g_data_ptr || !g_cuda_stream) return nullptr;
    return PyModule_Create(&module_def);
}
