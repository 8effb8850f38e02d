// Python entry to the C calls that a training step makes, beside the ctypes binding of convbn.py.
// ctypes and the Python code that turned thirteen tensors into addresses took 2.8 us of a call of 5.9 us (forward of a 3x3
// 64 -> 64 layer, 1.4 of them for data_ptr alone).  With this, the plans of a layer kept (convbn_api.cu) and three allocations less
// per layer of a backbone (backbone.py): a ResNet-50 iteration that waits for the host 1820 -> 1300 us, 1x1 128 -> 256 at 9 x 13,
// N = 36 21.8 -> 18.3, depthwise 128 at 18 x 24 18.6 -> 16.4.  Arguments are converted by the declared parameter types
// of the C function: a descriptor is the object's buffer (ctypes structures export theirs), a pointer is None, an integer
// address or what data_ptr() returns.  The two arguments that every call ends with are resolved as the Python functions
// document them: workspace_bytes None is the workspace's nbytes, stream None is torch's current stream.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <cstdint>
#include <tuple>
#include <type_traits>
#include <utility>

#include "../../include/convbn.h"

namespace {

PyObject *s_data_ptr, *s_nbytes, *s_cuda_stream;      // attribute names
PyObject *g_get_device, *g_get_stream;                // torch._C._cuda_getDevice, _cuda_getCurrentRawStream

bool address(PyObject *o, void **out) {
    if (o == Py_None) { *out = nullptr; return true; }
    if (PyLong_Check(o)) {
        *out = PyLong_AsVoidPtr(o);
        return *out || !PyErr_Occurred();
    }
    PyObject *v = PyObject_CallMethodNoArgs(o, s_data_ptr);
    if (!v) return false;
    *out = PyLong_AsVoidPtr(v);
    Py_DECREF(v);
    return *out || !PyErr_Occurred();
}

bool stream(PyObject *o, void **out) {
    if (PyLong_Check(o)) { *out = PyLong_AsVoidPtr(o); return *out || !PyErr_Occurred(); }
    PyObject *v;
    if (o == Py_None) {
        if (!g_get_stream) {
            PyObject *m = PyImport_ImportModule("torch._C");
            if (!m) return false;
            g_get_device = PyObject_GetAttrString(m, "_cuda_getDevice");
            if (g_get_device) g_get_stream = PyObject_GetAttrString(m, "_cuda_getCurrentRawStream");
            Py_DECREF(m);
            if (!g_get_stream) return false;
        }
        PyObject *d = PyObject_CallNoArgs(g_get_device);
        if (!d) return false;
        v = PyObject_CallOneArg(g_get_stream, d);
        Py_DECREF(d);
    } else {
        v = PyObject_GetAttr(o, s_cuda_stream);
    }
    if (!v) return false;
    *out = PyLong_AsVoidPtr(v);
    Py_DECREF(v);
    return *out || !PyErr_Occurred();
}

template <class T>
bool convert(PyObject *o, T *out) {
    if constexpr (std::is_same_v<T, const convbn_desc *>) {
        if (o == Py_None) { *out = nullptr; return true; }
        Py_buffer b;
        if (PyObject_GetBuffer(o, &b, PyBUF_SIMPLE) != 0) return false;
        const bool fits = (size_t)b.len == sizeof(convbn_desc);
        *out = (const convbn_desc *)b.buf;            // (the caller holds the descriptor for the length of the call)
        PyBuffer_Release(&b);
        if (!fits) PyErr_SetString(PyExc_TypeError, "a convolution descriptor is expected");
        return fits;
    } else if constexpr (std::is_pointer_v<T>) {
        void *p = nullptr;
        if (!address(o, &p)) return false;
        *out = (T)p;
        return true;
    } else {
        // (as ctypes does: integers only, and cut to the parameter's width)
        if (!PyLong_Check(o)) {
            PyErr_Format(PyExc_TypeError, "an integer is expected, not %.100s", Py_TYPE(o)->tp_name);
            return false;
        }
        const unsigned long long v = PyLong_AsUnsignedLongLongMask(o);
        if (v == (unsigned long long)-1 && PyErr_Occurred()) return false;
        *out = (T)v;
        return true;
    }
}

// f(arguments ..., [workspace, workspace_bytes,] stream)
template <class... P, size_t... I>
PyObject *call(int (*f)(P...), PyObject *const *a, Py_ssize_t n, std::index_sequence<I...>) {
    constexpr size_t N = sizeof...(P);
    if (n != (Py_ssize_t)N) return PyErr_Format(PyExc_TypeError, "%zu arguments are expected", N);
    std::tuple<P...> v;
    using Bytes = std::tuple_element_t<N >= 2 ? N - 2 : 0, std::tuple<P...>>;
    bool ok = true;
    auto one = [&](auto index) {
        constexpr size_t K = decltype(index)::value;
        if (!ok) return;
        if constexpr (K == N - 1) {
            ok = stream(a[K], &std::get<K>(v));
        } else if constexpr (K + 2 == N && std::is_same_v<Bytes, size_t>) {
            if (a[K] != Py_None) { ok = convert(a[K], &std::get<K>(v)); return; }
            std::get<K>(v) = 0;
            if (a[K - 1] == Py_None) return;
            PyObject *b = PyObject_GetAttr(a[K - 1], s_nbytes);
            ok = b && convert(b, &std::get<K>(v));
            Py_XDECREF(b);
        } else {
            ok = convert(a[K], &std::get<K>(v));
        }
    };
    (one(std::integral_constant<size_t, I>()), ...);
    if (!ok) return nullptr;
    int status;
    Py_BEGIN_ALLOW_THREADS
    status = std::apply(f, v);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(status);
}

template <auto F>
struct Entry;
template <class... P, int (*F)(P...)>
struct Entry<F> {
    static PyObject *go(PyObject *, PyObject *const *a, Py_ssize_t n) { return call(F, a, n, std::index_sequence_for<P...>()); }
};

#define ENTRY(name) {#name, (PyCFunction)(void (*)(void))Entry<&name>::go, METH_FASTCALL, nullptr}
PyMethodDef g_methods[] = {
    ENTRY(convbn_tune_fwd), ENTRY(convbn_tune_bwd_data), ENTRY(convbn_tune_bwd_weight), ENTRY(convbn_tune_bwd),
    ENTRY(convbn_tune_bwd_begin), ENTRY(convbn_tune_bwd_join), ENTRY(convbn_tune_fwd_glue), ENTRY(convbn_tune_bwd_glue),
    ENTRY(convbn_tconv_tune_fwd), ENTRY(convbn_tconv_tune_bwd), ENTRY(convbn_eval_fwd), ENTRY(convbn_eval_bwd),
    ENTRY(convbn_deploy_fwd), ENTRY(convbn_deploy_bwd), {nullptr, nullptr, 0, nullptr}};
PyModuleDef g_module = {PyModuleDef_HEAD_INIT, "_binding", nullptr, -1, g_methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__binding(void) {
    s_data_ptr = PyUnicode_InternFromString("data_ptr");
    s_nbytes = PyUnicode_InternFromString("nbytes");
    s_cuda_stream = PyUnicode_InternFromString("cuda_stream");
    return s_data_ptr && s_nbytes && s_cuda_stream ? PyModule_Create(&g_module) : nullptr;
}
