// Python module `_native`: the functions of include/small.h called with Python arguments.  A layer call has some twenty
// arguments; converting them one by one in ctypes and asking torch for a Stream object took 7 of the 10 microseconds of a
// small layer's call, more than its kernel.  Here a wrapper per function is generated from the function's own C type:
// integers are read directly, device pointers come from an int, None or an object with data_ptr(), and a stream argument of
// None (always the last one) is the current stream's handle.  Argument marshalling only, like binding.py, which names the
// parameters and adds the defaults.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <cstdint>
#include <type_traits>
#include <tuple>
#include <utility>

#include "small.h"

namespace {

PyObject *g_fail, *g_device, *g_raw_stream;          // set by configure()
PyObject *s_data_ptr, *s_cuda_stream;

bool to_int(PyObject *o, long long &v) {
    if (PyLong_Check(o)) {
        v = PyLong_AsLongLong(o);
        if (v == -1 && PyErr_Occurred()) return false;
        return true;
    }
    PyObject *i = PyNumber_Index(o);
    if (!i) return false;
    v = PyLong_AsLongLong(i);
    Py_DECREF(i);
    return !(v == -1 && PyErr_Occurred());
}

bool long_to_ptr(PyObject *o, void *&p) {
    p = PyLong_AsVoidPtr(o);
    return !(p == nullptr && PyErr_Occurred());
}

// device (or host) memory: None, an address, or a tensor
bool to_memory(PyObject *o, void *&p) {
    if (o == Py_None) { p = nullptr; return true; }
    if (PyLong_Check(o)) return long_to_ptr(o, p);
    PyObject *a = PyObject_CallMethodNoArgs(o, s_data_ptr);
    if (!a) return false;
    const bool ok = long_to_ptr(a, p);
    Py_DECREF(a);
    return ok;
}

// a ctypes instance: its storage (an array of descriptors), or the pointer stored in it (the context's c_void_p)
bool to_ctypes(PyObject *o, void *&p, bool stored) {
    if (o == Py_None) { p = nullptr; return true; }
    if (PyLong_Check(o)) return long_to_ptr(o, p);
    Py_buffer b;
    if (PyObject_GetBuffer(o, &b, PyBUF_SIMPLE) != 0) return false;
    p = b.buf;
    if (stored) p = b.len >= (Py_ssize_t)sizeof(void *) ? *static_cast<void **>(b.buf) : nullptr;
    PyBuffer_Release(&b);
    return true;
}

bool to_stream(PyObject *o, void *&p) {
    if (PyLong_Check(o)) return long_to_ptr(o, p);
    PyObject *h;
    if (o == Py_None) {
        PyObject *dev = PyObject_CallNoArgs(g_device);
        if (!dev) return false;
        h = PyObject_CallOneArg(g_raw_stream, dev);
        Py_DECREF(dev);
    } else {
        h = PyObject_GetAttr(o, s_cuda_stream);
    }
    if (!h) return false;
    const bool ok = long_to_ptr(h, p);
    Py_DECREF(h);
    return ok;
}

template <typename T>
bool convert(PyObject *o, T &out, bool is_stream) {
    if constexpr (std::is_pointer_v<T>) {
        void *p = nullptr;
        bool ok;
        if constexpr (std::is_same_v<T, small_ctx *>) ok = to_ctypes(o, p, true);
        else if constexpr (std::is_same_v<T, const small_layer *>) ok = to_ctypes(o, p, false);
        else ok = is_stream ? to_stream(o, p) : to_memory(o, p);
        out = static_cast<T>(p);
        return ok;
    } else {
        long long v;
        if (!to_int(o, v)) return false;
        out = static_cast<T>(v);
        return true;
    }
}

template <auto Fn, bool kStatus>
struct Call;

template <typename R, typename... A, R (*Fn)(A...), bool kStatus>
struct Call<Fn, kStatus> {
    static constexpr size_t kArgs = sizeof...(A);
    template <size_t... I>
    static PyObject *run(PyObject *const *args, const char *name, std::index_sequence<I...>) {
        std::tuple<A...> v{};
        // a trailing void* is the stream
        if (!(convert(args[I], std::get<I>(v), I == kArgs - 1 && std::is_same_v<std::tuple_element_t<I, std::tuple<A...>>, void *>) && ...)) return nullptr;
        R r;
        Py_BEGIN_ALLOW_THREADS
        r = Fn(std::get<I>(v)...);
        Py_END_ALLOW_THREADS
        if constexpr (kStatus) {
            if (r != SMALL_OK) return PyObject_CallFunction(g_fail, "is", (int)r, name);
            Py_RETURN_NONE;
        } else if constexpr (std::is_same_v<R, size_t>) {
            return PyLong_FromSize_t(r);
        } else {
            return PyLong_FromLong((long)r);
        }
    }
    static PyObject *call(PyObject *const *args, Py_ssize_t n, const char *name) {
        if (n != (Py_ssize_t)kArgs) {
            PyErr_Format(PyExc_TypeError, "%s takes %zu arguments (%zd given)", name, kArgs, n);
            return nullptr;
        }
        return run(args, name, std::make_index_sequence<kArgs>{});
    }
};

#define STATUS(f) PyObject *py_##f(PyObject *, PyObject *const *a, Py_ssize_t n) { return Call<&f, true>::call(a, n, #f); }
#define VALUE(f) PyObject *py_##f(PyObject *, PyObject *const *a, Py_ssize_t n) { return Call<&f, false>::call(a, n, #f); }
#define EACH(S, V) \
    S(small_pack) S(small_unpack) S(small_pack_conv_weights) S(small_pack_group_conv_weights) S(small_pack_dw_weights) S(small_pack_fc_weights) \
    S(small_conv2d) S(small_group_conv2d) S(small_dwpw_conv2d) S(small_conv_maxpool2d) S(small_dwconv2d) S(small_pool2d) S(small_relu) \
    S(small_scale_shift) S(small_upsample_nearest) S(small_add) S(small_fc) S(small_gap_fc) S(small_set_net_fusion) S(small_run_net) \
    S(small_run_net_host) S(small_run_net_static) S(small_q_pack) S(small_q_unpack) S(small_q_pack_conv_weights) S(small_q_conv2d) \
    S(small_q_pack_dw_weights) S(small_q_dwconv2d) S(small_q_maxpool2d) S(small_q_relu) V(small_out_size) V(small_packed_elems) V(small_q_packed_bytes)

EACH(STATUS, VALUE)

// configure(fail, device, raw_stream): what raises a status, and torch's current device and that device's current stream
PyObject *configure(PyObject *, PyObject *args) {
    PyObject *f, *d, *s;
    if (!PyArg_ParseTuple(args, "OOO", &f, &d, &s)) return nullptr;
    Py_INCREF(f); Py_INCREF(d); Py_INCREF(s);
    Py_XDECREF(g_fail); Py_XDECREF(g_device); Py_XDECREF(g_raw_stream);
    g_fail = f; g_device = d; g_raw_stream = s;
    Py_RETURN_NONE;
}

#define ENTRY(f) {#f, (PyCFunction)(void (*)(void))py_##f, METH_FASTCALL, nullptr},
PyMethodDef methods[] = {{"configure", configure, METH_VARARGS, nullptr}, EACH(ENTRY, ENTRY){nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native() {
    s_data_ptr = PyUnicode_InternFromString("data_ptr");
    s_cuda_stream = PyUnicode_InternFromString("cuda_stream");
    return PyModule_Create(&module);
}
