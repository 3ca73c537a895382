// Python entry points of the library's launching calls: argument marshalling in native code.
//
// A call made from Python spent 12 us on the host, of which the launch itself is a quarter: ctypes converts
// every argument through an object, and the stream and the addresses are looked up through Python layers.  A step
// of a few small launches is bound by that.  Here a call's C signature says how its arguments are converted:
// pointers come from tensors (their data_ptr()), integers or None, a workspace gives its address and its size,
// and a stream that is not given is torch's current one.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <tuple>
#include <type_traits>
#include <utility>

#include "eagle2.h"

namespace {

PyObject* g_data_ptr;      // the interned method names
PyObject* g_numel;
PyObject* g_element_size;
PyObject* g_cuda_stream;
PyObject* g_device_fn;     // torch: current device, raw stream of a device; NULL where there is no GPU
PyObject* g_raw_stream_fn;

bool as_long(PyObject* o, long long* v) {
    *v = PyLong_AsLongLong(o);
    if (*v != -1 || !PyErr_Occurred()) return true;
    if (!PyErr_ExceptionMatches(PyExc_TypeError)) return false;
    PyErr_Clear();  // anything else that can say which integer it is
    PyObject* i = PyNumber_Index(o);
    if (!i) return false;
    *v = PyLong_AsLongLong(i);
    Py_DECREF(i);
    return !(*v == -1 && PyErr_Occurred());
}
bool method_long(PyObject* o, PyObject* name, long long* v) {
    PyObject* r = PyObject_CallMethodNoArgs(o, name);
    if (!r) return false;
    const bool ok = PyLong_Check(r) ? (*v = (long long)PyLong_AsUnsignedLongLong(r), !PyErr_Occurred()) : as_long(r, v);
    Py_DECREF(r);
    return ok;
}
// None, an address, or a tensor
bool as_pointer(PyObject* o, void** p) {
    if (o == Py_None) {
        *p = nullptr;
        return true;
    }
    if (PyLong_Check(o)) {
        *p = (void*)PyLong_AsUnsignedLongLong(o);
        return !PyErr_Occurred();
    }
    long long v;
    if (!method_long(o, g_data_ptr, &v)) return false;
    *p = (void*)v;
    return true;
}
bool as_stream(PyObject* o, eagle2_stream_t* s) {
    if (o != Py_None) {
        if (PyLong_Check(o)) {
            *s = (eagle2_stream_t)PyLong_AsUnsignedLongLong(o);
            return !PyErr_Occurred();
        }
        PyObject* r = PyObject_GetAttr(o, g_cuda_stream);
        if (!r) return false;
        *s = (eagle2_stream_t)PyLong_AsUnsignedLongLong(r);
        Py_DECREF(r);
        return !PyErr_Occurred();
    }
    *s = nullptr;
    if (!g_raw_stream_fn) return true;
    PyObject* dev = PyObject_CallNoArgs(g_device_fn);
    if (!dev) return false;
    PyObject* r = PyObject_CallOneArg(g_raw_stream_fn, dev);
    Py_DECREF(dev);
    if (!r) return false;
    *s = (eagle2_stream_t)PyLong_AsUnsignedLongLong(r);
    Py_DECREF(r);
    return !PyErr_Occurred();
}

// Conversion of one argument.
template <class T>
struct Arg;
template <class T>
struct Arg<T*> {
    static bool get(PyObject* o, T** v) { return as_pointer(o, (void**)v); }
};
template <>
struct Arg<eagle2_stream_t> {
    static bool get(PyObject* o, eagle2_stream_t* v) { return as_stream(o, v); }
};
template <>
struct Arg<int> {
    static bool get(PyObject* o, int* v) {
        long long x;
        if (!as_long(o, &x)) return false;
        if (x != (long long)(int)x) {
            PyErr_SetString(PyExc_OverflowError, "argument does not fit in an int");
            return false;
        }
        *v = (int)x;
        return true;
    }
};
template <>
struct Arg<unsigned> {
    static bool get(PyObject* o, unsigned* v) {
        long long x;
        if (!as_long(o, &x)) return false;
        *v = (unsigned)x;
        return true;
    }
};
template <>
struct Arg<long long> {
    static bool get(PyObject* o, long long* v) { return as_long(o, v); }
};
template <>
struct Arg<float> {
    static bool get(PyObject* o, float* v) {
        const double x = PyFloat_AsDouble(o);
        if (x == -1.0 && PyErr_Occurred()) return false;
        *v = (float)x;
        return true;
    }
};
// the size of a workspace: of the tensor in front of it
template <>
struct Arg<size_t> {
    static bool get(PyObject* o, size_t* v) {
        *v = 0;
        if (o == Py_None || PyLong_Check(o)) return true;
        long long n, e;
        if (!method_long(o, g_numel, &n) || !method_long(o, g_element_size, &e)) return false;
        *v = (size_t)(n * e);
        return true;
    }
};

template <auto F>
struct Call;
template <class... A, int (*F)(A...)>
struct Call<F> {
    static constexpr bool kIsSize[sizeof...(A)] = {std::is_same_v<A, size_t>...};
    static constexpr Py_ssize_t count() {
        Py_ssize_t n = 0;
        for (bool s : kIsSize) n += s ? 0 : 1;
        return n;
    }
    template <size_t... I>
    static PyObject* run(PyObject* const* args, std::index_sequence<I...>) {
        // Python argument of C argument i: a size shares its workspace's
        int at[sizeof...(A)], n = 0;
        for (size_t i = 0; i < sizeof...(A); ++i) at[i] = kIsSize[i] ? n - 1 : n++;
        std::tuple<A...> v;
        if (!(Arg<A>::get(args[at[I]], &std::get<I>(v)) && ...)) return nullptr;
        int code;
        Py_BEGIN_ALLOW_THREADS
        code = F(std::get<I>(v)...);
        Py_END_ALLOW_THREADS
        return PyLong_FromLong(code);
    }
    static PyObject* call(PyObject*, PyObject* const* args, Py_ssize_t n) {
        if (n != count()) {
            PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", count(), n);
            return nullptr;
        }
        return run(args, std::make_index_sequence<sizeof...(A)>{});
    }
};

PyObject* set_stream_source(PyObject*, PyObject* const* args, Py_ssize_t n) {
    if (n != 2) {
        PyErr_SetString(PyExc_TypeError, "expected the device and the raw stream function");
        return nullptr;
    }
    Py_XSETREF(g_device_fn, Py_NewRef(args[0]));
    Py_XSETREF(g_raw_stream_fn, Py_NewRef(args[1]));
    Py_RETURN_NONE;
}

#define ENTRY(name) {#name, (PyCFunction)(void (*)(void))Call<eagle2_##name>::call, METH_FASTCALL, nullptr}
PyMethodDef g_methods[] = {ENTRY(workspace_init),
                           ENTRY(lm_head),
                           ENTRY(lm_head_expand),
                           ENTRY(expand),
                           ENTRY(expand_variant),
                           ENTRY(expand_static),
                           ENTRY(rerank),
                           ENTRY(rerank_skipped),
                           ENTRY(rerank_mask),
                           ENTRY(tree_mask),
                           ENTRY(tree_attention),
                           ENTRY(accept),
                           ENTRY(kv_compact),
                           {"set_stream_source", (PyCFunction)(void (*)(void))set_stream_source, METH_FASTCALL, nullptr},
                           {nullptr, nullptr, 0, nullptr}};
PyModuleDef g_module = {PyModuleDef_HEAD_INIT, "_native", "Launching calls of libeagle2.so.", -1, g_methods};

}  // namespace

PyMODINIT_FUNC PyInit__native() {
    g_data_ptr = PyUnicode_InternFromString("data_ptr");
    g_numel = PyUnicode_InternFromString("numel");
    g_element_size = PyUnicode_InternFromString("element_size");
    g_cuda_stream = PyUnicode_InternFromString("cuda_stream");
    if (!g_data_ptr || !g_numel || !g_element_size || !g_cuda_stream) return nullptr;
    return PyModule_Create(&g_module);
}
