// Argument marshalling of the entry points that a serving loop calls per token or per round, as a CPython extension.
//
// The smallest launches take about 3 us on the GPU, and ctypes needs longer than that to convert the dozen arguments
// of a call (measured, one draft step of one 32000-token row back to back: 5.3 us through ctypes, of which 3.4 us are
// Python and ctypes; see binding.py).  Conversions are those of the ctypes binding: a pointer may be None, an integer
// address, a torch tensor (its data_ptr()) or, for the last argument, a torch stream (its cuda_stream).  The GIL is
// released while the library runs.  The extension is not linked against the library: binding.py hands over the
// addresses of the functions it has loaded.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <tuple>

#include "svip.h"

namespace {

PyObject* g_data_ptr;      // interned "data_ptr" and "cuda_stream"
PyObject* g_cuda_stream;

// Each returns false with a Python exception set if the object does not convert.
bool to_address(PyObject* o, bool is_stream, void** out) {
    if (o == Py_None) { *out = nullptr; return true; }
    if (PyLong_Check(o)) { *out = reinterpret_cast<void*>(PyLong_AsUnsignedLongLongMask(o)); return !PyErr_Occurred(); }
    PyObject* v = is_stream ? PyObject_GetAttr(o, g_cuda_stream) : PyObject_CallMethodNoArgs(o, g_data_ptr);
    if (!v) return false;
    *out = reinterpret_cast<void*>(PyLong_AsUnsignedLongLongMask(v));
    Py_DECREF(v);
    return !PyErr_Occurred();
}

bool to_integer(PyObject* o, long* out) {
    if (PyLong_Check(o)) { *out = static_cast<long>(PyLong_AsUnsignedLongLongMask(o)); return !PyErr_Occurred(); }
    PyObject* v = PyNumber_Long(o);
    if (!v) return false;
    *out = static_cast<long>(PyLong_AsUnsignedLongLongMask(v));
    Py_DECREF(v);
    return !PyErr_Occurred();
}

template <class T> struct Arg;
template <class T> struct Arg<T*> {
    static bool get(PyObject* o, bool last, T** out) {
        void* p = nullptr;
        if (!to_address(o, last, &p)) return false;
        *out = static_cast<T*>(p);
        return true;
    }
};
template <> struct Arg<float> {
    static bool get(PyObject* o, bool, float* out) {
        if (PyFloat_CheckExact(o)) { *out = static_cast<float>(PyFloat_AS_DOUBLE(o)); return true; }
        PyObject* v = PyNumber_Float(o);      // what float() takes, texts included
        if (!v) return false;
        *out = static_cast<float>(PyFloat_AS_DOUBLE(v));
        Py_DECREF(v);
        return true;
    }
};
template <class T> struct IntegerArg {
    static bool get(PyObject* o, bool, T* out) {
        long v = 0;
        if (!to_integer(o, &v)) return false;
        *out = static_cast<T>(v);
        return true;
    }
};
template <> struct Arg<int> : IntegerArg<int> {};
template <> struct Arg<long> : IntegerArg<long> {};
template <> struct Arg<svip_dtype> : IntegerArg<svip_dtype> {};

// The arguments one after another into a recursion of typed locals, then the call.
template <class R, class... All>
struct Caller {
    template <class... Done>
    static bool run(R (*f)(All...), PyObject* const* a, int* rc, Done... done) {
        if constexpr (sizeof...(Done) == sizeof...(All)) {
            Py_BEGIN_ALLOW_THREADS
            *rc = f(done...);
            Py_END_ALLOW_THREADS
            return true;
        } else {
            using T = std::tuple_element_t<sizeof...(Done), std::tuple<All...>>;
            T v;
            if (!Arg<T>::get(a[sizeof...(Done)], sizeof...(Done) + 1 == sizeof...(All), &v)) return false;
            return run(f, a, rc, done..., v);
        }
    }
};

template <class... A>
PyObject* invoke(int (*f)(A...), const char* name, PyObject* const* args, Py_ssize_t n) {
    if (!f) return PyErr_Format(PyExc_RuntimeError, "%s: the library is not loaded", name);
    if (n != static_cast<Py_ssize_t>(sizeof...(A)))
        return PyErr_Format(PyExc_TypeError, "%s takes %d arguments, %zd given", name, static_cast<int>(sizeof...(A)), n);
    int rc = 0;
    if (!Caller<int, A...>::run(f, args, &rc)) return nullptr;
    return PyLong_FromLong(rc);
}

// clang-format off
#define SVIP_ENTRY_POINTS(X) \
    X(draft_step) X(draft_step_masked) X(draft_step_at) X(draft_step_filtered) X(draft_step_truncated) X(row_threshold) \
    X(policy_advance) X(policy_update) X(pack_ragged) X(verify) X(verify_early_exit) X(verify_filtered) X(verify_tree) \
    X(vp_partial) X(vp_combine) X(vp_locate) X(pair_stats) X(pair_stats_given)

#define X(name) \
    decltype(&svip_##name) f_##name; \
    PyObject* py_##name(PyObject*, PyObject* const* args, Py_ssize_t n) { return invoke(f_##name, #name, args, n); }
SVIP_ENTRY_POINTS(X)
#undef X

// graph_launch takes the graph handle in place of a context
decltype(&svip_graph_launch) f_graph_launch;
PyObject* py_graph_launch(PyObject*, PyObject* const* args, Py_ssize_t n) { return invoke(f_graph_launch, "graph_launch", args, n); }

// load({name: address}): the library's functions
PyObject* py_load(PyObject*, PyObject* table) {
    if (!PyDict_Check(table)) { PyErr_SetString(PyExc_TypeError, "a dict of addresses is wanted"); return nullptr; }
#define X(name) \
    if (PyObject* v = PyDict_GetItemString(table, #name)) f_##name = reinterpret_cast<decltype(f_##name)>(PyLong_AsVoidPtr(v));
    SVIP_ENTRY_POINTS(X)
    X(graph_launch)
#undef X
    if (PyErr_Occurred()) return nullptr;
    Py_RETURN_NONE;
}

PyMethodDef g_methods[] = {
#define X(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)(void)>(py_##name)), METH_FASTCALL, nullptr},
    SVIP_ENTRY_POINTS(X)
    X(graph_launch)
#undef X
    {"load", py_load, METH_O, nullptr},
    {nullptr, nullptr, 0, nullptr}};
// clang-format on

PyModuleDef g_module = {PyModuleDef_HEAD_INIT, "native_calls", nullptr, -1, g_methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

#ifndef SVIP_ABI_FINGERPRINT
#define SVIP_ABI_FINGERPRINT ""
#endif

PyMODINIT_FUNC PyInit_native_calls(void) {
    g_data_ptr = PyUnicode_InternFromString("data_ptr");
    g_cuda_stream = PyUnicode_InternFromString("cuda_stream");
    if (!g_data_ptr || !g_cuda_stream) return nullptr;
    PyObject* m = PyModule_Create(&g_module);
    // the function types above are those of the header this was compiled with; binding.py compares
    if (m && PyModule_AddStringConstant(m, "abi_fingerprint", SVIP_ABI_FINGERPRINT) < 0) { Py_DECREF(m); return nullptr; }
    return m;
}
