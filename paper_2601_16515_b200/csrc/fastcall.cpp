// Python's way into the entry points that a layer calls on every step: the same functions of libsalad as through ctypes,
// with their arguments converted here by their C++ types instead of by ctypes' interpreter (a call with its 21 arguments
// costs 0.2 us instead of 2.5, of the 15 us that the host spends on the smallest fused call).  Addresses come from the
// loaded library (bind), so nothing is linked.  What these conversions do not take (anything but plain integers, floats
// and None) they leave to ctypes: the answer is None then and nothing has been called.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <stddef.h>
#include <stdint.h>
#include <string.h>

#include <tuple>
#include <type_traits>
#include <utility>

#include "../../include/salad.h"

namespace {

template <typename T>
T convert(PyObject* o, bool& bad) {
    if constexpr (std::is_pointer_v<T>) {
        if (o == Py_None) return nullptr;
        if (!PyLong_CheckExact(o)) { bad = true; return nullptr; }
        const unsigned long long v = PyLong_AsUnsignedLongLongMask(o);
        return reinterpret_cast<T>(static_cast<uintptr_t>(v));
    } else if constexpr (std::is_floating_point_v<T>) {
        if (!PyFloat_CheckExact(o)) { bad = true; return T(0); }
        return static_cast<T>(PyFloat_AS_DOUBLE(o));
    } else {
        if (!PyLong_CheckExact(o)) { bad = true; return T(0); }
        return static_cast<T>(PyLong_AsUnsignedLongLongMask(o));        // as many low bits as the type has, like ctypes
    }
}

template <typename... A, size_t... I>
PyObject* call_with(int (*fn)(A...), PyObject* const* args, std::index_sequence<I...>) {
    bool bad = false;
    std::tuple<A...> values{convert<A>(args[I], bad)...};
    if (bad) { PyErr_Clear(); Py_RETURN_NONE; }
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = fn(std::get<I>(values)...);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

template <typename... A>
PyObject* call(int (*fn)(A...), PyObject* const* args, Py_ssize_t n) {
    if (!fn || n != Py_ssize_t(sizeof...(A))) Py_RETURN_NONE;
    return call_with(fn, args, std::index_sequence_for<A...>{});
}

#define SALAD_FAST(X) \
    X(salad_fused_fwd) X(salad_fused_drop_fwd) X(salad_sparse_attn_fwd) X(salad_linear_attn_fwd) X(salad_linear_state_fwd) \
    X(salad_fused_prepared_fwd) X(salad_fused_rope_fwd) X(salad_linear_attn_rope_fwd) X(salad_fused_proj_fwd) \
    X(salad_topk_mask_build) X(salad_dynamic_scale) X(salad_proj_combine_fwd) X(salad_fused_stswa_fwd)

#define X(name) \
    decltype(&name) g_##name = nullptr; \
    PyObject* py_##name(PyObject*, PyObject* const* args, Py_ssize_t n) { return call(g_##name, args, n); }
SALAD_FAST(X)
#undef X

// bind(name, address): whether there is such a function
PyObject* py_bind(PyObject*, PyObject* args) {
    const char* name = nullptr;
    unsigned long long address = 0;
    if (!PyArg_ParseTuple(args, "sK", &name, &address)) return nullptr;
#define X(fn) \
    if (strcmp(name, #fn) == 0) { g_##fn = reinterpret_cast<decltype(&fn)>(static_cast<uintptr_t>(address)); Py_RETURN_TRUE; }
    SALAD_FAST(X)
#undef X
    Py_RETURN_FALSE;
}

PyMethodDef methods[] = {
#define X(fn) {#fn, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(py_##fn)), METH_FASTCALL, nullptr},
    SALAD_FAST(X)
#undef X
    {"bind", py_bind, METH_VARARGS, nullptr},
    {nullptr, nullptr, 0, nullptr}};

PyModuleDef module = {PyModuleDef_HEAD_INIT, "_fastcall", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__fastcall() { return PyModule_Create(&module); }
