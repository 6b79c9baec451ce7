// Native callers of the C ABI for the Python binding: the entry points that a decode step calls, without ctypes in between.
// What bounds a small op-level call is the host: ctypes takes 2 - 4 us to marshal the 17 to 20 arguments of such a call, a
// function below well under one.  The functions are bound by address to the library that the binding has loaded; argument
// types come from include/trj.h at compile time.  The GIL is released during a call, as ctypes does.
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>
#include <string.h>
#include <tuple>
#include <type_traits>
#include <utility>
#include "trj.h"

namespace {

// None, an address, or (for memory that is only read) a bytes object.
template <typename T>
bool convert(PyObject* o, T*& out) {
    if (o == Py_None) { out = nullptr; return true; }
    if (PyLong_Check(o)) {
        out = (T*)PyLong_AsVoidPtr(o);
        return out != nullptr || !PyErr_Occurred();
    }
    if (std::is_const<T>::value && PyBytes_Check(o)) { out = (T*)PyBytes_AS_STRING(o); return true; }
    PyErr_Format(PyExc_TypeError, "expected an address, got %.80s", Py_TYPE(o)->tp_name);
    return false;
}
bool convert(PyObject* o, int32_t& out) {
    const long v = PyLong_AsLong(o);
    if (v == -1 && PyErr_Occurred()) return false;
    if (v != (long)(int32_t)v) { PyErr_SetString(PyExc_OverflowError, "does not fit 32 bits"); return false; }
    out = (int32_t)v;
    return true;
}
bool convert(PyObject* o, size_t& out) {
    out = PyLong_AsSize_t(o);
    return out != (size_t)-1 || !PyErr_Occurred();
}

template <typename F> struct Caller;
template <typename R, typename... A>
struct Caller<R (*)(A...)> {
    template <size_t... I>
    static PyObject* go(R (*fn)(A...), PyObject* const* args, std::index_sequence<I...>) {
        std::tuple<A...> a;
        if (!(convert(args[I], std::get<I>(a)) && ...)) return nullptr;
        long r;
        Py_BEGIN_ALLOW_THREADS
        r = (long)fn(std::get<I>(a)...);
        Py_END_ALLOW_THREADS
        return PyLong_FromLong(r);
    }
    static PyObject* call(PyObject* self, PyObject* const* args, Py_ssize_t n) {
        if (n != (Py_ssize_t)sizeof...(A)) return PyErr_Format(PyExc_TypeError, "expected %d arguments, got %d", (int)sizeof...(A), (int)n);
        return go((R (*)(A...))PyCapsule_GetPointer(self, nullptr), args, std::index_sequence_for<A...>());
    }
};
#define ENTRY(name) {#name, (PyCFunction)(void (*)(void))Caller<decltype(&name)>::call, METH_FASTCALL, nullptr}
PyMethodDef entries[] = {
    ENTRY(trj_tree_attention_gqa), ENTRY(trj_argmax_accept), ENTRY(trj_topk_accept), ENTRY(trj_verify_step), ENTRY(trj_node_topk),
    ENTRY(trj_accept), ENTRY(trj_compact_kv), ENTRY(trj_step_host), ENTRY(trj_retrieve), ENTRY(trj_refill_window),
};

// bind(name, address): the caller of one entry point, None if this module has none for it.
PyObject* bind(PyObject*, PyObject* args) {
    const char* name;
    unsigned long long address;
    if (!PyArg_ParseTuple(args, "sK", &name, &address)) return nullptr;
    for (PyMethodDef& e : entries)
        if (strcmp(e.ml_name, name) == 0) {
            PyObject* self = PyCapsule_New((void*)(uintptr_t)address, nullptr, nullptr);
            if (!self) return nullptr;
            PyObject* f = PyCFunction_New(&e, self);
            Py_DECREF(self);
            return f;
        }
    Py_RETURN_NONE;
}

// pointer(tensor, dtype): the address behind a contiguous CUDA tensor of that type, None for anything else.
PyObject *s_is_cuda, *s_dtype, *s_is_contiguous, *s_data_ptr;
int holds(PyObject* t, PyObject* name, PyObject* want) {
    PyObject* got = PyObject_GetAttr(t, name);
    if (!got) { PyErr_Clear(); return 0; }
    Py_DECREF(got);
    return got == want;
}
PyObject* pointer(PyObject*, PyObject* const* args, Py_ssize_t n) {
    if (n != 2) return PyErr_Format(PyExc_TypeError, "expected 2 arguments");
    if (!holds(args[0], s_is_cuda, Py_True) || !holds(args[0], s_dtype, args[1])) Py_RETURN_NONE;
    PyObject* contiguous = PyObject_CallMethodNoArgs(args[0], s_is_contiguous);
    if (!contiguous) return nullptr;
    Py_DECREF(contiguous);
    if (contiguous != Py_True) Py_RETURN_NONE;
    return PyObject_CallMethodNoArgs(args[0], s_data_ptr);
}

PyMethodDef methods[] = {{"bind", bind, METH_VARARGS, nullptr},
                         {"pointer", (PyCFunction)(void (*)(void))pointer, METH_FASTCALL, nullptr},
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_calls", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__calls(void) {
    s_is_cuda = PyUnicode_InternFromString("is_cuda");
    s_dtype = PyUnicode_InternFromString("dtype");
    s_is_contiguous = PyUnicode_InternFromString("is_contiguous");
    s_data_ptr = PyUnicode_InternFromString("data_ptr");
    return s_is_cuda && s_dtype && s_is_contiguous && s_data_ptr ? PyModule_Create(&module) : nullptr;
}
