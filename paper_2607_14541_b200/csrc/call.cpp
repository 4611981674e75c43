// Calls of C entry points from Python: bind(address, n_args) gives a callable that passes whole numbers, None
// (a null pointer) and buffers (their address) as 64-bit words and returns the C function's int.
//
// A small call of this library is host time: through ctypes one with four arguments takes about 0.5 us for their
// conversion, and an array's address another 1 us; here the whole crossing takes about 0.1 us.  The interpreter
// lock is given up during the call, as ctypes does.  (Every parameter behind these entry points is an integer or
// a pointer, each passed in a 64-bit register or stack word on this platform; a narrower one reads its low bits.)
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <cstdint>

namespace {

constexpr Py_ssize_t MAX_ARGS = 12;
using W = uint64_t;

struct Target {
    void* function;
    Py_ssize_t n_args;
};
const char* const CAPSULE = "atrex_call_target";

int invoke(const Target& t, const W* a) {
    void* f = t.function;
    switch (t.n_args) {
        case 1: return ((int (*)(W))f)(a[0]);
        case 2: return ((int (*)(W, W))f)(a[0], a[1]);
        case 3: return ((int (*)(W, W, W))f)(a[0], a[1], a[2]);
        case 4: return ((int (*)(W, W, W, W))f)(a[0], a[1], a[2], a[3]);
        case 5: return ((int (*)(W, W, W, W, W))f)(a[0], a[1], a[2], a[3], a[4]);
        case 6: return ((int (*)(W, W, W, W, W, W))f)(a[0], a[1], a[2], a[3], a[4], a[5]);
        default:
            return ((int (*)(W, W, W, W, W, W, W, W, W, W, W, W))f)(a[0], a[1], a[2], a[3], a[4], a[5], a[6], a[7], a[8], a[9], a[10], a[11]);
    }
}

PyObject* call(PyObject* self, PyObject* const* args, Py_ssize_t n) {
    const Target* t = (const Target*)PyCapsule_GetPointer(self, CAPSULE);
    if (!t) return nullptr;
    if (n != t->n_args) return PyErr_Format(PyExc_TypeError, "%zd arguments expected, %zd given", t->n_args, n);
    W a[MAX_ARGS];
    Py_buffer view[MAX_ARGS];
    Py_ssize_t n_views = 0;
    bool ok = true;
    for (Py_ssize_t i = 0; i < n && ok; ++i) {
        if (PyLong_Check(args[i])) {
            a[i] = PyLong_AsUnsignedLongLongMask(args[i]);
            ok = !(a[i] == ~(W)0 && PyErr_Occurred());
        } else if (args[i] == Py_None) {
            a[i] = 0;
        } else if (PyObject_CheckBuffer(args[i])) {
            ok = PyObject_GetBuffer(args[i], &view[n_views], PyBUF_SIMPLE) == 0;
            if (ok) a[i] = (W)(uintptr_t)view[n_views++].buf;
        } else {
            PyErr_SetString(PyExc_TypeError, "an argument is neither a whole number, None nor a buffer");
            ok = false;
        }
    }
    int rc = 0;
    if (ok) {
        Py_BEGIN_ALLOW_THREADS
        rc = invoke(*t, a);
        Py_END_ALLOW_THREADS
    }
    while (n_views > 0) PyBuffer_Release(&view[--n_views]);
    return ok ? PyLong_FromLong(rc) : nullptr;
}

PyMethodDef g_call = {"call", (PyCFunction)(void (*)(void))call, METH_FASTCALL, "the C entry point that bind() was given"};

void forget(PyObject* capsule) { delete (Target*)PyCapsule_GetPointer(capsule, CAPSULE); }

PyObject* bind(PyObject*, PyObject* args) {
    unsigned long long address;
    Py_ssize_t n_args;
    if (!PyArg_ParseTuple(args, "Kn", &address, &n_args)) return nullptr;
    if (address == 0 || !((n_args >= 1 && n_args <= 6) || n_args == MAX_ARGS)) {
        PyErr_SetString(PyExc_ValueError, "bind: an address and 1 to 6 or 12 arguments");
        return nullptr;
    }
    Target* t = new Target{(void*)(uintptr_t)address, n_args};
    PyObject* capsule = PyCapsule_New(t, CAPSULE, forget);
    if (!capsule) {
        delete t;
        return nullptr;
    }
    PyObject* f = PyCFunction_New(&g_call, capsule);
    Py_DECREF(capsule);
    return f;
}

PyMethodDef g_methods[] = {{"bind", bind, METH_VARARGS, "bind(address, n_args) -> callable"}, {nullptr, nullptr, 0, nullptr}};
PyModuleDef g_module = {PyModuleDef_HEAD_INIT, "_call", "calls of C entry points", -1, g_methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__call() { return PyModule_Create(&g_module); }
