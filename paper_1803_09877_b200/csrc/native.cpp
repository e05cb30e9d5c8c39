// The calls of a training loop, marshalled natively for CPython: arguments are torch tensors (or anything with data_ptr()), addresses
// or None, as in binding.py, which uses ctypes for everything else.  A call of a library that only launches a kernel is the caller's
// time.  By ctypes / so, us a call: cyclic encode n = 15, s = 2, d = 12,000 3.84 / 3.12, n = 45, s = 5, d = 4096 5.28 / 4.42, repetition encode
// n = 15, d = 100,000 5.65 / 4.71, all on one host (others are faster throughout).
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>

#include "draco.h"

namespace {

PyObject* g_check = nullptr;          // binding._check: raises for a negative status
PyObject* g_stream = nullptr;         // binding._stream: any stream argument to a handle
PyObject* g_raw = nullptr;            // handle of a device's current stream, and the current device, once torch's are known
PyObject* g_device = nullptr;
PyObject* g_data_ptr = nullptr;       // "data_ptr"

bool address(PyObject* x, void** out) {
    if (x == Py_None) {
        *out = nullptr;
        return true;
    }
    PyObject* owned = nullptr;
    if (!PyLong_Check(x)) {
        x = owned = PyObject_CallMethodNoArgs(x, g_data_ptr);
        if (!x) return false;
    }
    *out = reinterpret_cast<void*>(static_cast<uintptr_t>(PyLong_AsUnsignedLongLongMask(x)));
    Py_XDECREF(owned);
    return !PyErr_Occurred();
}

bool stream_of(PyObject* x, void** out) {
    PyObject* handle;
    if (x == Py_None && g_raw) {
        PyObject* device = PyObject_CallNoArgs(g_device);
        if (!device) return false;
        handle = PyObject_CallOneArg(g_raw, device);
        Py_DECREF(device);
    } else {
        handle = PyObject_CallOneArg(g_stream, x);
    }
    if (!handle) return false;
    const bool ok = address(handle, out);
    Py_DECREF(handle);
    return ok;
}

// The plan, `count` addresses and, last, the stream.
bool arguments(PyObject* const* args, Py_ssize_t nargs, Py_ssize_t want, int count, void** p, void** stream) {
    if (nargs != want) {
        PyErr_Format(PyExc_TypeError, "%zd arguments, not %zd", want, nargs);
        return false;
    }
    for (int k = 0; k < count; ++k)
        if (!address(args[k], &p[k])) return false;
    return stream_of(args[nargs - 1], stream);
}

PyObject* status(int rc) {
    PyObject* value = PyLong_FromLong(rc);
    if (rc >= 0 || !value) return value;
    PyObject* result = PyObject_CallOneArg(g_check, value);
    Py_DECREF(value);
    return result;
}

#define PLAN reinterpret_cast<draco_plan*>(p[0])

PyObject* encode(PyObject*, PyObject* const* args, Py_ssize_t nargs) {
    void *p[3], *st;
    if (!arguments(args, nargs, 4, 3, p, &st)) return nullptr;
    int rc;
    Py_BEGIN_ALLOW_THREADS rc = draco_encode(PLAN, (const float*)p[1], p[2], st);
    Py_END_ALLOW_THREADS return status(rc);
}

PyObject* locate(PyObject*, PyObject* const* args, Py_ssize_t nargs) {
    void *p[4], *st;
    if (!arguments(args, nargs, 5, 4, p, &st)) return nullptr;
    int rc;
    Py_BEGIN_ALLOW_THREADS rc = draco_locate(PLAN, p[1], (const float*)p[2], (uint8_t*)p[3], st);
    Py_END_ALLOW_THREADS return status(rc);
}

PyObject* decode(PyObject*, PyObject* const* args, Py_ssize_t nargs) {
    void *p[4], *st;
    if (!arguments(args, nargs, 5, 4, p, &st)) return nullptr;
    int rc;
    Py_BEGIN_ALLOW_THREADS rc = draco_decode(PLAN, p[1], (const uint8_t*)p[2], (float*)p[3], st);
    Py_END_ALLOW_THREADS return status(rc);
}

PyObject* decode_update(PyObject*, PyObject* const* args, Py_ssize_t nargs) {
    void *p[4], *st;
    if (!arguments(args, nargs, 6, 4, p, &st)) return nullptr;
    const float scale = (float)PyFloat_AsDouble(args[4]);
    if (PyErr_Occurred()) return nullptr;
    int rc;
    Py_BEGIN_ALLOW_THREADS rc = draco_decode_update(PLAN, p[1], (const uint8_t*)p[2], (float*)p[3], scale, st);
    Py_END_ALLOW_THREADS return status(rc);
}

PyObject* locate_decode(PyObject*, PyObject* const* args, Py_ssize_t nargs) {
    void *p[5], *st;
    if (!arguments(args, nargs, 6, 5, p, &st)) return nullptr;
    int rc;
    Py_BEGIN_ALLOW_THREADS rc = draco_locate_decode(PLAN, p[1], (const float*)p[2], (uint8_t*)p[3], (float*)p[4], st);
    Py_END_ALLOW_THREADS return status(rc);
}

void keep(PyObject*& slot, PyObject* value) {
    Py_INCREF(value);
    Py_XSETREF(slot, value);
}

PyObject* set_functions(PyObject*, PyObject* args) {          // (check, stream)
    PyObject *check, *stream;
    if (!PyArg_ParseTuple(args, "OO", &check, &stream)) return nullptr;
    keep(g_check, check);
    keep(g_stream, stream);
    Py_RETURN_NONE;
}

PyObject* set_current_stream(PyObject*, PyObject* args) {     // (raw, device)
    PyObject *raw, *device;
    if (!PyArg_ParseTuple(args, "OO", &raw, &device)) return nullptr;
    keep(g_device, device);
    keep(g_raw, raw);
    Py_RETURN_NONE;
}

#define FAST(name) {#name, (PyCFunction)(void (*)(void))name, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {FAST(encode), FAST(locate), FAST(decode), FAST(decode_update), FAST(locate_decode),
                         {"set_functions", set_functions, METH_VARARGS, nullptr},
                         {"set_current_stream", set_current_stream, METH_VARARGS, nullptr},
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native(void) {
    g_data_ptr = PyUnicode_InternFromString("data_ptr");
    return g_data_ptr ? PyModule_Create(&module) : nullptr;
}
