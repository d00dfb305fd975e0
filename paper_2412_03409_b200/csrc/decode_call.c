/* prefixkv_decode_attn as a Python function: the arguments of one decode call taken from their objects without ctypes.
 *
 * A model that calls the library once per layer and token is bound by the host where its cache is small: 5.5 us a call
 * through ctypes, of which 2.8 in the library (the launch), against 4.3 on the device (32 heads, 128 rows).
 * The conversions are the ones ctypes made: None is a null pointer, a tensor gives its data_ptr(), and whole
 * numbers are taken as int() takes them, to 32 bits.  The interpreter lock is released for the call, as ctypes does.
 */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stddef.h>
#include <stdint.h>

#include "prefixkv.h"

typedef int (*decode_fn)(const pkv_shape *, pkv_cache *, const void *, const void *, const void *, const float *, int32_t,
                         int32_t, void *, int32_t *, void *, size_t, void *);

static decode_fn g_decode;
static PyObject *g_stream;   /* callable: the current stream's handle on a device ... */
static PyObject *g_device;   /* ... which this one gives; NULL: g_stream takes no argument */
static PyObject *s_data_ptr, *s_numel;

static int pointer_of(PyObject *o, void **p)
{
    PyObject *r;
    if (o == Py_None) {
        *p = NULL;
        return 0;
    }
    r = PyObject_CallMethodNoArgs(o, s_data_ptr);
    if (!r) return -1;
    *p = PyLong_AsVoidPtr(r);
    Py_DECREF(r);
    return *p == NULL && PyErr_Occurred() ? -1 : 0;
}

static int int32_of(PyObject *o, int32_t *v)
{
    PyObject *r = PyLong_CheckExact(o) ? Py_NewRef(o) : PyNumber_Long(o);
    if (!r) return -1;
    *v = (int32_t)PyLong_AsUnsignedLongMask(r);
    Py_DECREF(r);
    return PyErr_Occurred() ? -1 : 0;
}

static int current_stream(void **p)
{
    PyObject *d, *r;
    if (g_device) {
        d = PyObject_CallNoArgs(g_device);
        if (!d) return -1;
        r = PyObject_CallOneArg(g_stream, d);
        Py_DECREF(d);
    } else {
        r = PyObject_CallNoArgs(g_stream);
    }
    if (!r) return -1;
    *p = PyLong_AsVoidPtr(r);
    Py_DECREF(r);
    return *p == NULL && PyErr_Occurred() ? -1 : 0;
}

/* shape, cache (ctypes structures), q, k_new, v_new, layer_scale, layer_begin, layer_end, out, dev_status, ws -> status */
static PyObject *decode_attn(PyObject *self, PyObject *const *args, Py_ssize_t nargs)
{
    Py_buffer shape, cache;
    void *q, *k, *v, *scale, *out, *status, *ws, *stream;
    int32_t lb, le;
    size_t ws_bytes = 0;
    int rc;
    (void)self;
    if (nargs != 11 || !g_decode) {
        PyErr_SetString(PyExc_TypeError, "decode_attn takes 11 arguments, after bind()");
        return NULL;
    }
    if (pointer_of(args[2], &q) || pointer_of(args[3], &k) || pointer_of(args[4], &v) || pointer_of(args[5], &scale) ||
        int32_of(args[6], &lb) || int32_of(args[7], &le) || pointer_of(args[8], &out) || pointer_of(args[9], &status) ||
        pointer_of(args[10], &ws) || current_stream(&stream))
        return NULL;
    if (args[10] != Py_None) {
        PyObject *n = PyObject_CallMethodNoArgs(args[10], s_numel);
        if (!n) return NULL;
        ws_bytes = PyLong_AsSize_t(n);
        Py_DECREF(n);
        if (PyErr_Occurred()) return NULL;
    }
    if (PyObject_GetBuffer(args[0], &shape, PyBUF_SIMPLE)) return NULL;
    if (PyObject_GetBuffer(args[1], &cache, PyBUF_WRITABLE)) {
        PyBuffer_Release(&shape);
        return NULL;
    }
    if (shape.len < (Py_ssize_t)sizeof(pkv_shape) || cache.len < (Py_ssize_t)sizeof(pkv_cache)) {
        PyBuffer_Release(&cache);
        PyBuffer_Release(&shape);
        PyErr_SetString(PyExc_TypeError, "shape and cache must be the binding's structures");
        return NULL;
    }
    Py_BEGIN_ALLOW_THREADS
    rc = g_decode((const pkv_shape *)shape.buf, (pkv_cache *)cache.buf, q, k, v, (const float *)scale, lb, le, out,
                  (int32_t *)status, ws, ws_bytes, stream);
    Py_END_ALLOW_THREADS
    PyBuffer_Release(&cache);
    PyBuffer_Release(&shape);
    return PyLong_FromLong(rc);
}

/* address of prefixkv_decode_attn, stream callable, device callable or None */
static PyObject *bind_library(PyObject *self, PyObject *args)
{
    PyObject *address, *stream, *device;
    void *p;
    (void)self;
    if (!PyArg_ParseTuple(args, "OOO", &address, &stream, &device)) return NULL;
    p = PyLong_AsVoidPtr(address);
    if (!p) {
        if (!PyErr_Occurred()) PyErr_SetString(PyExc_ValueError, "null function address");
        return NULL;
    }
    Py_XSETREF(g_stream, Py_NewRef(stream));
    Py_XSETREF(g_device, device == Py_None ? NULL : Py_NewRef(device));
    g_decode = (decode_fn)(uintptr_t)p;
    Py_RETURN_NONE;
}

static PyMethodDef methods[] = {
    {"bind", bind_library, METH_VARARGS, NULL},
    {"decode_attn", (PyCFunction)(void (*)(void))decode_attn, METH_FASTCALL, NULL},
    {NULL, NULL, 0, NULL},
};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_decode_call", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__decode_call(void)
{
    s_data_ptr = PyUnicode_InternFromString("data_ptr");
    s_numel = PyUnicode_InternFromString("numel");
    if (!s_data_ptr || !s_numel) return NULL;
    return PyModule_Create(&module);
}
