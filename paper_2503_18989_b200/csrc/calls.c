/* The binding's calls of every layer of a step as a CPython extension: what the ctypes declarations in binding.py do, without their cost
 * per argument.  libhat.so is loaded by binding.py, which hands the entry points' addresses to init(). */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>

#include "../../include/hat.h"

typedef int (*attention_fn)(const hat_cache_desc*, const hat_plan*, const void*, const void*, const void*, void*, float*, float, void*, size_t, void*);
static attention_fn g_attention, g_attention_out16;
static PyObject *g_data_ptr, *g_ctypes, *g_data, *g_handle, *g_plan_type, *g_cache_type;

/* Raw address of a torch tensor, numpy array, int or None */
static int address(PyObject* x, void** out) {
    if (x == Py_None) { *out = NULL; return 0; }
    PyObject* v;
    if (PyLong_Check(x)) {
        Py_INCREF(x);
        v = x;
    } else {
        v = PyObject_CallMethodNoArgs(x, g_data_ptr);
        if (!v) {
            if (!PyErr_ExceptionMatches(PyExc_AttributeError)) return -1;
            PyErr_Clear();
            PyObject* c = PyObject_GetAttr(x, g_ctypes);
            if (!c) return -1;
            v = PyObject_GetAttr(c, g_data);
            Py_DECREF(c);
            if (!v) return -1;
            if (v == Py_None) { Py_DECREF(v); *out = NULL; return 0; }
        }
    }
    *out = PyLong_AsVoidPtr(v);
    Py_DECREF(v);
    return *out == NULL && PyErr_Occurred() ? -1 : 0;
}

/* A handle (the plan's, a stream's): an int or None; 1 for anything else, whose memory is not what the library wants there */
static int handle(PyObject* x, void** out) {
    if (x == Py_None) { *out = NULL; return 0; }
    if (!PyLong_Check(x)) return 1;
    *out = PyLong_AsVoidPtr(x);
    return *out == NULL && PyErr_Occurred() ? -1 : 0;
}

static int plan_address(PyObject* plan, void** out) {
    const int owned = PyObject_IsInstance(plan, g_plan_type);
    if (owned < 0) return -1;
    if (!owned) return handle(plan, out);
    PyObject* h = PyObject_GetAttr(plan, g_handle);
    if (!h) return -1;
    const int r = handle(h, out);
    Py_DECREF(h);
    return r;
}

static int number(PyObject* x, size_t* out) {
    if (!PyLong_Check(x)) return 1;
    *out = (size_t)PyLong_AsUnsignedLongLongMask(x);
    return *out == (size_t)-1 && PyErr_Occurred() ? -1 : 0;
}

/* (cache, plan, q, k_new, v_new, out, lse, sm_scale, workspace, workspace_bytes, stream) -> status, or None for arguments that only
 * ctypes takes, or refuses (its objects as pointers, wrong types) */
static PyObject* attention(attention_fn fn, PyObject* const* a, Py_ssize_t n) {
    void *plan, *p[5], *ws, *stream = NULL;
    size_t ws_bytes;
    Py_buffer cache;                                         /* the descriptor's own memory */
    if (n != 11 || !fn || PyObject_IsInstance(a[0], g_cache_type) != 1 || plan_address(a[1], &plan)) goto other;
    for (int i = 0; i < 5; ++i)
        if (address(a[2 + i], &p[i])) goto other;
    const double scale = PyFloat_AsDouble(a[7]);
    if ((scale == -1.0 && PyErr_Occurred()) || address(a[8], &ws) || number(a[9], &ws_bytes) || handle(a[10], &stream)) goto other;
    if (PyObject_GetBuffer(a[0], &cache, PyBUF_SIMPLE)) goto other;
    if (cache.len != (Py_ssize_t)sizeof(hat_cache_desc)) { PyBuffer_Release(&cache); goto other; }
    int status;
    Py_BEGIN_ALLOW_THREADS
    status = fn((const hat_cache_desc*)cache.buf, (const hat_plan*)plan, p[0], p[1], p[2], p[3], (float*)p[4], (float)scale, ws, ws_bytes, stream);
    Py_END_ALLOW_THREADS
    PyBuffer_Release(&cache);
    return PyLong_FromLong(status);
other:
    PyErr_Clear();
    Py_RETURN_NONE;
}
static PyObject* chunk_attention(PyObject* self, PyObject* const* a, Py_ssize_t n) { (void)self; return attention(g_attention, a, n); }
static PyObject* chunk_attention_out16(PyObject* self, PyObject* const* a, Py_ssize_t n) { (void)self; return attention(g_attention_out16, a, n); }

/* (address of hat_chunk_attention, of hat_chunk_attention_out16, the binding's Plan and hat_cache_desc classes) */
static PyObject* init(PyObject* self, PyObject* const* a, Py_ssize_t n) {
    (void)self;
    if (n != 4) { PyErr_SetString(PyExc_TypeError, "4 arguments are expected"); return NULL; }
    void* f[2];
    for (int i = 0; i < 2; ++i)
        if (address(a[i], &f[i])) return NULL;
    g_attention = (attention_fn)(uintptr_t)f[0];
    g_attention_out16 = (attention_fn)(uintptr_t)f[1];
    Py_INCREF(a[2]);
    Py_INCREF(a[3]);
    Py_XSETREF(g_plan_type, a[2]);
    Py_XSETREF(g_cache_type, a[3]);
    Py_RETURN_NONE;
}

static PyMethodDef methods[] = {{"init", (PyCFunction)(void (*)(void))init, METH_FASTCALL, NULL},
                                {"chunk_attention", (PyCFunction)(void (*)(void))chunk_attention, METH_FASTCALL, NULL},
                                {"chunk_attention_out16", (PyCFunction)(void (*)(void))chunk_attention_out16, METH_FASTCALL, NULL},
                                {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_calls", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__calls(void) {
    g_data_ptr = PyUnicode_InternFromString("data_ptr");
    g_ctypes = PyUnicode_InternFromString("ctypes");
    g_data = PyUnicode_InternFromString("data");
    g_handle = PyUnicode_InternFromString("handle");
    if (!g_data_ptr || !g_ctypes || !g_data || !g_handle) return NULL;
    return PyModule_Create(&module);
}
