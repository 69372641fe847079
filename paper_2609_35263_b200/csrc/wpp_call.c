/* The calls a stage makes once per layer, marshalled in C: a Python module `_wpp_call` whose functions take what the binding's
 * functions take and hand it to the library.  Through ctypes the fourteen to eighteen arguments of a call cost about as much
 * host time as its launches.  An argument that is memory is None (null) or an object with data_ptr(); a description is a
 * ctypes structure.  The library's functions come from the loaded libwpp.so (init), so that this module links to nothing. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>

#include "../../include/wpp.h"

static int (*p_append)(const wpp_ctx*, const wpp_batch_desc*, const void*, const void*, void*, void*, const int32_t*, const int32_t*,
                       const int32_t*, const void*, const void*, int32_t*, void*);
static int (*p_attention)(const wpp_ctx*, const wpp_batch_desc*, const void*, void*, float*, const void*, const void*, const int32_t*,
                          const int32_t*, const int32_t*, const void*, const void*, void*, size_t, int32_t*, void*);
static int (*p_kda)(const wpp_ctx*, const wpp_kda_desc*, const void*, const void*, const void*, const float*, const float*,
                    const int64_t*, const int32_t*, float*, const int32_t*, const int32_t*, const int32_t*, void*, void*, size_t,
                    int32_t*, void*);
static PyObject* s_data_ptr;

/* 0, or -1 with an exception set */
static int address(PyObject* o, void** out) {
    *out = NULL;
    if (o == Py_None) return 0;
    PyObject* v;
    if (PyLong_Check(o)) {
        v = o;
        Py_INCREF(v);
    } else {
        v = PyObject_CallMethodNoArgs(o, s_data_ptr);
        if (!v) return -1;
    }
    *out = PyLong_AsVoidPtr(v);
    Py_DECREF(v);
    return *out == NULL && PyErr_Occurred() ? -1 : 0;
}
static int addresses(PyObject* const* args, int n, void** out) {
    for (int i = 0; i < n; ++i)
        if (address(args[i], &out[i])) return -1;
    return 0;
}
/* copies a ctypes structure: what the caller does with it while the call runs without the interpreter lock is the caller's */
static int description(PyObject* o, void* out, Py_ssize_t size) {
    Py_buffer b;
    if (PyObject_GetBuffer(o, &b, PyBUF_SIMPLE)) return -1;
    if (b.len != size) {
        PyBuffer_Release(&b);
        PyErr_SetString(PyExc_TypeError, "description of another size");
        return -1;
    }
    memcpy(out, b.buf, (size_t)size);
    PyBuffer_Release(&b);
    return 0;
}
static int count(PyObject* const* args, Py_ssize_t n, Py_ssize_t want) {
    (void)args;
    if (n == want) return 0;
    PyErr_Format(PyExc_TypeError, "%zd arguments instead of %zd", n, want);
    return -1;
}

/* kv_append(ctx, desc, k_new, v_new, k_cache, v_cache, tables, prefix, chunks, plan_host, plan_dev, status, stream) */
static PyObject* kv_append(PyObject* self, PyObject* const* args, Py_ssize_t n) {
    (void)self;
    void *ctx, *a[11];
    wpp_batch_desc d;
    if (count(args, n, 13) || address(args[0], &ctx) || description(args[1], &d, sizeof(d)) || addresses(args + 2, 11, a)) return NULL;
    int st;
    Py_BEGIN_ALLOW_THREADS
    st = p_append(ctx, &d, a[0], a[1], a[2], a[3], a[4], a[5], a[6], a[7], a[8], a[9], a[10]);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(st);
}

/* attention(ctx, desc, q, out, lse, k_cache, v_cache, tables, prefix, chunks, plan_host, plan_dev, workspace, bytes, status, stream) */
static PyObject* attention(PyObject* self, PyObject* const* args, Py_ssize_t n) {
    (void)self;
    void *ctx, *a[11], *b[2];
    wpp_batch_desc d;
    if (count(args, n, 16) || address(args[0], &ctx) || description(args[1], &d, sizeof(d)) || addresses(args + 2, 11, a)) return NULL;
    const size_t bytes = PyLong_AsSize_t(args[13]);
    if ((bytes == (size_t)-1 && PyErr_Occurred()) || addresses(args + 14, 2, b)) return NULL;
    int st;
    Py_BEGIN_ALLOW_THREADS
    st = p_attention(ctx, &d, a[0], a[1], a[2], a[3], a[4], a[5], a[6], a[7], a[8], a[9], a[10], bytes, b[0], b[1]);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(st);
}

/* kda_chunk(ctx, desc, q, k, v, alpha, beta, rows, prefix, pool, state_in, state_out, snaps, out, workspace, bytes, status, stream) */
static PyObject* kda_chunk(PyObject* self, PyObject* const* args, Py_ssize_t n) {
    (void)self;
    void *ctx, *a[13], *b[2];
    wpp_kda_desc d;
    if (count(args, n, 18) || address(args[0], &ctx) || description(args[1], &d, sizeof(d)) || addresses(args + 2, 13, a)) return NULL;
    const size_t bytes = PyLong_AsSize_t(args[15]);
    if ((bytes == (size_t)-1 && PyErr_Occurred()) || addresses(args + 16, 2, b)) return NULL;
    int st;
    Py_BEGIN_ALLOW_THREADS
    st = p_kda(ctx, &d, a[0], a[1], a[2], a[3], a[4], a[5], a[6], a[7], a[8], a[9], a[10], a[11], a[12], bytes, b[0], b[1]);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(st);
}

/* init(append, attention, kda): the functions' addresses in the loaded library */
static PyObject* init(PyObject* self, PyObject* const* args, Py_ssize_t n) {
    (void)self;
    void* a[3];
    if (count(args, n, 3) || addresses(args, 3, a)) return NULL;
    memcpy(&p_append, &a[0], sizeof(void*));
    memcpy(&p_attention, &a[1], sizeof(void*));
    memcpy(&p_kda, &a[2], sizeof(void*));
    Py_RETURN_NONE;
}

static PyMethodDef methods[] = {
    {"init", (PyCFunction)(void (*)(void))init, METH_FASTCALL, NULL},
    {"kv_append", (PyCFunction)(void (*)(void))kv_append, METH_FASTCALL, NULL},
    {"attention", (PyCFunction)(void (*)(void))attention, METH_FASTCALL, NULL},
    {"kda_chunk", (PyCFunction)(void (*)(void))kda_chunk, METH_FASTCALL, NULL},
    {NULL, NULL, 0, NULL},
};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_wpp_call", NULL, -1, methods, NULL, NULL, NULL, NULL};
PyMODINIT_FUNC PyInit__wpp_call(void) {
    s_data_ptr = PyUnicode_InternFromString("data_ptr");
    return s_data_ptr ? PyModule_Create(&module) : NULL;
}
