/* The calls a stage makes once per layer, marshalled in C: a Python module `_wpp_call` whose functions take what the binding's
 * functions take and hand it to the library.  Through ctypes the fourteen to eighteen arguments of a call cost about as much
 * host time as its launches.  An argument that is memory is None (null) or an object with data_ptr(), never an integer; a
 * description is an instance of the binding's ctypes structure; contexts and streams are integers.  The library's functions
 * come from the loaded libwpp.so (init), so that this module links to nothing. */
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
static PyObject *s_data_ptr, *t_batch, *t_kda;         /* the method's name; the binding's BatchDesc and KdaDesc */

/* Each of these returns 0, or -1 with an exception set. */
static int integer(PyObject* o, void** out) {           /* a context, a stream, a function: None is null */
    *out = o == Py_None ? NULL : PyLong_AsVoidPtr(o);
    return *out == NULL && PyErr_Occurred() ? -1 : 0;
}
static int memory(PyObject* o, void** out) {            /* what has no data_ptr() raises AttributeError, an integer too */
    *out = NULL;
    PyObject* v = PyObject_CallMethodNoArgs(o, s_data_ptr);
    if (!v) return -1;
    if (PyLong_Check(v)) *out = PyLong_AsVoidPtr(v);
    else PyErr_SetString(PyExc_TypeError, "data_ptr() is not an integer");
    Py_DECREF(v);
    return *out == NULL && PyErr_Occurred() ? -1 : 0;
}
static int memories(PyObject* const* args, int n, void** out) {         /* None is null */
    for (int i = 0; i < n; ++i) {
        out[i] = NULL;
        if (args[i] != Py_None && memory(args[i], &out[i])) return -1;
    }
    return 0;
}
/* copies a ctypes structure: what the caller does with it while the call runs without the interpreter lock is the caller's */
static int description(PyObject* o, PyObject* type, void* out, Py_ssize_t size) {
    const int is = PyObject_IsInstance(o, type);
    if (is < 0) return -1;
    if (!is) {
        PyErr_Format(PyExc_TypeError, "a description has to be a %s, not %.100s", ((PyTypeObject*)type)->tp_name, Py_TYPE(o)->tp_name);
        return -1;
    }
    Py_buffer b;
    if (PyObject_GetBuffer(o, &b, PyBUF_SIMPLE)) return -1;
    if (b.len >= size) memcpy(out, b.buf, (size_t)size);      /* (a subclass may have fields of its own behind) */
    else PyErr_SetString(PyExc_TypeError, "description of another size");
    const int rc = b.len >= size ? 0 : -1;
    PyBuffer_Release(&b);
    return rc;
}
static int count(Py_ssize_t n, Py_ssize_t want) {
    if (n == want) return 0;
    PyErr_Format(PyExc_TypeError, "%zd arguments instead of %zd", n, want);
    return -1;
}

/* kv_append(ctx, desc, k_new, v_new, k_cache, v_cache, tables, prefix, chunks, plan_host, plan_dev, status, stream) */
static PyObject* kv_append(PyObject* self, PyObject* const* args, Py_ssize_t n) {
    (void)self;
    void *ctx, *a[11];
    wpp_batch_desc d;
    if (count(n, 13) || integer(args[0], &ctx) || description(args[1], t_batch, &d, sizeof(d)) || memories(args + 2, 7, a) ||
        memory(args[9], &a[7]) || memories(args + 10, 2, a + 8) || integer(args[12], &a[10]))
        return NULL;
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
    if (count(n, 16) || integer(args[0], &ctx) || description(args[1], t_batch, &d, sizeof(d)) || memories(args + 2, 8, a) ||
        memory(args[10], &a[8]) || memories(args + 11, 2, a + 9))
        return NULL;
    const size_t bytes = PyLong_AsSize_t(args[13]);
    if ((bytes == (size_t)-1 && PyErr_Occurred()) || memories(args + 14, 1, b) || integer(args[15], &b[1])) return NULL;
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
    if (count(n, 18) || integer(args[0], &ctx) || description(args[1], t_kda, &d, sizeof(d)) || memories(args + 2, 13, a)) return NULL;
    const size_t bytes = PyLong_AsSize_t(args[15]);
    if ((bytes == (size_t)-1 && PyErr_Occurred()) || memories(args + 16, 1, b) || integer(args[17], &b[1])) return NULL;
    int st;
    Py_BEGIN_ALLOW_THREADS
    st = p_kda(ctx, &d, a[0], a[1], a[2], a[3], a[4], a[5], a[6], a[7], a[8], a[9], a[10], a[11], a[12], bytes, b[0], b[1]);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(st);
}

/* init(append, attention, kda, BatchDesc, KdaDesc): the functions' addresses in the loaded library, the descriptions' types */
static PyObject* init(PyObject* self, PyObject* const* args, Py_ssize_t n) {
    (void)self;
    void* a[3];
    if (count(n, 5) || integer(args[0], &a[0]) || integer(args[1], &a[1]) || integer(args[2], &a[2])) return NULL;
    if (!PyType_Check(args[3]) || !PyType_Check(args[4])) {
        PyErr_SetString(PyExc_TypeError, "the descriptions' types");
        return NULL;
    }
    memcpy(&p_append, &a[0], sizeof(void*));
    memcpy(&p_attention, &a[1], sizeof(void*));
    memcpy(&p_kda, &a[2], sizeof(void*));
    Py_XSETREF(t_batch, Py_NewRef(args[3]));
    Py_XSETREF(t_kda, Py_NewRef(args[4]));
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
