/* The forward calls as a CPython extension module.  A one-token layer runs about as long as the host needs to queue it (two launches of
 * 2 us), so the way from Python to the library counts: ctypes converts six arguments through their declared types and the marshalling
 * around it is interpreted, 0.9 us for mdbf_linear_forward; this way it is 0.2 us (4096 x 4096, k = 1664, one token, a layer called
 * over and over: 10.0 -> 8.9 us a call; a sum of two terms: 12.1 -> 9.5).  Only the calls of a forward pass are here, everything else
 * goes through ctypes.  The interpreter lock is released around each call, as ctypes does.  The module is not linked to the library: it is
 * handed the functions of the one that ctypes has loaded. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>

#include "mdbf.h"

static PyObject *g_addr;                  /* mdbf._addr: the address of an array */

/* the library's functions, in the order set_library takes their addresses in */
typedef mdbf_status_t (*forward_fn)(mdbf_handle_t, const void *, void *, int32_t, int32_t, void *);
static struct {
    forward_fn forward, forward_host, forward_host_async;
    mdbf_status_t (*sum)(const mdbf_handle_t *, int32_t, const void *, void *, float *, int32_t, int32_t, void *);
    mdbf_status_t (*siblings)(const mdbf_handle_t *, int32_t, const void *, void *const *, int32_t, int32_t, void *);
    mdbf_status_t (*group)(const mdbf_handle_t *, int32_t, const void *const *, void *const *, int32_t, int32_t, void *);
} g_lib;

/* integers as they are, None as NULL, a ctypes pointer by its value, anything else through _addr */
static int pointer_arg(PyObject *o, void **out) {
    if (PyLong_Check(o)) {
        *out = (void *)(uintptr_t)PyLong_AsUnsignedLongLongMask(o);
        return !PyErr_Occurred();
    }
    if (o == Py_None) { *out = NULL; return 1; }
    PyObject *v = PyObject_HasAttrString(o, "value") ? PyObject_GetAttrString(o, "value") : PyObject_CallOneArg(g_addr, o);
    if (!v) return 0;
    *out = v == Py_None ? NULL : (void *)(uintptr_t)PyLong_AsUnsignedLongLongMask(v);
    Py_DECREF(v);
    return !PyErr_Occurred();
}
static int int_arg(PyObject *o, int32_t *out) {
    *out = (int32_t)(uint32_t)PyLong_AsUnsignedLongLongMask(o);      /* wraps as ctypes does */
    return !PyErr_Occurred();
}
#define MAX_LAYERS 64                     /* the library's own limit; a longer list is handed on as its length alone and refused there */
static int pointer_list(PyObject *o, void **out, Py_ssize_t at_least, int32_t *n) {
    PyObject *s = PySequence_Fast(o, "a sequence of addresses is wanted");
    if (!s) return 0;
    const Py_ssize_t len = PySequence_Fast_GET_SIZE(s);
    int ok = 1;
    if (len < at_least) { PyErr_SetString(PyExc_ValueError, "fewer buffers than layers"); ok = 0; }
    for (Py_ssize_t i = 0; ok && i < len && i < MAX_LAYERS; ++i) ok = pointer_arg(PySequence_Fast_GET_ITEM(s, i), &out[i]);
    Py_DECREF(s);
    if (n) *n = len > INT32_MAX ? INT32_MAX : (int32_t)len;
    return ok;
}
static int count_is(Py_ssize_t n, Py_ssize_t want) {
    if (!g_addr) { PyErr_SetString(PyExc_RuntimeError, "set_library has not been called"); return 0; }
    if (n == want) return 1;
    PyErr_Format(PyExc_TypeError, "%zd arguments instead of %zd", n, want);
    return 0;
}

static PyObject *forward(forward_fn f, PyObject *const *a, Py_ssize_t n) {
    void *h, *x, *y, *stream;
    int32_t T, act;
    if (!count_is(n, 6) || !pointer_arg(a[0], &h) || !pointer_arg(a[1], &x) || !pointer_arg(a[2], &y) || !int_arg(a[3], &T) || !int_arg(a[4], &act) ||
        !pointer_arg(a[5], &stream))
        return NULL;
    mdbf_status_t rc;
    Py_BEGIN_ALLOW_THREADS
    rc = f((mdbf_handle_t)h, x, y, T, act, stream);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}
static PyObject *linear_forward(PyObject *m, PyObject *const *a, Py_ssize_t n) { (void)m; return forward(g_lib.forward, a, n); }
static PyObject *linear_forward_host(PyObject *m, PyObject *const *a, Py_ssize_t n) { (void)m; return forward(g_lib.forward_host, a, n); }
static PyObject *linear_forward_host_async(PyObject *m, PyObject *const *a, Py_ssize_t n) { (void)m; return forward(g_lib.forward_host_async, a, n); }

static PyObject *linear_forward_sum(PyObject *m, PyObject *const *a, Py_ssize_t n) {
    void *hs[MAX_LAYERS], *x, *y, *acc, *stream;
    int32_t P, T, act;
    (void)m;
    if (!count_is(n, 7) || !pointer_list(a[0], hs, 0, &P) || !pointer_arg(a[1], &x) || !pointer_arg(a[2], &y) || !pointer_arg(a[3], &acc) ||
        !int_arg(a[4], &T) || !int_arg(a[5], &act) || !pointer_arg(a[6], &stream))
        return NULL;
    mdbf_status_t rc;
    Py_BEGIN_ALLOW_THREADS
    rc = g_lib.sum((const mdbf_handle_t *)hs, P, x, y, (float *)acc, T, act, stream);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}
static PyObject *linear_forward_siblings(PyObject *m, PyObject *const *a, Py_ssize_t n) {
    void *hs[MAX_LAYERS], *ys[MAX_LAYERS], *x, *stream;
    int32_t L, T, act;
    (void)m;
    if (!count_is(n, 6) || !pointer_list(a[0], hs, 0, &L) || !pointer_arg(a[1], &x) || !pointer_list(a[2], ys, L, NULL) || !int_arg(a[3], &T) ||
        !int_arg(a[4], &act) || !pointer_arg(a[5], &stream))
        return NULL;
    mdbf_status_t rc;
    Py_BEGIN_ALLOW_THREADS
    rc = g_lib.siblings((const mdbf_handle_t *)hs, L, x, ys, T, act, stream);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}
static PyObject *linear_forward_group(PyObject *m, PyObject *const *a, Py_ssize_t n) {
    void *hs[MAX_LAYERS], *xs[MAX_LAYERS], *ys[MAX_LAYERS], *stream;
    int32_t L, T, act;
    (void)m;
    if (!count_is(n, 6) || !pointer_list(a[0], hs, 0, &L) || !pointer_list(a[1], xs, L, NULL) || !pointer_list(a[2], ys, L, NULL) || !int_arg(a[3], &T) ||
        !int_arg(a[4], &act) || !pointer_arg(a[5], &stream))
        return NULL;
    mdbf_status_t rc;
    Py_BEGIN_ALLOW_THREADS
    rc = g_lib.group((const mdbf_handle_t *)hs, L, (const void *const *)xs, ys, T, act, stream);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}
/* set_library(_addr, (six addresses)) */
static PyObject *set_library(PyObject *m, PyObject *args) {
    PyObject *f;
    unsigned long long p[6];
    (void)m;
    if (!PyArg_ParseTuple(args, "O(KKKKKK)", &f, &p[0], &p[1], &p[2], &p[3], &p[4], &p[5])) return NULL;
    for (int i = 0; i < 6; ++i)
        if (!p[i]) { PyErr_SetString(PyExc_ValueError, "a function's address is missing"); return NULL; }
    g_lib.forward = (forward_fn)(uintptr_t)p[0];
    g_lib.forward_host = (forward_fn)(uintptr_t)p[1];
    g_lib.forward_host_async = (forward_fn)(uintptr_t)p[2];
    *(void **)&g_lib.sum = (void *)(uintptr_t)p[3];
    *(void **)&g_lib.siblings = (void *)(uintptr_t)p[4];
    *(void **)&g_lib.group = (void *)(uintptr_t)p[5];
    Py_XSETREF(g_addr, Py_NewRef(f));
    Py_RETURN_NONE;
}

#define FAST(name) {#name, (PyCFunction)(void (*)(void))name, METH_FASTCALL, NULL}
static PyMethodDef methods[] = {FAST(linear_forward), FAST(linear_forward_host), FAST(linear_forward_host_async), FAST(linear_forward_sum),
                                FAST(linear_forward_siblings), FAST(linear_forward_group), {"set_library", set_library, METH_VARARGS, NULL}, {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "mdbf_calls", NULL, -1, methods, NULL, NULL, NULL, NULL};
PyMODINIT_FUNC PyInit_mdbf_calls(void) { return PyModule_Create(&module); }
