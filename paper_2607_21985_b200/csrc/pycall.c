/* The Python side's calls that are made once per layer and token, as vectorcall functions: ctypes converts eight arguments
 * in 1.1 us, a quarter of what such a call costs on the host; this takes 0.2.  Every function gets the address of the
 * library's entry point first (so it follows whichever build of the library is loaded) and then that entry point's arguments
 * as numbers, None for a null pointer.  The status comes back as an int; the GIL is released around the call. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>

/* What ctypes takes for a number or an address besides an int: one of its own simple values (a handle or stream kept as a
 * c_void_p, say) and anything with _as_parameter_.  A new reference, or NULL with the error set. */
static PyObject* plain(PyObject* o) {
    static PyObject* simple = NULL;
    PyObject* v = PyObject_GetAttrString(o, "_as_parameter_");
    if (v != NULL) return v;
    PyErr_Clear();
    if (simple == NULL) {
        PyObject* m = PyImport_ImportModule("ctypes");
        simple = m != NULL ? PyObject_GetAttrString(m, "_SimpleCData") : NULL;
        Py_XDECREF(m);
        if (simple == NULL) return NULL;
    }
    switch (PyObject_IsInstance(o, simple)) {
        case 1: return PyObject_GetAttrString(o, "value");
        case 0: PyErr_Format(PyExc_TypeError, "an int or None, not %.80s", Py_TYPE(o)->tp_name);
    }
    return NULL;
}

/* kind 'p': an address, or None for a null pointer; 'i': an integer.  Kept out of the converters, which are inlined. */
static __attribute__((noinline)) int from_other(PyObject* o, char kind, void** ptr, int64_t* i64) {
    PyObject* v = plain(o);
    int ok = v != NULL;
    if (ok && kind == 'p' && v == Py_None) *ptr = NULL;
    else if (ok && PyLong_Check(v)) {
        if (kind == 'p') *ptr = PyLong_AsVoidPtr(v);
        else *i64 = PyLong_AsLongLong(v);
        ok = !PyErr_Occurred();
    } else if (ok) {
        PyErr_Format(PyExc_TypeError, "an int or None, not %.80s", Py_TYPE(o)->tp_name);
        ok = 0;
    }
    Py_XDECREF(v);
    return ok;
}
static int as_ptr(PyObject* o, void** out) {
    if (o == Py_None) { *out = NULL; return 1; }
    if (!PyLong_Check(o)) return from_other(o, 'p', out, NULL);
    *out = PyLong_AsVoidPtr(o);
    return !(*out == NULL && PyErr_Occurred());
}
static int as_i64(PyObject* o, int64_t* out) {
    if (!PyLong_Check(o)) return from_other(o, 'i', NULL, out);
    *out = PyLong_AsLongLong(o);
    return !(*out == -1 && PyErr_Occurred());
}
static int as_int(PyObject* o, int* out) {
    int64_t v;
    if (!as_i64(o, &v)) return 0;
    if (v != (int64_t)(int)v) { PyErr_SetString(PyExc_OverflowError, "argument does not fit a C int"); return 0; }
    *out = (int)v;
    return 1;
}
static int as_float(PyObject* o, float* out) {
    const double v = PyFloat_AsDouble(o);
    *out = (float)v;
    return !(v == -1.0 && PyErr_Occurred());
}
static int count(Py_ssize_t n, Py_ssize_t want) {
    if (n == want) return 1;
    PyErr_Format(PyExc_TypeError, "%zd arguments, not %zd", want, n);
    return 0;
}

typedef int (*spmspv_fn)(void*, const void*, int, float, const void*, void*, int, void*);
static PyObject* call_spmspv(PyObject* self, PyObject* const* a, Py_ssize_t n) {
    void *f, *h, *x, *mask, *y, *stream;
    int rule, ydt, st;
    float thr;
    if (!count(n, 9) || !as_ptr(a[0], &f) || !as_ptr(a[1], &h) || !as_ptr(a[2], &x) || !as_int(a[3], &rule) || !as_float(a[4], &thr) ||
        !as_ptr(a[5], &mask) || !as_ptr(a[6], &y) || !as_int(a[7], &ydt) || !as_ptr(a[8], &stream))
        return NULL;
    Py_BEGIN_ALLOW_THREADS
    st = ((spmspv_fn)f)(h, x, rule, thr, mask, y, ydt, stream);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(st);
}

typedef int (*batch_fn)(void*, const void*, int64_t, int, int, float, const void*, int64_t, void*, int64_t, int, void*);
static PyObject* call_spmspv_batch(PyObject* self, PyObject* const* a, Py_ssize_t n) {
    void *f, *h, *x, *mask, *y, *stream;
    int64_t ldx, mstride, ldy;
    int batch, rule, ydt, st;
    float thr;
    if (!count(n, 13) || !as_ptr(a[0], &f) || !as_ptr(a[1], &h) || !as_ptr(a[2], &x) || !as_i64(a[3], &ldx) || !as_int(a[4], &batch) ||
        !as_int(a[5], &rule) || !as_float(a[6], &thr) || !as_ptr(a[7], &mask) || !as_i64(a[8], &mstride) || !as_ptr(a[9], &y) ||
        !as_i64(a[10], &ldy) || !as_int(a[11], &ydt) || !as_ptr(a[12], &stream))
        return NULL;
    Py_BEGIN_ALLOW_THREADS
    st = ((batch_fn)f)(h, x, ldx, batch, rule, thr, mask, mstride, y, ldy, ydt, stream);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(st);
}

typedef int (*spmm_fn)(void*, const void*, int64_t, int64_t, void*, int64_t, int, void*);
static PyObject* call_spmm(PyObject* self, PyObject* const* a, Py_ssize_t n) {
    void *f, *h, *x, *y, *stream;
    int64_t rows, ldx, ldy;
    int ydt, st;
    if (!count(n, 9) || !as_ptr(a[0], &f) || !as_ptr(a[1], &h) || !as_ptr(a[2], &x) || !as_i64(a[3], &rows) || !as_i64(a[4], &ldx) ||
        !as_ptr(a[5], &y) || !as_i64(a[6], &ldy) || !as_int(a[7], &ydt) || !as_ptr(a[8], &stream))
        return NULL;
    Py_BEGIN_ALLOW_THREADS
    st = ((spmm_fn)f)(h, x, rows, ldx, y, ldy, ydt, stream);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(st);
}

typedef int (*swiglu_fn)(const void*, const void*, int64_t, float, void*, void*, void*, void*);
static PyObject* call_swiglu_dp(PyObject* self, PyObject* const* a, Py_ssize_t n) {
    void *f, *gate, *up, *x, *mask, *cnt, *stream;
    int64_t k;
    float thr;
    int st;
    if (!count(n, 9) || !as_ptr(a[0], &f) || !as_ptr(a[1], &gate) || !as_ptr(a[2], &up) || !as_i64(a[3], &k) || !as_float(a[4], &thr) ||
        !as_ptr(a[5], &x) || !as_ptr(a[6], &mask) || !as_ptr(a[7], &cnt) || !as_ptr(a[8], &stream))
        return NULL;
    Py_BEGIN_ALLOW_THREADS
    st = ((swiglu_fn)f)(gate, up, k, thr, x, mask, cnt, stream);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(st);
}

static PyMethodDef methods[] = {
    {"spmspv", (PyCFunction)(void (*)(void))call_spmspv, METH_FASTCALL, "spdp_spmspv"},
    {"spmspv_batch", (PyCFunction)(void (*)(void))call_spmspv_batch, METH_FASTCALL, "spdp_spmspv_batch"},
    {"spmm", (PyCFunction)(void (*)(void))call_spmm, METH_FASTCALL, "spdp_spmm"},
    {"swiglu_dp", (PyCFunction)(void (*)(void))call_swiglu_dp, METH_FASTCALL, "spdp_swiglu_dp"},
    {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_pycall", "Per-token entry points of libspdp.", -1, methods, NULL, NULL, NULL, NULL};
PyMODINIT_FUNC PyInit__pycall(void) { return PyModule_Create(&module); }
