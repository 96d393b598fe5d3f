/* Argument marshalling of binding.py's calls in native code: reads addresses and sizes off tensors
 * and arrays and calls the library function whose address it is given.  (With ctypes the marshalling
 * of a recurrent call took 9 us on the measuring host, as much as the smallest call itself; this
 * takes about 1 us.)  Every function returns the library's status code. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>

enum { kMaxList = 64 };

static PyObject *s_data_ptr, *s_shape, *s_stride, *s_handle, *s_value, *s_zero;

/* Address of a torch tensor (data_ptr()) or of a numpy array (its buffer); None is NULL. */
static int address(PyObject* o, void** out) {
    *out = NULL;
    if (o == Py_None) return 0;
    if (PyObject_CheckBuffer(o)) {
        Py_buffer b;
        if (PyObject_GetBuffer(o, &b, PyBUF_STRIDED_RO)) return -1;
        *out = b.buf;
        PyBuffer_Release(&b);
        return 0;
    }
    PyObject* p = PyObject_CallMethodNoArgs(o, s_data_ptr);
    if (!p) return -1;
    *out = PyLong_AsVoidPtr(p);
    Py_DECREF(p);
    return PyErr_Occurred() ? -1 : 0;
}
/* A ctypes number or pointer counts as its value; everything else as itself.  A new reference. */
static PyObject* plain(PyObject* o) {
    if (o != Py_None && !PyLong_Check(o) && !PyIndex_Check(o)) {
        PyObject* v = PyObject_GetAttr(o, s_value);
        if (v) return v;
        PyErr_Clear();
    }
    Py_INCREF(o);
    return o;
}
static int pointer(PyObject* o, void** out) {      /* an integer, a ctypes pointer or None */
    *out = NULL;
    PyObject* v = plain(o);
    if (!v) return -1;
    if (v != Py_None) *out = PyLong_AsVoidPtr(v);
    Py_DECREF(v);
    return PyErr_Occurred() ? -1 : 0;
}
static int flag_bits(PyObject* o, unsigned* out) {
    PyObject* v = plain(o);
    if (!v) return -1;
    *out = (unsigned)PyLong_AsUnsignedLongMask(v);
    Py_DECREF(v);
    return PyErr_Occurred() ? -1 : 0;
}
static int handle_of(PyObject* o, void** out) {
    PyObject* h = PyObject_GetAttr(o, s_handle);
    if (!h) return -1;
    const int rc = pointer(h, out);
    Py_DECREF(h);
    return rc;
}
static int size_at(PyObject* o, Py_ssize_t i, int64_t* out) {
    PyObject* s = PyObject_GetAttr(o, s_shape);
    if (!s) return -1;
    PyObject* v = PySequence_GetItem(s, i);
    Py_DECREF(s);
    if (!v) return -1;
    *out = PyLong_AsLongLong(v);
    Py_DECREF(v);
    return PyErr_Occurred() ? -1 : 0;
}
static int row_stride(PyObject* o, int64_t* out) {
    PyObject* v = PyObject_CallMethodOneArg(o, s_stride, s_zero);
    if (!v) return -1;
    *out = PyLong_AsLongLong(v);
    Py_DECREF(v);
    return PyErr_Occurred() ? -1 : 0;
}
/* The first n items of a sequence: handles of matrices (None is NULL, which the library refuses), or addresses. */
static int list_of(PyObject* o, Py_ssize_t n, int handles, void** out) {
    PyObject* s = PySequence_Fast(o, "a sequence is expected");
    if (!s) return -1;
    int rc = 0;
    if (PySequence_Fast_GET_SIZE(s) < n) { PyErr_SetString(PyExc_IndexError, "list index out of range"); rc = -1; }
    for (Py_ssize_t i = 0; i < n && !rc; ++i) {
        PyObject* v = PySequence_Fast_GET_ITEM(s, i);
        rc = handles && v != Py_None ? handle_of(v, &out[i]) : address(v, &out[i]);
    }
    Py_DECREF(s);
    return rc;
}
static int arity(Py_ssize_t n, Py_ssize_t want) {
    if (n == want) return 0;
    PyErr_Format(PyExc_TypeError, "%zd arguments, expected %zd", n, want);
    return -1;
}

/* spmv(function, matrix, x, y, stream) */
static PyObject* py_spmv(PyObject* self, PyObject* const* a, Py_ssize_t n) {
    void *f, *h, *x, *y, *st;
    int rc;
    if (arity(n, 5) || pointer(a[0], &f) || handle_of(a[1], &h) || address(a[2], &x) || address(a[3], &y) || pointer(a[4], &st)) return NULL;
    Py_BEGIN_ALLOW_THREADS
    rc = ((int (*)(void*, void*, void*, void*))f)(h, x, y, st);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}
/* spmm(function, matrix, X, Y, stream): batch and row strides from the tensors (strides 0 for an empty batch) */
static PyObject* py_spmm(PyObject* self, PyObject* const* a, Py_ssize_t n) {
    void *f, *h, *x, *y, *st;
    int64_t batch = 0, ldx = 0, ldy = 0;
    int rc;
    if (arity(n, 5) || pointer(a[0], &f) || handle_of(a[1], &h) || address(a[2], &x) || address(a[3], &y) || pointer(a[4], &st)) return NULL;
    if (size_at(a[2], 0, &batch) || (batch && (row_stride(a[2], &ldx) || row_stride(a[3], &ldy)))) return NULL;
    Py_BEGIN_ALLOW_THREADS
    rc = ((int (*)(void*, void*, int64_t, int, void*, int64_t, void*))f)(h, x, ldx, (int)batch, y, ldy, st);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}
/* recurrent(function, kind, W, Wp, bias, x, h0, c0, y, hT, cT, flags, stream)
 * kind 0: (L, W, bias, x, T, B, h0, c0, y, hT, cT, flags, stream); 1: without the cell states;
 * 2: with projections behind W. */
static PyObject* py_recurrent(PyObject* self, PyObject* const* a, Py_ssize_t n) {
    void *f, *st, *x, *h0, *c0, *y, *hT, *cT, *W[kMaxList], *Wp[kMaxList], *bias[kMaxList];
    int64_t T, B;
    int rc;
    if (arity(n, 13) || pointer(a[0], &f)) return NULL;
    const long kind = PyLong_AsLong(a[1]);
    const Py_ssize_t L = PyObject_Length(a[2]);
    unsigned flags;
    if (PyErr_Occurred() || flag_bits(a[11], &flags)) return NULL;
    const Py_ssize_t m = L < kMaxList ? L : kMaxList;      /* more layers than the library takes: it refuses by L */
    if (list_of(a[2], m, 1, W) || (kind == 2 && list_of(a[3], m, 1, Wp)) || (a[4] != Py_None && list_of(a[4], m, 0, bias))) return NULL;
    if (address(a[5], &x) || size_at(a[5], 0, &T) || size_at(a[5], 1, &B) || address(a[6], &h0) || address(a[7], &c0) || address(a[8], &y) ||
        address(a[9], &hT) || address(a[10], &cT) || pointer(a[12], &st)) return NULL;
    void* const* pb = a[4] == Py_None ? NULL : bias;
    Py_BEGIN_ALLOW_THREADS
    if (kind == 0)
        rc = ((int (*)(int, void* const*, void* const*, void*, int64_t, int, void*, void*, void*, void*, void*, unsigned, void*))f)(
            (int)L, W, pb, x, T, (int)B, h0, c0, y, hT, cT, flags, st);
    else if (kind == 1)
        rc = ((int (*)(int, void* const*, void* const*, void*, int64_t, int, void*, void*, void*, unsigned, void*))f)((int)L, W, pb, x, T, (int)B, h0, y,
                                                                                                                  hT, flags, st);
    else
        rc = ((int (*)(int, void* const*, void* const*, void* const*, void*, int64_t, int, void*, void*, void*, void*, void*, unsigned, void*))f)(
            (int)L, W, Wp, pb, x, T, (int)B, h0, c0, y, hT, cT, flags, st);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

static PyMethodDef methods[] = {{"spmv", (PyCFunction)(void (*)(void))py_spmv, METH_FASTCALL, NULL},
                                {"spmm", (PyCFunction)(void (*)(void))py_spmm, METH_FASTCALL, NULL},
                                {"recurrent", (PyCFunction)(void (*)(void))py_recurrent, METH_FASTCALL, NULL},
                                {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_csb_py", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__csb_py(void) {
    s_data_ptr = PyUnicode_InternFromString("data_ptr");
    s_shape = PyUnicode_InternFromString("shape");
    s_stride = PyUnicode_InternFromString("stride");
    s_handle = PyUnicode_InternFromString("handle");
    s_value = PyUnicode_InternFromString("value");
    s_zero = PyLong_FromLong(0);
    if (!s_data_ptr || !s_shape || !s_stride || !s_handle || !s_value || !s_zero) return NULL;
    return PyModule_Create(&module);
}
