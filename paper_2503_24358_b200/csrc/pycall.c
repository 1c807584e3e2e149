/*
 * The calls that a serving loop makes for every window and token, for Python without ctypes: ctypes converts an argument in
 * about 0.1 us, which for 17 to 33 of them is as much as a kernel launch.  Arguments are plain integers (addresses, sizes,
 * strides, the stream) and one float; the functions are those of the library that bind() was given the addresses of, so
 * that whatever build of it the binding has loaded is the one that is called.  The GIL is released during a call.
 */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include "../../include/squat.h"

typedef long long ll;

static struct {
    __typeof__(&squat_quantize_keys) keys;
    __typeof__(&squat_quantize_keys_m16) keys_m16;
    __typeof__(&squat_quantize_values) values;
    __typeof__(&squat_quantize_values_m16) values_m16;
    __typeof__(&squat_dequantize) deq;
    __typeof__(&squat_dequantize_m16) deq_m16;
    __typeof__(&squat_decode_attention_ex) attend;
} lib;

/* n integers (None: 0) out of args */
static int integers(PyObject *const *args, Py_ssize_t given, Py_ssize_t n, ll *a)
{
    if (given != n) {
        PyErr_Format(PyExc_TypeError, "%zd arguments expected, %zd given", n, given);
        return 0;
    }
    for (Py_ssize_t i = 0; i < n; ++i) {
        if (args[i] == Py_None) {
            a[i] = 0;
            continue;
        }
        a[i] = PyLong_AsLongLong(args[i]);
        if (a[i] == -1 && PyErr_Occurred()) {
            PyErr_Clear();                                  /* an address above 2^63 */
            a[i] = (ll)PyLong_AsUnsignedLongLong(args[i]);
            if (PyErr_Occurred()) return 0;
        }
    }
    return 1;
}
#define P(i) ((void *)(uintptr_t)a[i])
#define I(i) ((int)a[i])

static PyObject *bind(PyObject *self, PyObject *const *args, Py_ssize_t n)
{
    ll a[7];
    (void)self;
    if (!integers(args, n, 7, a)) return NULL;
    lib.keys = (__typeof__(lib.keys))P(0);
    lib.keys_m16 = (__typeof__(lib.keys_m16))P(1);
    lib.values = (__typeof__(lib.values))P(2);
    lib.values_m16 = (__typeof__(lib.values_m16))P(3);
    lib.deq = (__typeof__(lib.deq))P(4);
    lib.deq_m16 = (__typeof__(lib.deq_m16))P(5);
    lib.attend = (__typeof__(lib.attend))P(6);
    Py_RETURN_NONE;
}

/* meta16, then the arguments of squat_quantize_keys */
static PyObject *quantize_keys(PyObject *self, PyObject *const *args, Py_ssize_t n)
{
    ll a[19];
    int rc;
    (void)self;
    if (!integers(args, n, 19, a)) return NULL;
    Py_BEGIN_ALLOW_THREADS
    if (a[0]) rc = lib.keys_m16(P(1), P(2), I(3), I(4), I(5), I(6), I(7), a[8], a[9], a[10], I(11), I(12), P(13), P(14), P(15), a[16], a[17], P(18));
    else rc = lib.keys(P(1), P(2), I(3), I(4), I(5), I(6), I(7), a[8], a[9], a[10], I(11), I(12), P(13), P(14), P(15), a[16], a[17], P(18));
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

/* meta16, then the arguments of squat_quantize_values */
static PyObject *quantize_values(PyObject *self, PyObject *const *args, Py_ssize_t n)
{
    ll a[18];
    int rc;
    (void)self;
    if (!integers(args, n, 18, a)) return NULL;
    Py_BEGIN_ALLOW_THREADS
    if (a[0]) rc = lib.values_m16(P(1), I(2), I(3), I(4), I(5), I(6), a[7], a[8], a[9], I(10), I(11), P(12), P(13), P(14), a[15], a[16], P(17));
    else rc = lib.values(P(1), I(2), I(3), I(4), I(5), I(6), a[7], a[8], a[9], I(10), I(11), P(12), P(13), P(14), a[15], a[16], P(17));
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

/* meta16, then the arguments of squat_dequantize */
static PyObject *dequantize(PyObject *self, PyObject *const *args, Py_ssize_t n)
{
    ll a[16];
    int rc;
    (void)self;
    if (!integers(args, n, 16, a)) return NULL;
    Py_BEGIN_ALLOW_THREADS
    if (a[0]) rc = lib.deq_m16(I(1), P(2), P(3), P(4), I(5), I(6), I(7), I(8), I(9), I(10), a[11], a[12], P(13), I(14), P(15));
    else rc = lib.deq(I(1), P(2), P(3), P(4), I(5), I(6), I(7), I(8), I(9), I(10), a[11], a[12], P(13), I(14), P(15));
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

/* softmax_scale, then the other arguments of squat_decode_attention_ex in their order */
static PyObject *decode_attention(PyObject *self, PyObject *const *args, Py_ssize_t n)
{
    ll a[29];
    int rc;
    (void)self;
    if (n < 1) {
        PyErr_SetString(PyExc_TypeError, "30 arguments expected");
        return NULL;
    }
    const double scale = PyFloat_AsDouble(args[0]);
    if (scale == -1.0 && PyErr_Occurred()) return NULL;
    if (!integers(args + 1, n - 1, 29, a)) return NULL;
    Py_BEGIN_ALLOW_THREADS
    rc = lib.attend(P(0), I(1), I(2), I(3), I(4), I(5), P(6), P(7), P(8), P(9), P(10), P(11), I(12), I(13), a[14], a[15], I(16), I(17),
                    P(18), P(19), I(20), I(21), (float)scale, P(22), I(23), a[24], P(25), P(26), (size_t)a[27], P(28));
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

static PyMethodDef methods[] = {
    {"bind", (PyCFunction)(void (*)(void))bind, METH_FASTCALL, "addresses of the library's functions"},
    {"quantize_keys", (PyCFunction)(void (*)(void))quantize_keys, METH_FASTCALL, NULL},
    {"quantize_values", (PyCFunction)(void (*)(void))quantize_values, METH_FASTCALL, NULL},
    {"dequantize", (PyCFunction)(void (*)(void))dequantize, METH_FASTCALL, NULL},
    {"decode_attention", (PyCFunction)(void (*)(void))decode_attention, METH_FASTCALL, NULL},
    {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_squatcall", "direct calls into libsquat", -1, methods, NULL, NULL, NULL, NULL};
PyMODINIT_FUNC PyInit__squatcall(void) { return PyModule_Create(&module); }
