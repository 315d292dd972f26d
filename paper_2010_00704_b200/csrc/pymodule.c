/* CPython front of the C ABI's launching calls.  A call on a small layer is a few microseconds of GPU work, and
 * converting thirteen arguments through ctypes took longer than that; here an argument costs some tens of
 * nanoseconds.  Every function takes its pointers as None, an integer address or an object with a data_ptr() method
 * (a torch tensor), then its integers, then the stream's address, and returns the call's status. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include "bcnn.h"

static PyObject *s_data_ptr;

static int as_pointer(PyObject *o, void **out)
{
    PyObject *v;
    if (o == Py_None) { *out = NULL; return 0; }
    if (PyLong_Check(o)) {
        *out = PyLong_AsVoidPtr(o);
        return PyErr_Occurred() ? -1 : 0;
    }
    v = PyObject_CallMethodNoArgs(o, s_data_ptr);
    if (!v) return -1;
    *out = PyLong_AsVoidPtr(v);
    Py_DECREF(v);
    return PyErr_Occurred() ? -1 : 0;
}

/* np pointers, ni integers, the stream */
static int parse(PyObject *const *args, Py_ssize_t n, int np, void **p, int ni, long long *v, void **stream)
{
    int i;
    if (n != np + ni + 1) {
        PyErr_Format(PyExc_TypeError, "%d arguments expected, got %zd", np + ni + 1, n);
        return -1;
    }
    for (i = 0; i < np; ++i)
        if (as_pointer(args[i], &p[i])) return -1;
    for (i = 0; i < ni; ++i) {
        v[i] = PyLong_AsLongLong(args[np + i]);
        if (v[i] == -1 && PyErr_Occurred()) return -1;
    }
    return as_pointer(args[np + ni], stream);
}

/* an int argument of the ABI, truncated as a C conversion would */
#define I(k) ((int)v[k])

#define CALL(name, NP, NI, expr)                                                    \
    static PyObject *name(PyObject *self, PyObject *const *args, Py_ssize_t n)      \
    {                                                                               \
        void *p[NP], *stream;                                                       \
        long long v[NI];                                                            \
        int st;                                                                     \
        (void)self;                                                                 \
        if (parse(args, n, NP, p, NI, v, &stream)) return NULL;                     \
        Py_BEGIN_ALLOW_THREADS                                                      \
        st = (expr);                                                                \
        Py_END_ALLOW_THREADS                                                        \
        return PyLong_FromLong(st);                                                 \
    }

CALL(pack, 3, 5, bcnn_pack(p[0], p[1], p[2], I(0), I(1), I(2), I(3), I(4), stream))
CALL(stem_fused, 5, 6, bcnn_stem_fused(p[0], p[1], p[2], p[3], p[4], I(0), I(1), I(2), I(3), I(4), I(5), stream))
CALL(conv2d, 4, 10, bcnn_conv2d_b1_engine(I(0), p[0], p[1], p[2], p[3], I(1), I(2), I(3), I(4), I(5), I(6), I(7), I(8), I(9), stream))
CALL(gemm, 4, 4, bcnn_gemm_b1_engine(I(0), p[0], p[1], p[2], p[3], v[1], I(2), I(3), stream))
CALL(conv2d_module, 9, 9, bcnn_conv2d_b1_module(p[0], p[1], p[2], p[3], p[4], p[5], p[6], p[7], p[8], I(0), I(1), I(2), I(3), I(4), I(5), I(6), I(7), I(8), stream))
CALL(conv2d_branches, 10, 8, bcnn_conv2d_b1_branches(p[0], p[1], p[2], p[3], p[4], p[5], p[6], p[7], p[8], p[9], I(0), I(1), I(2), I(3), I(4), I(5), I(6), I(7), stream))
CALL(dwconv3x3_module, 8, 6, bcnn_dwconv3x3_module(p[0], p[1], p[2], p[3], p[4], p[5], p[6], p[7], I(0), I(1), I(2), I(3), I(4), I(5), stream))
CALL(avgpool, 2, 6, bcnn_avgpool(p[0], p[1], I(0), I(1), I(2), I(3), I(4), I(5), stream))
CALL(gap, 2, 4, bcnn_gap(p[0], p[1], I(0), I(1), I(2), I(3), stream))
CALL(fc, 4, 3, bcnn_fc(p[0], p[1], p[2], p[3], I(0), I(1), I(2), stream))
CALL(prepare_weights, 2, 2, bcnn_prepare_weights(p[0], p[1], I(0), I(1), stream))
CALL(conv2d_prepared, 4, 9, bcnn_conv2d_b1_prepared(p[0], p[1], p[2], p[3], I(0), I(1), I(2), I(3), I(4), I(5), I(6), I(7), I(8), stream))
CALL(gemm_prepared, 4, 3, bcnn_gemm_b1_prepared(p[0], p[1], p[2], p[3], v[0], I(1), I(2), stream))
CALL(conv2d_fused_noalloc, 4, 9, bcnn_conv2d_b1_fused_noalloc(p[0], p[1], p[2], p[3], I(0), I(1), I(2), I(3), I(4), I(5), I(6), I(7), I(8), stream))

#define METHOD(name) {#name, (PyCFunction)(void (*)(void))name, METH_FASTCALL, NULL}
static PyMethodDef methods[] = {
    METHOD(pack), METHOD(stem_fused), METHOD(conv2d), METHOD(gemm), METHOD(conv2d_module), METHOD(conv2d_branches),
    METHOD(dwconv3x3_module), METHOD(avgpool), METHOD(gap), METHOD(fc), METHOD(prepare_weights), METHOD(conv2d_prepared),
    METHOD(gemm_prepared), METHOD(conv2d_fused_noalloc), {NULL, NULL, 0, NULL}};

static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__native(void)
{
    s_data_ptr = PyUnicode_InternFromString("data_ptr");
    return s_data_ptr ? PyModule_Create(&module) : NULL;
}
