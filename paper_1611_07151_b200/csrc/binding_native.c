/* Marshalling of the binding's two calls that a program makes once per layer: tensors and numbers of a Python call to a call of
 * the library's function at a given address.  ctypes and the Python code around it took 3.0 us a call (of the 6.5 us that a small
 * convolution's call takes on the host, 2.7 of them the launch).  Anything but None, plain integers and objects with a
 * data_ptr() method is left to the ctypes path: the functions then return None. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <limits.h>
#include <stdint.h>

#include "sqn.h"

static PyObject* s_data_ptr;

/* 0: *p is the address; 1: not for this path; -1: an exception is set */
static int address_of(PyObject* o, void** p)
{
    if (o == Py_None) { *p = NULL; return 0; }
    PyObject* r = o;
    if (PyLong_Check(o)) Py_INCREF(r);
    else {
        r = PyObject_CallMethodNoArgs(o, s_data_ptr);
        if (!r) {
            if (!PyErr_ExceptionMatches(PyExc_AttributeError)) return -1;
            PyErr_Clear();
            return 1;
        }
        if (!PyLong_Check(r)) { Py_DECREF(r); return 1; }
    }
    *p = (void*)(uintptr_t)PyLong_AsUnsignedLongLongMask(r);
    Py_DECREF(r);
    return PyErr_Occurred() ? -1 : 0;
}

static int int_of(PyObject* o, int* v)
{
    int overflow = 0;
    if (!PyLong_Check(o)) return 1;
    const long n = PyLong_AsLongAndOverflow(o, &overflow);
    if (overflow || n < INT_MIN || n > INT_MAX) return 1;
    *v = (int)n;
    return 0;
}

#define TRY(e) do { const int rc_ = (e); if (rc_ < 0) return NULL; if (rc_ > 0) Py_RETURN_NONE; } while (0)

/* (address, in, weights, bias, out, 8 sizes, dtype, relu, out_c_offset, out_c_total, stream, workspace, workspace_bytes,
 *  fuse_maxpool, fuse_global_avgpool) -> status, None: not for this path */
static PyObject* native_conv_forward_ex(PyObject* self, PyObject* const* a, Py_ssize_t n)
{
    (void)self;
    if (n != 22) { PyErr_SetString(PyExc_TypeError, "22 arguments"); return NULL; }
    void *fn, *p[4], *stream, *workspace;
    int v[8], relu, fmax, favg;
    sqn_conv_opts o;
    TRY(address_of(a[0], &fn));
    for (int i = 0; i < 4; ++i) TRY(address_of(a[1 + i], &p[i]));
    for (int i = 0; i < 8; ++i) TRY(int_of(a[5 + i], &v[i]));
    TRY(int_of(a[13], &o.dtype));
    if ((relu = PyObject_IsTrue(a[14])) < 0) return NULL;
    o.relu = relu;
    TRY(int_of(a[15], &o.out_c_offset));
    TRY(int_of(a[16], &o.out_c_total));
    if (a[17] != Py_None && !PyLong_Check(a[17])) Py_RETURN_NONE;
    TRY(address_of(a[17], &stream));
    TRY(address_of(a[18], &workspace));
    if (!PyLong_Check(a[19])) Py_RETURN_NONE;
    o.workspace_bytes = (size_t)PyLong_AsUnsignedLongLongMask(a[19]);
    if (PyErr_Occurred()) return NULL;
    if ((fmax = PyObject_IsTrue(a[20])) < 0 || (favg = PyObject_IsTrue(a[21])) < 0) return NULL;
    o.stream = stream;
    o.workspace = workspace;
    o.fuse_maxpool = fmax;
    o.fuse_global_avgpool = favg;
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = ((int (*)(const void*, const void*, const void*, void*, int, int, int, int, int, int, int, int, const sqn_conv_opts*))fn)(
        p[0], p[1], p[2], p[3], v[0], v[1], v[2], v[3], v[4], v[5], v[6], v[7], &o);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

/* (address, 9 addresses, 8 numbers, stream) -> status, None: not for this path */
static PyObject* native_fire_forward(PyObject* self, PyObject* const* a, Py_ssize_t n)
{
    (void)self;
    if (n != 19) { PyErr_SetString(PyExc_TypeError, "19 arguments"); return NULL; }
    void *fn, *p[9], *stream;
    int v[8];
    TRY(address_of(a[0], &fn));
    for (int i = 0; i < 9; ++i) TRY(address_of(a[1 + i], &p[i]));
    for (int i = 0; i < 8; ++i) TRY(int_of(a[10 + i], &v[i]));
    if (a[18] != Py_None && !PyLong_Check(a[18])) Py_RETURN_NONE;
    TRY(address_of(a[18], &stream));
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = ((int (*)(const void*, const void*, const void*, const void*, const void*, const void*, const void*, void*, void*, int, int, int,
                   int, int, int, int, int, void*))fn)(p[0], p[1], p[2], p[3], p[4], p[5], p[6], p[7], p[8], v[0], v[1], v[2], v[3], v[4],
                                                       v[5], v[6], v[7], stream);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

static PyMethodDef methods[] = {
    {"conv_forward_ex", (PyCFunction)(void (*)(void))native_conv_forward_ex, METH_FASTCALL, NULL},
    {"fire_forward", (PyCFunction)(void (*)(void))native_fire_forward, METH_FASTCALL, NULL},
    {NULL, NULL, 0, NULL}};

static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__native(void)
{
    s_data_ptr = PyUnicode_InternFromString("data_ptr");
    PyObject* m = s_data_ptr ? PyModule_Create(&module) : NULL;
    if (m && PyModule_AddIntConstant(m, "sizeof_conv_opts", (long)sizeof(sqn_conv_opts)) < 0) Py_CLEAR(m);
    return m;
}
