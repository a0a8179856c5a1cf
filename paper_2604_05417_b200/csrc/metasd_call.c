/* The calls of a round as Python sees them, for the binding: argument conversion and the call, nothing else.
 *
 * The functions are those of libmetasd.so (include/metasd.h), whose addresses come with every call.  Conversions are ctypes'
 * own for the same signatures (whole numbers are cut to their width, None is a null pointer), and a tensor's data_ptr() is
 * called here as the binding does for ctypes: a number in a tensor's place is refused, with the module and without.  Arguments
 * of other types are left to ctypes (NotImplemented), which says what is wrong with them.
 * The interpreter lock is released around the call, as ctypes does.
 *
 * What it is for: a round of a few sequences is as long as its host calls.  One sequence, V = 32000, verify and select: ctypes'
 * conversions and the Python calls around them took 4.5 of 11.8 us.
 */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>

#include "metasd.h"

static PyObject *data_ptr_name;

/* 1: done; 0: not a type handled here; -1: an exception is set. */
static int as_address(PyObject *o, void **out)
{
    if (o != Py_None && !PyLong_CheckExact(o)) return 0;
    *out = o == Py_None ? NULL : (void *)(uintptr_t)PyLong_AsUnsignedLongLongMask(o);
    return 1;
}

/* What has no data_ptr(), a number for one, is an AttributeError. */
static int as_tensor(PyObject *o, void **out)
{
    if (o == Py_None) {
        *out = NULL;
        return 1;
    }
    PyObject *at = PyObject_CallMethodNoArgs(o, data_ptr_name);
    if (!at) return -1;
    const int ok = as_address(at, out);
    Py_DECREF(at);
    return ok;
}

static int as_bits(PyObject *o, uint64_t *out)
{
    if (!PyLong_Check(o)) return 0;
    *out = (uint64_t)PyLong_AsUnsignedLongLongMask(o);
    return 1;
}

static int as_float(PyObject *o, float *out)
{
    if (!PyFloat_Check(o) && !PyLong_Check(o)) return 0;
    const double x = PyFloat_AsDouble(o);
    if (x == -1.0 && PyErr_Occurred()) return -1;
    *out = (float)x;
    return 1;
}

#define MOST 20

/* Converts the arguments by their kinds: a address (of a function, a context or a stream), t tensor, i whole number, f float.
 * Returns as as_address does. */
static int convert(const char *kinds, PyObject *const *args, Py_ssize_t n, void **p, uint64_t *i, float *f)
{
    for (Py_ssize_t a = 0; a < n; ++a) {
        const int r = kinds[a] == 't' ? as_tensor(args[a], p + a) : kinds[a] == 'a' ? as_address(args[a], p + a) :
                      kinds[a] == 'i' ? as_bits(args[a], i + a) : as_float(args[a], f + a);
        if (r != 1) return r;
    }
    return 1;
}

#define CONVERTED(kinds)                                                                             \
    void *p[MOST];                                                                                   \
    uint64_t i[MOST];                                                                                \
    float f[MOST];                                                                                   \
    int rc;                                                                                          \
    if (n != (Py_ssize_t)sizeof(kinds) - 1) {                                                        \
        PyErr_SetString(PyExc_TypeError, "wrong number of arguments");                               \
        return NULL;                                                                                 \
    }                                                                                                \
    rc = convert(kinds, args, n, p, i, f);                                                           \
    if (rc < 0) return NULL;                                                                         \
    if (rc == 0) Py_RETURN_NOTIMPLEMENTED

static PyObject *call_verify(PyObject *self, PyObject *const *args, Py_ssize_t n)
{
    CONVERTED("aaiittttifitttta");
    __typeof__(&metasd_verify) verify = p[0];   /* as the header declares it: the arguments are checked */
    Py_BEGIN_ALLOW_THREADS
    rc = verify(p[1], (int32_t)i[2], (int32_t)i[3], p[4], p[5], p[6], p[7], (int64_t)i[8], f[9], i[10], p[11], p[12], p[13], p[14],
                p[15]);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

static PyObject *call_select(PyObject *self, PyObject *const *args, Py_ssize_t n)
{
    CONVERTED("aaita");
    __typeof__(&metasd_select) select = p[0];
    Py_BEGIN_ALLOW_THREADS
    rc = select(p[1], (int32_t)i[2], p[3], p[4]);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

static PyObject *call_verify_noalloc(PyObject *self, PyObject *const *args, Py_ssize_t n)
{
    CONVERTED("aiiiitttffiiiitttta");
    __typeof__(&metasd_verify_noalloc) verify = p[0];
    Py_BEGIN_ALLOW_THREADS
    rc = verify((int32_t)i[1], (int32_t)i[2], (int32_t)i[3], (int32_t)i[4], p[5], p[6], p[7], f[8], f[9], (int32_t)i[10], i[11],
                (uint32_t)i[12], (uint32_t)i[13], p[14], p[15], p[16], p[17], p[18]);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

static PyMethodDef methods[] = {
    {"verify", (PyCFunction)(void (*)(void))call_verify, METH_FASTCALL, "metasd_verify; its address comes first"},
    {"select", (PyCFunction)(void (*)(void))call_select, METH_FASTCALL, "metasd_select; its address comes first"},
    {"verify_noalloc", (PyCFunction)(void (*)(void))call_verify_noalloc, METH_FASTCALL, "metasd_verify_noalloc; its address comes first"},
    {NULL, NULL, 0, NULL},
};

static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_call", "Calls into libmetasd.so", -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__call(void)
{
    data_ptr_name = PyUnicode_InternFromString("data_ptr");
    return data_ptr_name ? PyModule_Create(&module) : NULL;
}
