/* The calls of include/bcs.h that enqueue work, for Python: addresses and sizes in, status out.  (Through ctypes the
 * conversion of eight to nineteen arguments took 0.8 to 1.4 us of a call, as much as the smallest kernels last.) */
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include "bcs.h"

#define MOST 19

static PyObject *library;      /* the same calls through ctypes, for arguments that are not plain */

/* ints as 64-bit patterns, None as 0 where bit i of `pointers` is set; 0 if there is anything else */
static int words(PyObject *const *args, Py_ssize_t n, Py_ssize_t want, unsigned pointers, unsigned long long *w)
{
    if (n != want) return 0;
    for (Py_ssize_t i = 0; i < n; ++i) {
        if (args[i] == Py_None && (pointers >> i) & 1u) {
            w[i] = 0;
        } else if (PyLong_Check(args[i])) {
            w[i] = PyLong_AsUnsignedLongLongMask(args[i]);
        } else if (PyIndex_Check(args[i])) {
            PyObject *index = PyNumber_Index(args[i]);
            if (index == NULL) {
                PyErr_Clear();
                return 0;
            }
            w[i] = PyLong_AsUnsignedLongLongMask(index);
            Py_DECREF(index);
        } else {
            return 0;
        }
    }
    return 1;
}

static PyObject *through_ctypes(const char *name, PyObject *const *args, Py_ssize_t n)
{
    if (library == NULL) return PyErr_Format(PyExc_TypeError, "%s: integers and addresses expected", name);
    PyObject *call = PyObject_GetAttrString(library, name);
    if (call == NULL) return NULL;
    PyObject *status = PyObject_Vectorcall(call, args, (size_t)n, NULL);
    Py_DECREF(call);
    return status;
}

static PyObject *py_set_library(PyObject *self, PyObject *given)
{
    (void)self;
    Py_INCREF(given);
    Py_XSETREF(library, given);
    Py_RETURN_NONE;
}

#define P(i) ((void *)(uintptr_t)w[i])
#define U(i) ((uint32_t)w[i])

/* One wrapper: its name, its number of arguments, which of them are pointers (a bit each), the call. */
#define WRAP(name, count, pointers, call)                                                    \
    static PyObject *py_##name(PyObject *self, PyObject *const *args, Py_ssize_t n)          \
    {                                                                                        \
        unsigned long long w[MOST];                                                          \
        bcs_status st;                                                                       \
        (void)self;                                                                          \
        if (!words(args, n, count, pointers, w)) return through_ctypes("bcs_" #name, args, n); \
        Py_BEGIN_ALLOW_THREADS                                                               \
        st = call;                                                                           \
        Py_END_ALLOW_THREADS                                                                 \
        return PyLong_FromLong((long)st);                                                    \
    }

WRAP(build, 8, 0xb8u, bcs_build(U(0), w[1], w[2], P(3), P(4), P(5), (size_t)w[6], P(7)))
WRAP(build_rooted, 9, 0x170u, bcs_build_rooted(U(0), U(1), w[2], w[3], P(4), P(5), P(6), (size_t)w[7], P(8)))
WRAP(prepare, 4, 0xau, bcs_prepare(U(0), P(1), (size_t)w[2], P(3)))
WRAP(prepare_codes, 4, 0xau, bcs_prepare_codes(U(0), P(1), (size_t)w[2], P(3)))
WRAP(prepare_rows, 7, 0x58u, bcs_prepare_rows(U(0), w[1], w[2], P(3), P(4), (size_t)w[5], P(6)))
WRAP(build_prepared, 8, 0xb8u, bcs_build_prepared(U(0), w[1], w[2], P(3), P(4), P(5), (size_t)w[6], P(7)))
WRAP(build_static, 6, 0x38u, bcs_build_static(U(0), w[1], w[2], P(3), P(4), P(5)))
WRAP(build_batch, 17, 0x1707fu, bcs_build_batch(P(0), P(1), P(2), P(3), P(4), P(5), P(6), U(7), w[8], w[9], w[10], w[11], P(12),
                                      P(13), P(14), (size_t)w[15], P(16)))
WRAP(expand, 8, 0xf0u, bcs_expand(U(0), U(1), w[2], w[3], P(4), P(5), P(6), P(7)))
WRAP(allgather_tables, 8, 0xf8u, bcs_allgather_tables(U(0), U(1), U(2), P(3), P(4), P(5), P(6), P(7)))

#define ENTRY(name) {#name, (PyCFunction)(void (*)(void))py_##name, METH_FASTCALL, NULL}

static PyMethodDef methods[] = {ENTRY(build),          ENTRY(build_rooted), ENTRY(prepare),     ENTRY(prepare_codes),
                                ENTRY(prepare_rows),   ENTRY(build_prepared), ENTRY(build_static), ENTRY(build_batch),
                                ENTRY(expand),         ENTRY(allgather_tables),
                                {"set_library", py_set_library, METH_O, NULL}, {NULL, NULL, 0, NULL}};

static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_calls", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__calls(void) { return PyModule_Create(&module); }
