/* The calls of include/bcs.h that enqueue work, for Python: addresses and sizes in, status out.  (Through ctypes the
 * conversion of eight to nineteen arguments took 0.8 to 1.4 us of a call, as much as the smallest kernels last.) */
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include "bcs.h"

#define MOST 19

/* ints as 64-bit patterns, None as 0 */
static int words(PyObject *const *args, Py_ssize_t n, Py_ssize_t want, unsigned long long *w)
{
    if (n != want) {
        PyErr_Format(PyExc_TypeError, "%zd arguments, %zd expected", n, want);
        return -1;
    }
    for (Py_ssize_t i = 0; i < n; ++i) {
        if (args[i] == Py_None) {
            w[i] = 0;
        } else if (PyLong_Check(args[i])) {
            w[i] = PyLong_AsUnsignedLongLongMask(args[i]);
        } else {
            PyObject *index = PyNumber_Index(args[i]);
            if (index == NULL) return -1;
            w[i] = PyLong_AsUnsignedLongLongMask(index);
            Py_DECREF(index);
        }
        if (w[i] == (unsigned long long)-1 && PyErr_Occurred()) return -1;
    }
    return 0;
}

#define P(i) ((void *)(uintptr_t)w[i])
#define U(i) ((uint32_t)w[i])

/* One wrapper: its name, its number of arguments, the call. */
#define WRAP(name, count, call)                                                              \
    static PyObject *py_##name(PyObject *self, PyObject *const *args, Py_ssize_t n)          \
    {                                                                                        \
        unsigned long long w[MOST];                                                          \
        bcs_status st;                                                                       \
        (void)self;                                                                          \
        if (words(args, n, count, w) < 0) return NULL;                                       \
        Py_BEGIN_ALLOW_THREADS                                                               \
        st = call;                                                                           \
        Py_END_ALLOW_THREADS                                                                 \
        return PyLong_FromLong((long)st);                                                    \
    }

WRAP(build, 8, bcs_build(U(0), w[1], w[2], P(3), P(4), P(5), (size_t)w[6], P(7)))
WRAP(build_rooted, 9, bcs_build_rooted(U(0), U(1), w[2], w[3], P(4), P(5), P(6), (size_t)w[7], P(8)))
WRAP(prepare, 4, bcs_prepare(U(0), P(1), (size_t)w[2], P(3)))
WRAP(prepare_codes, 4, bcs_prepare_codes(U(0), P(1), (size_t)w[2], P(3)))
WRAP(prepare_rows, 7, bcs_prepare_rows(U(0), w[1], w[2], P(3), P(4), (size_t)w[5], P(6)))
WRAP(build_prepared, 8, bcs_build_prepared(U(0), w[1], w[2], P(3), P(4), P(5), (size_t)w[6], P(7)))
WRAP(build_static, 6, bcs_build_static(U(0), w[1], w[2], P(3), P(4), P(5)))
WRAP(build_batch, 17, bcs_build_batch(P(0), P(1), P(2), P(3), P(4), P(5), P(6), U(7), w[8], w[9], w[10], w[11], P(12),
                                      P(13), P(14), (size_t)w[15], P(16)))
WRAP(expand, 8, bcs_expand(U(0), U(1), w[2], w[3], P(4), P(5), P(6), P(7)))
WRAP(allgather_tables, 8, bcs_allgather_tables(U(0), U(1), U(2), P(3), P(4), P(5), P(6), P(7)))

#define ENTRY(name) {#name, (PyCFunction)(void (*)(void))py_##name, METH_FASTCALL, NULL}

static PyMethodDef methods[] = {ENTRY(build),          ENTRY(build_rooted), ENTRY(prepare),     ENTRY(prepare_codes),
                                ENTRY(prepare_rows),   ENTRY(build_prepared), ENTRY(build_static), ENTRY(build_batch),
                                ENTRY(expand),         ENTRY(allgather_tables), {NULL, NULL, 0, NULL}};

static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_calls", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__calls(void) { return PyModule_Create(&module); }
