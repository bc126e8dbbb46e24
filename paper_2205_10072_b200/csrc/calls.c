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

/* The same calls with tensors, as binding.py has them: on_build(p, r_begin, r_end, recv_out, send_out, workspace, stream) and so on.  (Python took
 * 0.6 to 0.75 us of a call to ask three or four tensors for their addresses and torch for the stream, of 3.0 to 3.2 us in all; this takes half.) */
static PyObject *data_ptr, *nbytes;            /* names */
static PyObject *initialized, *device, *raw_stream;      /* torch.cuda.is_initialized, current device, its stream as an integer; or None */
static PyObject *any_stream, *plain;           /* binding._stream; the calls through ctypes, by name */

static PyObject *py_set_torch(PyObject *self, PyObject *const *args, Py_ssize_t n)
{
    (void)self;
    if (n != 5) return PyErr_Format(PyExc_TypeError, "set_torch: 5 arguments expected");
    PyObject **to[] = {&initialized, &device, &raw_stream, &any_stream, &plain};
    for (Py_ssize_t i = 0; i < n; ++i) {
        Py_INCREF(args[i]);
        Py_XSETREF(*to[i], args[i]);
    }
    Py_RETURN_NONE;
}

/* The following return 1 with a word, 0 with an error set, -1 where something is not a plain integer. */

/* an integer, or None for 0, whose reference is given up */
static int taken(PyObject *value, unsigned long long *w)
{
    if (value == NULL) return 0;
    int got = 1;
    if (value == Py_None) *w = 0;
    else if (PyLong_Check(value)) *w = PyLong_AsUnsignedLongLongMask(value);
    else got = -1;
    Py_DECREF(value);
    return got;
}

static int address_of(PyObject *tensor, unsigned long long *w)
{
    if (tensor == Py_None) {
        *w = 0;
        return 1;
    }
    return taken(PyObject_CallMethodNoArgs(tensor, data_ptr), w);
}

static int size_of(PyObject *tensor, unsigned long long *w)
{
    if (tensor == Py_None) {
        *w = 0;
        return 1;
    }
    return taken(PyObject_GetAttr(tensor, nbytes), w);
}

static int stream_of(PyObject *stream, unsigned long long *w)
{
    if (stream == Py_None && raw_stream != Py_None && device != Py_None) {
        PyObject *ready = PyObject_CallNoArgs(initialized);
        if (ready == NULL) return 0;
        const int is = PyObject_IsTrue(ready);
        Py_DECREF(ready);
        if (is < 0) return 0;
        if (is) {
            PyObject *index = PyObject_CallNoArgs(device);
            if (index == NULL) return 0;
            PyObject *raw = PyObject_CallOneArg(raw_stream, index);
            Py_DECREF(index);
            return taken(raw, w);
        }
    }
    return taken(PyObject_CallOneArg(any_stream, stream), w);
}

/* Arguments by kind: n a number, p a tensor's address, w address and size of a workspace, s the stream. */
static int tensor_words(PyObject *const *args, const char *kinds, unsigned long long *w)
{
    for (const char *k = kinds; *k; ++k)
        if (*k == 'n' && !PyLong_Check(args[k - kinds])) return -1;
    for (; *kinds; ++kinds, ++args) {
        int got = 1;
        if (*kinds == 'n') *w++ = PyLong_AsUnsignedLongLongMask(*args);
        else if (*kinds == 's') got = stream_of(*args, w++);
        else got = address_of(*args, w++);
        if (*kinds == 'w' && got == 1) got = size_of(*args, w++);
        if (got != 1) return got;
    }
    return 1;
}

#define WRAP_TENSORS(name, kinds, call)                                                      \
    static PyObject *py_on_##name(PyObject *self, PyObject *const *args, Py_ssize_t n)       \
    {                                                                                        \
        unsigned long long w[MOST];                                                          \
        bcs_status st;                                                                       \
        (void)self;                                                                          \
        if (plain == NULL || n != (Py_ssize_t)sizeof kinds - 1)                              \
            return PyErr_Format(PyExc_TypeError, "on_" #name ": %d arguments expected", (int)sizeof kinds - 1); \
        const int got = tensor_words(args, kinds, w);                                        \
        if (got == 0) return NULL;                                                           \
        if (got < 0) {                                                                       \
            PyObject *by = PyObject_GetItem(plain, PyTuple_GET_ITEM(names, AT_##name));      \
            if (by == NULL) return NULL;                                                     \
            PyObject *status = PyObject_Vectorcall(by, args, (size_t)n, NULL);               \
            Py_DECREF(by);                                                                   \
            return status;                                                                   \
        }                                                                                    \
        Py_BEGIN_ALLOW_THREADS                                                               \
        st = call;                                                                           \
        Py_END_ALLOW_THREADS                                                                 \
        return PyLong_FromLong((long)st);                                                    \
    }

enum { AT_build, AT_build_rooted, AT_prepare_rows, AT_build_prepared, AT_build_static, AT_expand, AT_allgather_tables };
static PyObject *names;

WRAP_TENSORS(build, "nnnppws", bcs_build(U(0), w[1], w[2], P(3), P(4), P(5), (size_t)w[6], P(7)))
WRAP_TENSORS(build_rooted, "nnnnppws", bcs_build_rooted(U(0), U(1), w[2], w[3], P(4), P(5), P(6), (size_t)w[7], P(8)))
WRAP_TENSORS(prepare_rows, "nnnpws", bcs_prepare_rows(U(0), w[1], w[2], P(3), P(4), (size_t)w[5], P(6)))
WRAP_TENSORS(build_prepared, "nnnppws", bcs_build_prepared(U(0), w[1], w[2], P(3), P(4), P(5), (size_t)w[6], P(7)))
WRAP_TENSORS(build_static, "nnnpps", bcs_build_static(U(0), w[1], w[2], P(3), P(4), P(5)))
WRAP_TENSORS(expand, "nnnnppps", bcs_expand(U(0), U(1), w[2], w[3], P(4), P(5), P(6), P(7)))
WRAP_TENSORS(allgather_tables, "nnnpppps", bcs_allgather_tables(U(0), U(1), U(2), P(3), P(4), P(5), P(6), P(7)))

#define ENTRY(name) {#name, (PyCFunction)(void (*)(void))py_##name, METH_FASTCALL, NULL}

static PyMethodDef methods[] = {ENTRY(build),          ENTRY(build_rooted), ENTRY(prepare),     ENTRY(prepare_codes),
                                ENTRY(prepare_rows),   ENTRY(build_prepared), ENTRY(build_static), ENTRY(build_batch),
                                ENTRY(expand),         ENTRY(allgather_tables),
                                ENTRY(on_build),       ENTRY(on_build_rooted), ENTRY(on_prepare_rows), ENTRY(on_build_prepared),
                                ENTRY(on_build_static), ENTRY(on_expand),   ENTRY(on_allgather_tables), ENTRY(set_torch),
                                {"set_library", py_set_library, METH_O, NULL}, {NULL, NULL, 0, NULL}};

static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_calls", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__calls(void)
{
    data_ptr = PyUnicode_InternFromString("data_ptr");
    nbytes = PyUnicode_InternFromString("nbytes");
    names = Py_BuildValue("(sssssss)", "build", "build_rooted", "prepare_rows", "build_prepared", "build_static", "expand", "allgather_tables");
    if (data_ptr == NULL || nbytes == NULL || names == NULL) return NULL;
    return PyModule_Create(&module);
}
