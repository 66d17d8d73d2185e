/* CPython helper of the binding: one call of a C entry point from Python arguments.
 *
 * A call of the smallest layers takes the device a few microseconds, and marshalling its arguments in Python (a function call,
 * is_contiguous() and data_ptr() per tensor, then the conversions of ctypes) took the host 2 us of the 4.5 that a call with one
 * launch costs it.  Here that is the two tensor methods and nothing else. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>

#define MAX_ARGS 17   /* moe_layer_fwd_bwd_host */

static PyObject *str_is_contiguous, *str_data_ptr;

/* None: 0.  An integer: itself.  Anything else: the data_ptr() of a contiguous tensor. */
static int argument(PyObject *o, uint64_t *out) {
    if (o == Py_None) { *out = 0; return 0; }
    if (!PyLong_Check(o)) {
        PyObject *r = PyObject_CallMethodNoArgs(o, str_is_contiguous);
        if (r == NULL) return -1;
        const int yes = PyObject_IsTrue(r);
        Py_DECREF(r);
        if (yes < 0) return -1;
        if (!yes) { PyErr_SetString(PyExc_ValueError, "tensor must be contiguous"); return -1; }
        r = PyObject_CallMethodNoArgs(o, str_data_ptr);
        if (r == NULL) return -1;
        *out = PyLong_AsUnsignedLongLongMask(r);
        Py_DECREF(r);
    } else {
        *out = PyLong_AsUnsignedLongLongMask(o);
    }
    return *out == (uint64_t)-1 && PyErr_Occurred() ? -1 : 0;
}

/* call(entry, dims, argument, ...) -> status.  `entry` is a function's address, or (address, number of parameters after `dims`), which
 * the arguments are then counted against.  Every parameter of the entry points after `dims` is a pointer, a size_t or an int:
 * an integer register or an eight-byte stack slot each, so a caller of 64-bit integers fits them all (x86-64 and AArch64 ABIs). */
static PyObject *call(PyObject *self, PyObject *const *args, Py_ssize_t n) {
    (void)self;
    if (n < 2 || n - 2 > MAX_ARGS) { PyErr_SetString(PyExc_TypeError, "call(entry, dims, up to 17 arguments)"); return NULL; }
    PyObject *address = args[0];
    if (PyTuple_Check(address)) {
        if (PyTuple_GET_SIZE(address) != 2) { PyErr_SetString(PyExc_TypeError, "entry must be an address or (address, parameters)"); return NULL; }
        const Py_ssize_t want = PyLong_AsSsize_t(PyTuple_GET_ITEM(address, 1));
        if (want == -1 && PyErr_Occurred()) return NULL;
        if (want != n - 2) { PyErr_Format(PyExc_TypeError, "%zd arguments after dims, the function takes %zd", n - 2, want); return NULL; }
        address = PyTuple_GET_ITEM(address, 0);
    }
    void *fn = PyLong_AsVoidPtr(address);
    if (fn == NULL) {
        if (!PyErr_Occurred()) PyErr_SetString(PyExc_ValueError, "null address");
        return NULL;
    }
    uint64_t a[MAX_ARGS] = {0};
    for (Py_ssize_t i = 2; i < n; ++i)
        if (argument(args[i], &a[i - 2]) != 0) return NULL;
    Py_buffer dims;   /* a ctypes structure: its own memory */
    if (PyObject_GetBuffer(args[1], &dims, PyBUF_SIMPLE) != 0) return NULL;
    if (dims.len != 5 * (Py_ssize_t)sizeof(int32_t)) {
        PyBuffer_Release(&dims);
        PyErr_SetString(PyExc_TypeError, "dims must be a MoeDims");
        return NULL;
    }
    int rc;
    typedef uint64_t u;
    Py_BEGIN_ALLOW_THREADS
    switch (n - 2) {
        case 0: rc = ((int (*)(void *))fn)(dims.buf); break;
        case 1: rc = ((int (*)(void *, u))fn)(dims.buf, a[0]); break;
        case 2: rc = ((int (*)(void *, u, u))fn)(dims.buf, a[0], a[1]); break;
        case 3: rc = ((int (*)(void *, u, u, u))fn)(dims.buf, a[0], a[1], a[2]); break;
        case 4: rc = ((int (*)(void *, u, u, u, u))fn)(dims.buf, a[0], a[1], a[2], a[3]); break;
        case 5: rc = ((int (*)(void *, u, u, u, u, u))fn)(dims.buf, a[0], a[1], a[2], a[3], a[4]); break;
        case 6: rc = ((int (*)(void *, u, u, u, u, u, u))fn)(dims.buf, a[0], a[1], a[2], a[3], a[4], a[5]); break;
        case 7: rc = ((int (*)(void *, u, u, u, u, u, u, u))fn)(dims.buf, a[0], a[1], a[2], a[3], a[4], a[5], a[6]); break;
        case 8: rc = ((int (*)(void *, u, u, u, u, u, u, u, u))fn)(dims.buf, a[0], a[1], a[2], a[3], a[4], a[5], a[6], a[7]); break;
        case 9: rc = ((int (*)(void *, u, u, u, u, u, u, u, u, u))fn)(dims.buf, a[0], a[1], a[2], a[3], a[4], a[5], a[6], a[7], a[8]); break;
        case 10: rc = ((int (*)(void *, u, u, u, u, u, u, u, u, u, u))fn)(dims.buf, a[0], a[1], a[2], a[3], a[4], a[5], a[6], a[7], a[8], a[9]); break;
        case 11: rc = ((int (*)(void *, u, u, u, u, u, u, u, u, u, u, u))fn)(dims.buf, a[0], a[1], a[2], a[3], a[4], a[5], a[6], a[7], a[8], a[9], a[10]); break;
        default:   /* a callee never looks at slots behind its own parameters */
            rc = ((int (*)(void *, u, u, u, u, u, u, u, u, u, u, u, u, u, u, u, u, u))fn)(
                dims.buf, a[0], a[1], a[2], a[3], a[4], a[5], a[6], a[7], a[8], a[9], a[10], a[11], a[12], a[13], a[14], a[15], a[16]);
            break;
    }
    Py_END_ALLOW_THREADS
    PyBuffer_Release(&dims);
    return PyLong_FromLong(rc);
}

static PyMethodDef methods[] = {{"call", (PyCFunction)(void (*)(void))call, METH_FASTCALL, "call(entry, dims, *arguments) -> status"},
                                {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_pycall", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__pycall(void) {
    str_is_contiguous = PyUnicode_InternFromString("is_contiguous");
    str_data_ptr = PyUnicode_InternFromString("data_ptr");
    if (str_is_contiguous == NULL || str_data_ptr == NULL) return NULL;
    return PyModule_Create(&module);
}
