// A call of the library from Python without ctypes: function(address) returns a callable for a function of harp_apply_ex's
// signature at that address.  ctypes converts seven arguments in 1.7 us (0.3 us here, argument checks included), a
// fifth of a decode step's call.  Plain C beside CPython's headers, of the stable interface since 3.10, so that one build serves every
// later interpreter; it does not link to the library.
#define PY_SSIZE_T_CLEAN
#define Py_LIMITED_API 0x030a0000
#include <Python.h>
#include <stdint.h>

typedef int (*apply_fn)(const void *plan, void *x, int64_t n_rows, int dtype, int transpose, int kernel, void *stream);

// integers, None for a null pointer alone; whatever has __index__ counts as an integer, and pointers and codes wrap, as with ctypes
static int to_u64(PyObject *o, int pointer, uint64_t *out) {
    if (pointer && o == Py_None) { *out = 0; return 1; }
    PyObject *i = PyNumber_Index(o);
    if (!i) return 0;
    *out = PyLong_AsUnsignedLongLongMask(i);
    Py_DECREF(i);
    return !(*out == (uint64_t)-1 && PyErr_Occurred());
}

static PyObject *call(PyObject *self, PyObject *const *args, Py_ssize_t n) {
    uint64_t a[7];
    if (n != 7) {
        PyErr_Format(PyExc_TypeError, "7 arguments expected, %zd given", n);
        return NULL;
    }
    for (int k = 0; k < 7; ++k)
        if (!to_u64(args[k], k < 2 || k == 6, &a[k])) return NULL;
    const apply_fn fn = (apply_fn)PyLong_AsVoidPtr(self);
    int st;
    Py_BEGIN_ALLOW_THREADS
    st = fn((const void *)(uintptr_t)a[0], (void *)(uintptr_t)a[1], (int64_t)a[2], (int)a[3], (int)a[4], (int)a[5], (void *)(uintptr_t)a[6]);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(st);
}

static PyMethodDef call_def = {"apply_ex", (PyCFunction)(void (*)(void))call, METH_FASTCALL, "harp_apply_ex(plan, x, n_rows, dtype, transpose, kernel, stream) -> status"};

static PyObject *function(PyObject *self, PyObject *address) {
    (void)self;
    if (!PyLong_Check(address) || !PyLong_AsVoidPtr(address)) {
        if (!PyErr_Occurred()) PyErr_SetString(PyExc_TypeError, "the address of a function expected");
        return NULL;
    }
    return PyCFunction_New(&call_def, address);
}

static PyMethodDef methods[] = {{"function", function, METH_O, "callable for the function at this address"}, {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_harpcall", NULL, -1, methods, NULL, NULL, NULL, NULL};
PyMODINIT_FUNC PyInit__harpcall(void) { return PyModule_Create(&module); }
