/*
 * Argument marshalling of the two calls of a scheduler's loop (slaq_append_losses, slaq_schedule) for Python.
 *
 * Through ctypes the pointers of four arrays cost about ten microseconds per append, more than the call's own work on the
 * host for a cluster of a few hundred jobs.  Here the arrays are taken through the buffer protocol; an argument
 * that is not a contiguous array of the right type makes the function return None, and the caller converts it.
 */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>

typedef int (*append_fn)(void*, int32_t, const int32_t*, const double*, const double*);
typedef int (*append_ex_fn)(void*, int32_t, const int32_t*, const double*, const double*, const int32_t*);
typedef int (*schedule_fn)(void*, double, int64_t, int32_t*);

/* 1: `v` holds a contiguous array of `size`-byte entries of kind `kind` ('i' or 'd'); 0: it does not (no error is set) */
static int take(PyObject* o, int flags, Py_ssize_t size, char kind, Py_buffer* v) {
    if (PyObject_GetBuffer(o, v, flags | PyBUF_C_CONTIGUOUS | PyBUF_FORMAT) != 0) {
        PyErr_Clear();
        return 0;
    }
    const char* f = v->format ? v->format : "B";
    const int match = f[0] == kind || (kind == 'i' && f[0] == 'l');
    if (v->itemsize != size || !match || f[1] != 0) {
        PyBuffer_Release(v);
        return 0;
    }
    return 1;
}

/* append(append address, append_ex address, handle, ids, losses, times or None, cores or None) -> status or None */
static PyObject* append(PyObject* self, PyObject* const* args, Py_ssize_t n_args) {
    (void)self;
    if (n_args != 7) {
        PyErr_SetString(PyExc_TypeError, "append takes 7 arguments");
        return NULL;
    }
    void* const plain = PyLong_AsVoidPtr(args[0]);
    void* const ex = PyLong_AsVoidPtr(args[1]);
    void* const handle = PyLong_AsVoidPtr(args[2]);
    if (PyErr_Occurred()) return NULL;
    Py_buffer v[4];
    int held = 0, fits = 1, rc = 0;
    const int has_times = args[5] != Py_None, has_cores = args[6] != Py_None;
    fits = take(args[3], PyBUF_SIMPLE, 4, 'i', &v[0]);
    held = fits;
    if (fits && (fits = take(args[4], PyBUF_SIMPLE, 8, 'd', &v[1]))) held = 2;
    if (fits && has_times && (fits = take(args[5], PyBUF_SIMPLE, 8, 'd', &v[2]))) held = 3;
    if (fits && has_cores && !has_times) fits = 0;
    if (fits && has_cores && (fits = take(args[6], PyBUF_SIMPLE, 4, 'i', &v[3]))) held = 4;
    const Py_ssize_t n = fits ? v[0].len / 4 : 0;
    if (fits && (v[1].len != 8 * n || (has_times && v[2].len != 8 * n) || (has_cores && v[3].len != 4 * n) || n > INT32_MAX))
        fits = 0;
    if (fits) {
        const double* const times = has_times ? (const double*)v[2].buf : NULL;
        Py_BEGIN_ALLOW_THREADS;
        if (has_cores)
            rc = ((append_ex_fn)ex)(handle, (int32_t)n, (const int32_t*)v[0].buf, (const double*)v[1].buf, times,
                                    (const int32_t*)v[3].buf);
        else
            rc = ((append_fn)plain)(handle, (int32_t)n, (const int32_t*)v[0].buf, (const double*)v[1].buf, times);
        Py_END_ALLOW_THREADS;
    }
    for (int i = 0; i < held; ++i) PyBuffer_Release(&v[i]);
    if (!fits) Py_RETURN_NONE;
    return PyLong_FromLong(rc);
}

/* schedule(address, handle, epoch seconds, cores, out array, entries it must have) -> status or None */
static PyObject* schedule(PyObject* self, PyObject* const* args, Py_ssize_t n_args) {
    (void)self;
    if (n_args != 6) {
        PyErr_SetString(PyExc_TypeError, "schedule takes 6 arguments");
        return NULL;
    }
    void* const fn = PyLong_AsVoidPtr(args[0]);
    void* const handle = PyLong_AsVoidPtr(args[1]);
    const double seconds = PyFloat_AsDouble(args[2]);
    const long long cores = PyLong_AsLongLong(args[3]);
    const Py_ssize_t want = PyLong_AsSsize_t(args[5]);
    if (PyErr_Occurred()) return NULL;
    Py_buffer v;
    if (!take(args[4], PyBUF_WRITABLE, 4, 'i', &v)) Py_RETURN_NONE;
    if (v.len < 4 * want) {
        PyBuffer_Release(&v);
        Py_RETURN_NONE;
    }
    int rc;
    Py_BEGIN_ALLOW_THREADS;
    rc = ((schedule_fn)fn)(handle, seconds, (int64_t)cores, (int32_t*)v.buf);
    Py_END_ALLOW_THREADS;
    PyBuffer_Release(&v);
    return PyLong_FromLong(rc);
}

static PyMethodDef methods[] = {
    {"append", (PyCFunction)(void (*)(void))append, METH_FASTCALL, "one slaq_append_losses / slaq_append_losses_ex call"},
    {"schedule", (PyCFunction)(void (*)(void))schedule, METH_FASTCALL, "one slaq_schedule call"},
    {NULL, NULL, 0, NULL}};

static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_marshal", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__marshal(void) { return PyModule_Create(&module); }
