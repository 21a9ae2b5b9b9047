/* CPython entries to perq_rotate_quantize and perq_swiglu_rotate_quantize: integers to C arguments, and the call without the interpreter lock.
 *
 * Small calls are bound by the host.  Of 4.8 us for one row, the general converter of foreign functions took 0.95 (its own call, one
 * object for each argument); this takes 0.2 (one row of 2048: 4.84 -> 4.1 us between calls).  Arguments that are not plain integers (None: a null pointer) are refused with a
 * TypeError, upon which the caller takes the general converter, so that what is accepted and what is raised stay its own. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>

typedef int (*rotate_fn)(const void *, const int32_t *, int64_t, int32_t, int32_t, int32_t, int32_t, void *, void *, void *);
typedef int (*swiglu_fn)(const void *, const void *, const int32_t *, int64_t, int32_t, int32_t, int32_t, int32_t, void *, void *, void *);

static rotate_fn rotate = NULL;
static swiglu_fn swiglu = NULL;

/* n arguments, of which five from `first` on are numbers and the others addresses. */
static int convert(PyObject *const *args, Py_ssize_t n, Py_ssize_t expected, int first, unsigned long long *a)
{
    if (n != expected) { PyErr_SetString(PyExc_TypeError, "number of arguments"); return 0; }
    for (int i = 0; i < n; ++i) {
        const int number = i >= first && i < first + 5;
        if (args[i] == Py_None && !number) { a[i] = 0; continue; }
        if (!PyLong_Check(args[i])) { PyErr_SetString(PyExc_TypeError, "an integer is required"); return 0; }
        a[i] = PyLong_AsUnsignedLongLongMask(args[i]);
    }
    return 1;
}
#define ADDRESS(v) ((void *)(uintptr_t)(v))

static PyObject *rotate_quantize(PyObject *self, PyObject *const *args, Py_ssize_t n)
{
    unsigned long long a[10];
    int rc;
    (void)self;
    if (!convert(args, n, 10, 2, a)) return NULL;
    Py_BEGIN_ALLOW_THREADS
    rc = rotate(ADDRESS(a[0]), ADDRESS(a[1]), (int64_t)a[2], (int32_t)a[3], (int32_t)a[4], (int32_t)a[5], (int32_t)a[6], ADDRESS(a[7]), ADDRESS(a[8]),
                ADDRESS(a[9]));
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

static PyObject *swiglu_rotate_quantize(PyObject *self, PyObject *const *args, Py_ssize_t n)
{
    unsigned long long a[11];
    int rc;
    (void)self;
    if (!convert(args, n, 11, 3, a)) return NULL;
    Py_BEGIN_ALLOW_THREADS
    rc = swiglu(ADDRESS(a[0]), ADDRESS(a[1]), ADDRESS(a[2]), (int64_t)a[3], (int32_t)a[4], (int32_t)a[5], (int32_t)a[6], (int32_t)a[7], ADDRESS(a[8]),
                ADDRESS(a[9]), ADDRESS(a[10]));
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

static PyObject *bind(PyObject *self, PyObject *const *args, Py_ssize_t n)
{
    (void)self;
    if (n != 2) { PyErr_SetString(PyExc_TypeError, "number of arguments"); return NULL; }
    void *const r = PyLong_AsVoidPtr(args[0]), *const s = PyLong_AsVoidPtr(args[1]);
    if (PyErr_Occurred()) return NULL;
    rotate = (rotate_fn)r;
    swiglu = (swiglu_fn)s;
    Py_RETURN_NONE;
}

static PyMethodDef methods[] = {
    {"rotate_quantize", (PyCFunction)(void (*)(void))rotate_quantize, METH_FASTCALL, "perq_rotate_quantize(x, perm, T, d, b, fmt, group, codes, scales, stream)"},
    {"swiglu_rotate_quantize", (PyCFunction)(void (*)(void))swiglu_rotate_quantize, METH_FASTCALL, "perq_swiglu_rotate_quantize(gate, up, perm, T, d, b, fmt, group, codes, scales, stream)"},
    {"bind", (PyCFunction)(void (*)(void))bind, METH_FASTCALL, "The addresses of both; before any call."},
    {NULL, NULL, 0, NULL},
};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_perq_call", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__perq_call(void) { return PyModule_Create(&module); }
