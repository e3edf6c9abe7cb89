/*
 * The binding's hot entry points as a CPython module (_binding): argument
 * marshalling only, the same names and arguments as the functions of
 * fasgd.py that they stand in for.
 *
 * Why: a small server step is bound by the host.  Through ctypes a call costs
 * 0.5 to 1 us beyond the C function (push + apply of P = 7,850, K = 1: 3.3 us
 * from Python against 1.6 us from C); here it costs about 0.1 us.
 *
 * Pointers are Python ints or None, integers are Python ints taken modulo
 * their width, as ctypes takes them.  A call with anything else (keywords, a
 * ctypes object, a wrong count of arguments) goes to the ctypes function of the same
 * name, which accepts or refuses it.  The GIL is released around every call,
 * as ctypes does.
 */
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include "fasgd.h"

enum { F_PUSH, F_PUSH_HOST, F_PUSH_SPARSE, F_APPLY, F_SELECT, F_FETCH, F_FETCH_APPLY, F_PUSH_MESSAGE,
       F_FETCH_MESSAGE, F_PUSH_BUDGET, F_FETCH_BUDGET, F_PULL, F_TIMESTAMP, F_PENDING, F_SIM_GRAD,
       F_SIM_LOSS, F_COUNT };

static PyObject* slow[F_COUNT];   /* the ctypes functions (install) */

/* n ints or Nones into x; 0 if an argument is neither. */
static int ints(PyObject* const* args, Py_ssize_t nargs, Py_ssize_t n, unsigned long long* x) {
    if (nargs != n) return 0;
    for (Py_ssize_t i = 0; i < n; ++i) {
        if (args[i] == Py_None) {
            x[i] = 0;
        } else if (PyLong_Check(args[i])) {
            x[i] = PyLong_AsUnsignedLongLongMask(args[i]);
        } else {
            return 0;
        }
    }
    return 1;
}
/* Nones only where a pointer is meant (bit i of `pointers`). */
static int nones(PyObject* const* args, Py_ssize_t n, unsigned pointers) {
    for (Py_ssize_t i = 0; i < n; ++i)
        if (args[i] == Py_None && !(pointers >> i & 1)) return 0;
    return 1;
}

#define H(i) ((fasgd_t*)(uintptr_t)x[i])
#define PTR(type, i) ((type*)(uintptr_t)x[i])
#define I32(i) ((int32_t)x[i])
#define I64(i) ((int64_t)x[i])

#define ENTRY(name, id, n, pointers, call)                                          \
    static PyObject* py_##name(PyObject* self, PyObject* const* args, Py_ssize_t nargs,   \
                               PyObject* kwnames) {                                 \
        unsigned long long x[n];                                                    \
        int64_t r;                                                                  \
        (void)self;                                                                 \
        if (kwnames != NULL || !ints(args, nargs, n, x) || !nones(args, n, pointers)) \
            return PyObject_Vectorcall(slow[id], args, (size_t)nargs, kwnames);     \
        Py_BEGIN_ALLOW_THREADS                                                      \
        r = (int64_t)(call);                                                        \
        Py_END_ALLOW_THREADS                                                        \
        return PyLong_FromLongLong(r);                                              \
    }

ENTRY(fasgd_push, F_PUSH, 4, 0x9, fasgd_push(H(0), I32(1), I64(2), PTR(const float, 3)))
ENTRY(fasgd_push_host, F_PUSH_HOST, 4, 0x9, fasgd_push_host(H(0), I32(1), I64(2), PTR(const float, 3)))
ENTRY(fasgd_push_sparse, F_PUSH_SPARSE, 7, 0x39,
      fasgd_push_sparse(H(0), I32(1), I64(2), PTR(const int32_t, 3), PTR(const float, 4),
                        PTR(const int64_t, 5), I64(6)))
ENTRY(fasgd_apply_pending, F_APPLY, 2, 0x1, fasgd_apply_pending(H(0), I32(1)))
ENTRY(bfasgd_select_compact, F_SELECT, 7, 0x7d,
      bfasgd_select_compact(H(0), I32(1), PTR(const float, 2), PTR(const float, 3), PTR(int32_t, 4),
                            PTR(float, 5), PTR(int64_t, 6)))
ENTRY(bfasgd_fetch_compact, F_FETCH, 6, 0x3d,
      bfasgd_fetch_compact(H(0), I32(1), PTR(const float, 2), PTR(int32_t, 3), PTR(float, 4),
                           PTR(int64_t, 5)))
ENTRY(bfasgd_fetch_apply, F_FETCH_APPLY, 8, 0xde,
      bfasgd_fetch_apply(I64(0), PTR(float, 1), PTR(const int32_t, 2), PTR(const float, 3),
                         PTR(const int64_t, 4), I64(5), PTR(void, 6), PTR(int32_t, 7)))
ENTRY(bfasgd_push_message, F_PUSH_MESSAGE, 5, 0x19,
      bfasgd_push_message(H(0), I32(1), I64(2), PTR(const float, 3), PTR(int32_t, 4)))
ENTRY(bfasgd_fetch_message, F_FETCH_MESSAGE, 4, 0xd,
      bfasgd_fetch_message(H(0), I32(1), PTR(float, 2), PTR(int32_t, 3)))
ENTRY(bfasgd_push_budget, F_PUSH_BUDGET, 8, 0xe9,
      bfasgd_push_budget(H(0), I32(1), I64(2), PTR(const float, 3), I64(4), PTR(uint8_t, 5),
                         PTR(float, 6), PTR(int64_t, 7)))
ENTRY(bfasgd_fetch_budget, F_FETCH_BUDGET, 7, 0x75,
      bfasgd_fetch_budget(H(0), I32(1), PTR(float, 2), I64(3), PTR(uint8_t, 4), PTR(float, 5),
                          PTR(int64_t, 6)))
ENTRY(fasgd_timestamp, F_TIMESTAMP, 1, 0x1, fasgd_timestamp(H(0)))
ENTRY(fasgd_pending, F_PENDING, 1, 0x1, fasgd_pending(H(0)))
ENTRY(fasgd_sim_quadratic_grad, F_SIM_GRAD, 10, 0x31e,
      fasgd_sim_quadratic_grad(I64(0), PTR(const float, 1), PTR(const float, 2), PTR(const float, 3),
                               PTR(const float, 4), (uint64_t)x[5], I32(6), (uint64_t)x[7],
                               PTR(float, 8), PTR(void, 9)))
ENTRY(fasgd_sim_quadratic_loss, F_SIM_LOSS, 7, 0x7e,
      fasgd_sim_quadratic_loss(I64(0), PTR(const float, 1), PTR(const float, 2), PTR(const float, 3),
                               PTR(double, 4), PTR(double, 5), PTR(void, 6)))

/* fasgd_pull(h, params) -> (status, T) */
static PyObject* py_fasgd_pull(PyObject* self, PyObject* const* args, Py_ssize_t nargs,
                               PyObject* kwnames) {
    unsigned long long x[2];
    int64_t T = 0;
    int rc;
    PyObject *out, *a, *b;
    (void)self;
    if (kwnames != NULL || !ints(args, nargs, 2, x))
        return PyObject_Vectorcall(slow[F_PULL], args, (size_t)nargs, kwnames);
    Py_BEGIN_ALLOW_THREADS
    rc = fasgd_pull(H(0), PTR(float, 1), &T);
    Py_END_ALLOW_THREADS
    out = PyTuple_New(2);
    a = PyLong_FromLong(rc);
    b = PyLong_FromLongLong(T);
    if (out == NULL || a == NULL || b == NULL) {
        Py_XDECREF(out);
        Py_XDECREF(a);
        Py_XDECREF(b);
        return NULL;
    }
    PyTuple_SET_ITEM(out, 0, a);
    PyTuple_SET_ITEM(out, 1, b);
    return out;
}

#define METHOD(name) {#name, (PyCFunction)(void (*)(void))py_##name, METH_FASTCALL | METH_KEYWORDS, NULL}
static const char* const names[F_COUNT] = {
    "fasgd_push", "fasgd_push_host", "fasgd_push_sparse", "fasgd_apply_pending", "bfasgd_select_compact",
    "bfasgd_fetch_compact", "bfasgd_fetch_apply", "bfasgd_push_message", "bfasgd_fetch_message",
    "bfasgd_push_budget", "bfasgd_fetch_budget", "fasgd_pull", "fasgd_timestamp", "fasgd_pending",
    "fasgd_sim_quadratic_grad", "fasgd_sim_quadratic_loss"};

/* install(namespace): keeps the ctypes functions of these names for the calls
 * this module does not take, and returns the names.  A namespace that holds one
 * of this module's own functions is refused whole: it would hand the call to
 * itself without end. */
static PyObject* py_install(PyObject* self, PyObject* space) {
    PyObject *out, *f[F_COUNT];
    if (!PyDict_Check(space)) {
        PyErr_SetString(PyExc_TypeError, "install: a dict is expected");
        return NULL;
    }
    for (int i = 0; i < F_COUNT; ++i) {
        f[i] = PyDict_GetItemString(space, names[i]);
        if (f[i] == NULL) {
            PyErr_Format(PyExc_KeyError, "install: no %s", names[i]);
            return NULL;
        }
        if (PyCFunction_Check(f[i]) && PyCFunction_GET_SELF(f[i]) == self) {
            PyErr_Format(PyExc_ValueError, "install: %s is this module's own", names[i]);
            return NULL;
        }
    }
    out = PyList_New(0);
    if (out == NULL) return NULL;
    for (int i = 0; i < F_COUNT; ++i) {
        PyObject *s = PyUnicode_FromString(names[i]), *old = slow[i];
        if (s == NULL || PyList_Append(out, s) < 0) {
            Py_XDECREF(s);
            Py_DECREF(out);
            return NULL;
        }
        Py_DECREF(s);
        Py_INCREF(f[i]);
        slow[i] = f[i];
        Py_XDECREF(old);
    }
    return out;
}

static PyMethodDef methods[] = {
    METHOD(fasgd_push), METHOD(fasgd_push_host), METHOD(fasgd_push_sparse), METHOD(fasgd_apply_pending),
    METHOD(bfasgd_select_compact), METHOD(bfasgd_fetch_compact), METHOD(bfasgd_fetch_apply),
    METHOD(bfasgd_push_message), METHOD(bfasgd_fetch_message), METHOD(bfasgd_push_budget),
    METHOD(bfasgd_fetch_budget), METHOD(fasgd_pull), METHOD(fasgd_timestamp), METHOD(fasgd_pending),
    METHOD(fasgd_sim_quadratic_grad), METHOD(fasgd_sim_quadratic_loss),
    {"install", py_install, METH_O, NULL}, {NULL, NULL, 0, NULL}};

static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_binding", NULL, -1, methods,
                                    NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__binding(void) { return PyModule_Create(&module); }
