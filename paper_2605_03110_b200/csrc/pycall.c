/* Native marshalling of the hot calls of binding.py: tensors (or None) become pointers, numbers
 * become C arguments, and the library call runs with the interpreter lock released.  ctypes does the
 * same, argument by argument through its type objects, in 5 to 10 us for a call of twenty
 * arguments -- more than the smallest selections take on the GPU. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include "../../include/ada.h"

static PyObject* s_data_ptr;

/* a tensor's data_ptr(); whatever has no such method raises, a number or None among them: a wrong argument
 * must not become a device address */
static void* tensor(PyObject* o, int* bad) {
    if (*bad) return NULL;
    PyObject* v = PyObject_CallMethodNoArgs(o, s_data_ptr);
    if (v == NULL) { *bad = 1; return NULL; }
    void* p = PyLong_AsVoidPtr(v);
    Py_DECREF(v);
    if (p == NULL && PyErr_Occurred()) *bad = 1;
    return p;
}
static void* optional(PyObject* o, int* bad) { return o == Py_None ? NULL : tensor(o, bad); }
/* handles that binding.py holds as numbers: context, stream, threshold policy (None: NULL) */
static void* handle(PyObject* o, int* bad) {
    if (*bad || o == Py_None) return NULL;
    void* p = PyLong_AsVoidPtr(o);
    if (p == NULL && PyErr_Occurred()) *bad = 1;
    return p;
}
static int64_t number(PyObject* o, int* bad) {
    if (*bad) return 0;
    const int64_t v = PyLong_AsLongLong(o);
    if (v == -1 && PyErr_Occurred()) *bad = 1;
    return v;
}
static double real(PyObject* o, int* bad) {
    if (*bad) return 0.0;
    PyObject* f = PyNumber_Float(o);               /* all that float() takes */
    if (f == NULL) { *bad = 1; return 0.0; }
    const double v = PyFloat_AS_DOUBLE(f);
    Py_DECREF(f);
    return v;
}

#define ARGS(n)                                                                     \
    if (na != (n)) return PyErr_Format(PyExc_TypeError, "%d arguments wanted", (n)); \
    int bad = 0, k = 0
#define H(type, name) type* name = (type*)handle(a[k++], &bad)
#define P(type, name) type* name = (type*)tensor(a[k++], &bad)
#define O(type, name) type* name = (type*)optional(a[k++], &bad)
#define N(name) const int64_t name = number(a[k++], &bad)
#define D(name) const double name = real(a[k++], &bad)
#define CALL(expr)                     \
    if (bad) return NULL;              \
    ada_status st;                     \
    Py_BEGIN_ALLOW_THREADS st = expr;  \
    Py_END_ALLOW_THREADS return PyLong_FromLong((long)st)

static PyObject* select_full(PyObject* self, PyObject* const* a, Py_ssize_t na) {
    ARGS(12);
    H(ada_ctx, c); P(void, X); N(B); N(T); N(d); N(ldx); N(dt); D(tau);
    P(int32_t, idx); P(int32_t, cnt); O(float, gamma); H(void, s);
    CALL(ada_select_full(c, X, B, T, d, ldx, (ada_dtype)dt, tau, idx, cnt, gamma, s));
}
static PyObject* select_full_heads(PyObject* self, PyObject* const* a, Py_ssize_t na) {
    ARGS(12);
    H(ada_ctx, c); P(void, X); N(T); N(h); N(d); N(ldx); N(dt); D(tau);
    P(int32_t, idx); P(int32_t, cnt); O(float, gamma); H(void, s);
    CALL(ada_select_full_heads(c, X, T, h, d, ldx, (ada_dtype)dt, tau, idx, cnt, gamma, s));
}
#define LISTS                                                                             \
    P(int32_t, ri); P(int32_t, ric); P(int32_t, ro); P(int32_t, roc); P(int32_t, ai);     \
    P(int32_t, ac); P(int32_t, mi); P(int32_t, mc); O(float, gr); O(float, gc)
static PyObject* cascade_step(PyObject* self, PyObject* const* a, Py_ssize_t na) {
    ARGS(20);
    H(ada_ctx, c); P(void, X); N(B); N(T); N(d); N(ldx); N(dt); D(tau); LISTS; N(flags); H(void, s);
    CALL(ada_cascade_step(c, X, B, T, d, ldx, (ada_dtype)dt, tau, ri, ric, ro, roc, ai, ac, mi, mc, gr, gc,
                          (uint32_t)flags, s));
}
static PyObject* cascade_step_heads(PyObject* self, PyObject* const* a, Py_ssize_t na) {
    ARGS(20);
    H(ada_ctx, c); P(void, X); N(T); N(h); N(d); N(ldx); N(dt); D(tau); LISTS; N(flags); H(void, s);
    CALL(ada_cascade_step_heads(c, X, T, h, d, ldx, (ada_dtype)dt, tau, ri, ric, ro, roc, ai, ac, mi, mc, gr, gc,
                                (uint32_t)flags, s));
}
static PyObject* cascade_step_adaptive(PyObject* self, PyObject* const* a, Py_ssize_t na) {
    ARGS(22);
    H(ada_ctx, c); P(void, X); N(B); N(T); N(d); N(ldx); N(dt); P(double, tau); H(ada_tau_policy, pol); LISTS;
    O(float, turnover); N(flags); H(void, s);
    CALL(ada_cascade_step_adaptive(c, X, B, T, d, ldx, (ada_dtype)dt, tau, pol, ri, ric, ro, roc, ai, ac, mi, mc,
                                   gr, gc, turnover, (uint32_t)flags, s));
}
static PyObject* nearest_rep(PyObject* self, PyObject* const* a, Py_ssize_t na) {
    ARGS(12);
    H(ada_ctx, c); P(void, X); N(B); N(T); N(d); N(ldx); N(dt);
    P(int32_t, ri); P(int32_t, ric); P(int32_t, near); O(float, gamma); H(void, s);
    CALL(ada_nearest_rep(c, X, B, T, d, ldx, (ada_dtype)dt, ri, ric, near, gamma, s));
}
static PyObject* attention_reps(PyObject* self, PyObject* const* a, Py_ssize_t na) {
    ARGS(16);
    H(ada_ctx, c); P(void, Q); P(void, K); P(void, V); N(T); N(h); N(dh); N(ld); N(dt);
    P(int32_t, ri); P(int32_t, ric); O(int32_t, near); P(float, out); N(ldo); N(flags); H(void, s);
    CALL(ada_attention_reps(c, Q, K, V, T, h, dh, ld, (ada_dtype)dt, ri, ric, near, out, ldo, (uint32_t)flags, s));
}

#define METHOD(f) {#f, (PyCFunction)(void (*)(void))f, METH_FASTCALL, NULL}
static PyMethodDef methods[] = {METHOD(select_full), METHOD(select_full_heads), METHOD(cascade_step),
                                METHOD(cascade_step_heads), METHOD(cascade_step_adaptive), METHOD(nearest_rep),
                                METHOD(attention_reps), {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_pycall", NULL, -1, methods};

PyMODINIT_FUNC PyInit__pycall(void) {
    s_data_ptr = PyUnicode_InternFromString("data_ptr");
    return s_data_ptr == NULL ? NULL : PyModule_Create(&module);
}
