/* The Python binding's calls of a step, as vector-call functions.
 *
 * Bound by host work: a round's one call has 18 arguments, which ctypes converts in 5 us and a Python
 * wrapper prepares in as much again (one core of the host), longer than a small round takes on the GPU.
 * Here an argument costs some tens of nanoseconds.  Device addresses are objects with a data_ptr()
 * method, integers, or None (NULL); the answer is the C call's status.  No state is kept but the
 * addresses of the library's entry points and the class of the rules, which bind() receives from the Python
 * side, so that any build of the library can stand behind them. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>
#include <string.h>

#include "dq.h"

static PyObject* g_data_ptr; /* the string "data_ptr" */
static PyObject* g_rule;     /* the class dq.Rule */

/* An integer argument: what int() makes of it (a number that lives in a tensor or an array among them). */
static int to_integer(PyObject* o, uint64_t* v)
{
    PyObject* n;
    if (PyLong_CheckExact(o)) {
        *v = PyLong_AsUnsignedLongLongMask(o);
        return (*v == (uint64_t)-1 && PyErr_Occurred()) ? -1 : 0;
    }
    n = PyNumber_Long(o);
    if (!n) return -1;
    *v = PyLong_AsUnsignedLongLongMask(n);
    Py_DECREF(n);
    return (*v == (uint64_t)-1 && PyErr_Occurred()) ? -1 : 0;
}

/* A device address: None (NULL), an integer, or what the object's data_ptr() says.  Nothing else is one: a number
 * given in the place of a tensor must not reach a kernel as a pointer. */
static int to_address(PyObject* o, uint64_t* v)
{
    PyObject* n;
    if (o == Py_None) {
        *v = 0;
        return 0;
    }
    if (PyLong_Check(o)) {
        *v = PyLong_AsUnsignedLongLongMask(o);
        return (*v == (uint64_t)-1 && PyErr_Occurred()) ? -1 : 0;
    }
    n = PyObject_VectorcallMethod(g_data_ptr, &o, 1 | PY_VECTORCALL_ARGUMENTS_OFFSET, NULL);
    if (!n) return -1;
    if (n == Py_None) {
        *v = 0;
    } else if (PyLong_Check(n)) {
        *v = PyLong_AsUnsignedLongLongMask(n);
    } else {
        PyErr_SetString(PyExc_TypeError, "data_ptr() did not return an address");
    }
    Py_DECREF(n);
    return PyErr_Occurred() ? -1 : 0;
}

/* The rule travels as the binding's ctypes structure of dq_rule_t's layout, and as no other object. */
static int to_rule(PyObject* o, dq_rule_t* r)
{
    Py_buffer b;
    if (!PyObject_TypeCheck(o, (PyTypeObject*)g_rule)) {
        PyErr_SetString(PyExc_TypeError, "a dq.Rule is wanted");
        return -1;
    }
    if (PyObject_GetBuffer(o, &b, PyBUF_SIMPLE) != 0) return -1;
    if (b.len < (Py_ssize_t)sizeof(dq_rule_t)) {
        PyBuffer_Release(&b);
        PyErr_SetString(PyExc_TypeError, "a dq.Rule is wanted");
        return -1;
    }
    memcpy(r, b.buf, sizeof(*r));
    PyBuffer_Release(&b);
    return 0;
}

/* A float argument: what float() makes of it. */
static int to_float(PyObject* o, float* f)
{
    PyObject* n;
    if (PyFloat_CheckExact(o)) {
        *f = (float)PyFloat_AS_DOUBLE(o);
        return 0;
    }
    n = PyNumber_Float(o);
    if (!n) return -1;
    *f = (float)PyFloat_AS_DOUBLE(n);
    Py_DECREF(n);
    return 0;
}

enum { MAX_ARGS = 18 };

/* Arguments by their kinds, a letter each: p a device address, i an integer, r the rule, f a float. */
static int convert(PyObject* const* args, Py_ssize_t n, const char* kinds, uint64_t* v, dq_rule_t* r, float* f)
{
    const Py_ssize_t want = (Py_ssize_t)strlen(kinds);
    Py_ssize_t i;
    if (n != want) {
        PyErr_Format(PyExc_TypeError, "%zd arguments are wanted, got %zd", want, n);
        return -1;
    }
    for (i = 0; i < n; ++i) {
        if (kinds[i] == 'i') {
            if (to_integer(args[i], &v[i]) != 0) return -1;
        } else if (kinds[i] == 'r') {
            if (to_rule(args[i], r) != 0) return -1;
        } else if (kinds[i] == 'f') {
            if (to_float(args[i], f) != 0) return -1;
        } else if (to_address(args[i], &v[i]) != 0) {
            return -1;
        }
    }
    return 0;
}

#define P(i) ((void*)(uintptr_t)v[i])
#define I64(i) ((int64_t)v[i])
#define I32(i) ((int32_t)v[i])
#define U32(i) ((uint32_t)v[i])

#define ENTRY(name, kinds, call)                                                                    \
    static __typeof__(&dq_##name) p_##name;                                                         \
    static PyObject* py_##name(PyObject* self, PyObject* const* args, Py_ssize_t n)                 \
    {                                                                                               \
        uint64_t v[MAX_ARGS];                                                                       \
        dq_rule_t r;                                                                                \
        float f = 0.0f;                                                                             \
        int rc;                                                                                     \
        (void)self; (void)f; (void)r;                                                               \
        if (convert(args, n, kinds, v, &r, &f) != 0) return NULL;                                   \
        Py_BEGIN_ALLOW_THREADS                                                                      \
        rc = p_##name call;                                                                         \
        Py_END_ALLOW_THREADS                                                                        \
        return PyLong_FromLong(rc);                                                                 \
    }

ENTRY(bucket_norms, "ppiippp", (P(0), P(1), I64(2), I32(3), P(4), P(5), P(6)))
ENTRY(tensor_norms, "ppiippipp", (P(0), P(1), I64(2), I32(3), P(4), P(5), (size_t)v[6], P(7), P(8)))
ENTRY(choose_bits, "ppirppipp", (P(0), P(1), I32(2), &r, P(4), P(5), (size_t)v[6], P(7), P(8)))
ENTRY(quantize_pack, "ppiippiipipp", (P(0), P(1), I64(2), I32(3), P(4), P(5), v[6], U32(7), P(8), I64(9), P(10), P(11)))
ENTRY(quantize_pack_worker, "ppiippiiipipp",
      (P(0), P(1), I64(2), I32(3), P(4), P(5), v[6], U32(7), U32(8), P(9), I64(10), P(11), P(12)))
ENTRY(norms_quantize_pack, "ppiipiippipp", (P(0), P(1), I64(2), I32(3), P(4), v[5], U32(6), P(7), P(8), I64(9), P(10), P(11)))
ENTRY(norms_quantize_pack_worker, "ppiipiiippipp",
      (P(0), P(1), I64(2), I32(3), P(4), v[5], U32(6), U32(7), P(8), P(9), I64(10), P(11), P(12)))
ENTRY(unpack_dequant_average, "ppipipppp", (P(0), P(1), I64(2), P(3), I32(4), P(5), P(6), P(7), P(8)))
ENTRY(unpack_average_update, "ppipipfppp", (P(0), P(1), I64(2), P(3), I32(4), P(5), f, P(7), P(8), P(9)))
ENTRY(norms_choose_bits, "ppiiprppipp", (P(0), P(1), I64(2), I32(3), P(4), &r, P(6), P(7), (size_t)v[8], P(9), P(10)))
ENTRY(quantize_average, "ppiippiipipifpp",
      (P(0), P(1), I64(2), I32(3), P(4), P(5), v[6], U32(7), P(8), I64(9), P(10), I32(11), f, P(13), P(14)))
ENTRY(norms_quantize_average, "ppiipiippipifrpipp",
      (P(0), P(1), I64(2), I32(3), P(4), v[5], U32(6), P(7), P(8), I64(9), P(10), I32(11), f, &r, P(14), (size_t)v[15], P(16), P(17)))

#define EACH(X)                                                                                     \
    X(bucket_norms) X(tensor_norms) X(choose_bits) X(quantize_pack) X(quantize_pack_worker)         \
    X(norms_quantize_pack) X(norms_quantize_pack_worker) X(unpack_dequant_average)                  \
    X(unpack_average_update) X(norms_choose_bits) X(quantize_average) X(norms_quantize_average)

/* bind({"dq_...": address}, Rule): the entry points of the library that was loaded, the class of the rules. */
static PyObject* py_bind(PyObject* self, PyObject* args)
{
    PyObject *dict, *rule, *old;
    (void)self;
    if (!PyArg_ParseTuple(args, "O!O!", &PyDict_Type, &dict, &PyType_Type, &rule)) return NULL;
#define X(name)                                                                                     \
    {                                                                                               \
        PyObject* o = PyDict_GetItemString(dict, "dq_" #name);                                      \
        uint64_t a = 0;                                                                             \
        if (!o || to_address(o, &a) != 0 || !a) {                                                       \
            if (!PyErr_Occurred()) PyErr_SetString(PyExc_KeyError, "dq_" #name);                    \
            return NULL;                                                                            \
        }                                                                                           \
        p_##name = (__typeof__(p_##name))(uintptr_t)a;                                              \
    }
    EACH(X)
#undef X
    old = g_rule;
    Py_INCREF(rule);
    g_rule = rule;
    Py_XDECREF(old);
    Py_RETURN_NONE;
}

static PyMethodDef methods[] = {
    {"bind", py_bind, METH_VARARGS, NULL},
#define X(name) {#name, (PyCFunction)(void (*)(void))py_##name, METH_FASTCALL, NULL},
    EACH(X)
#undef X
    {NULL, NULL, 0, NULL}};

static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_dqcall", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__dqcall(void)
{
    g_data_ptr = PyUnicode_InternFromString("data_ptr");
    if (!g_data_ptr) return NULL;
    return PyModule_Create(&module);
}
