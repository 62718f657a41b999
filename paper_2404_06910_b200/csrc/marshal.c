/* Argument marshalling for the Python front end: turns one call's Python arguments into the C ABI's and makes the call.
 *
 * Converting a decode step's twenty arguments with ctypes and reading a dozen tensors' addresses from Python took as long as
 * the launch itself (host time of a decode call 9.0 us, 6.1 through this module; a prefill call 15.1 and 7.8).  Here a tensor
 * costs two method calls and a number a conversion.
 * bind() receives the addresses of the library's entry points, call(index, ...) the arguments in the order of sp.h:
 * tensors (or None) for pointers, numbers otherwise.  What the arguments mean is checked by the library. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>

#include "../../include/sp.h"

#define MAX_FN 32
#define MAX_ARG 28

typedef union { void *p; long long q; double d; } val;

static struct { void *fn; char kinds[MAX_ARG + 1]; } entry[MAX_FN];
static PyObject *s_data_ptr, *s_is_contiguous;

/* kinds: t contiguous tensor or None, r tensor as it is (strided), a address, i integer, d floating point */
static int convert(char kind, PyObject *o, val *v)
{
    if (kind == 't' || kind == 'r') {
        if (o == Py_None) { v->p = NULL; return 0; }
        if (kind == 't') {
            PyObject *c = PyObject_CallMethodNoArgs(o, s_is_contiguous);
            if (!c) return -1;
            const int yes = c == Py_True;
            Py_DECREF(c);
            if (!yes) { PyErr_SetString(PyExc_AssertionError, "tensors must be contiguous"); return -1; }
        }
        PyObject *a = PyObject_CallMethodNoArgs(o, s_data_ptr);
        if (!a) return -1;
        v->p = PyLong_AsVoidPtr(a);
        Py_DECREF(a);
    } else if (kind == 'a') {
        v->p = PyLong_AsVoidPtr(o);
    } else if (kind == 'i') {
        v->q = PyLong_AsLongLong(o);
    } else {
        v->d = PyFloat_AsDouble(o);
    }
    return PyErr_Occurred() ? -1 : 0;
}

static PyObject *bind(PyObject *self, PyObject *args)
{
    int i;
    PyObject *address;
    const char *kinds;
    (void)self;
    if (!PyArg_ParseTuple(args, "iOs", &i, &address, &kinds)) return NULL;
    if (i < 0 || i >= MAX_FN || strlen(kinds) > MAX_ARG) { PyErr_SetString(PyExc_ValueError, "bind: index or argument list"); return NULL; }
    entry[i].fn = PyLong_AsVoidPtr(address);
    strcpy(entry[i].kinds, kinds);
    if (PyErr_Occurred()) return NULL;
    Py_RETURN_NONE;
}

/* The order of the cases is the order in which binding.py binds the entry points.  A call goes through the type that sp.h
 * declares: a changed parameter does not compile (build.py makes the conversions between integers and pointers errors). */
#define CALL(name) ((__typeof__(&name))f)
static int invoke(int i, const val *v)
{
    void *f = entry[i].fn;
    switch (i) {
    case 0:      /* sp_rope_apply */
        return CALL(sp_rope_apply)(
            v[0].p, v[1].p, v[2].q, v[3].q, (int)v[4].q, (int)v[5].q, (int)v[6].q, v[7].d, (int)v[8].q, (int)v[9].q, v[10].p);
    case 1:      /* sp_rope_apply_pair */
        return CALL(sp_rope_apply_pair)(
            v[0].p, v[1].q, (int)v[2].q, v[3].p, v[4].q, (int)v[5].q, v[6].p, v[7].q, (int)v[8].q, (int)v[9].q, v[10].d, (int)v[11].q,
            (int)v[12].q, v[13].p);
    case 2:      /* sp_superpose_prefill */
        return CALL(sp_superpose_prefill)(
            v[0].p, v[1].p, v[2].p, v[3].p, (int)v[4].q, (int)v[5].q, (int)v[6].q, (float)v[7].d, (int)v[8].q, v[9].p, v[10].p, v[11].p,
            (size_t)v[12].q, (int)v[13].q, v[14].p);
    case 3:      /* sp_superpose_prefill_alibi */
        return CALL(sp_superpose_prefill_alibi)(
            v[0].p, v[1].p, v[2].p, v[3].p, v[4].p, v[5].p, (int)v[6].q, (int)v[7].q, (int)v[8].q, (float)v[9].d, (int)v[10].q, v[11].p,
            v[12].p, v[13].p, (size_t)v[14].q, (int)v[15].q, v[16].p);
    case 4:      /* sp_superpose_prefill_rope */
        return CALL(sp_superpose_prefill_rope)(
            v[0].p, v[1].p, v[2].p, v[3].p, v[4].p, v[5].d, (int)v[6].q, (int)v[7].q, (int)v[8].q, (int)v[9].q, (float)v[10].d, v[11].p,
            v[12].p, v[13].p, (size_t)v[14].q, (int)v[15].q, v[16].p);
    case 5:      /* sp_path_scores */
        return CALL(sp_path_scores)(
            v[0].p, v[1].q, v[2].p, v[3].p, v[4].q, (int)v[5].q, (int)v[6].q, v[7].p, v[8].p, v[9].p, v[10].p, v[11].p, (size_t)v[12].q,
            (int)v[13].q, v[14].p);
    case 6:      /* sp_prune_topk */
        return CALL(sp_prune_topk)(v[0].p, v[1].p, (int)v[2].q, (int)v[3].q, v[4].p, v[5].p, v[6].p);
    case 7:      /* sp_pruned_decode */
        return CALL(sp_pruned_decode)(
            v[0].p, v[1].p, v[2].p, v[3].p, v[4].p, (int)v[5].q, v[6].p, v[7].p, v[8].p, (int)v[9].q, v[10].q, (int)v[11].q, (int)v[12].q,
            (int)v[13].q, (float)v[14].d, v[15].p, v[16].p, v[17].p, (size_t)v[18].q, (int)v[19].q, v[20].p);
    case 8:      /* sp_pruned_decode_alibi */
        return CALL(sp_pruned_decode_alibi)(
            v[0].p, v[1].p, v[2].p, v[3].p, v[4].p, (int)v[5].q, v[6].p, v[7].p, v[8].p, (int)v[9].q, v[10].q, v[11].p, v[12].p, v[13].p,
            v[14].p, (int)v[15].q, (int)v[16].q, (int)v[17].q, (float)v[18].d, v[19].p, v[20].p, v[21].p, (size_t)v[22].q, (int)v[23].q, v[24].p);
    case 9:      /* sp_pruned_decode_rope */
        return CALL(sp_pruned_decode_rope)(
            v[0].p, v[1].p, v[2].p, v[3].p, v[4].p, (int)v[5].q, v[6].p, v[7].p, v[8].p, (int)v[9].q, v[10].q, v[11].p, v[12].d, (int)v[13].q,
            (int)v[14].q, (int)v[15].q, (int)v[16].q, (float)v[17].d, v[18].p, v[19].p, (int)v[20].q, v[21].p);
    case 10:     /* sp_pruned_decode_static */
        return CALL(sp_pruned_decode_static)(
            v[0].p, v[1].p, v[2].p, v[3].p, v[4].p, (int)v[5].q, v[6].p, v[7].p, v[8].p, (int)v[9].q, v[10].q, (int)v[11].q, (int)v[12].q,
            (int)v[13].q, (float)v[14].d, v[15].p, v[16].p, (int)v[17].q, v[18].p);
    }
    return -1;
}

static PyObject *call(PyObject *self, PyObject *const *args, Py_ssize_t n)
{
    val v[MAX_ARG];
    int rc;
    (void)self;
    const long i = n > 0 ? PyLong_AsLong(args[0]) : -1;
    if (i < 0 || i >= MAX_FN || !entry[i].fn || n - 1 != (Py_ssize_t)strlen(entry[i].kinds)) {
        if (!PyErr_Occurred()) PyErr_SetString(PyExc_TypeError, "call: unknown entry point or wrong number of arguments");
        return NULL;
    }
    for (Py_ssize_t k = 0; k < n - 1; ++k)
        if (convert(entry[i].kinds[k], args[k + 1], &v[k])) return NULL;
    Py_BEGIN_ALLOW_THREADS
    rc = invoke((int)i, v);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

static PyMethodDef methods[] = {
    {"bind", bind, METH_VARARGS, "bind(index, address, kinds)"},
    {"call", (PyCFunction)(void (*)(void))call, METH_FASTCALL, "call(index, *arguments) -> status"},
    {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_marshal", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__marshal(void)
{
    s_data_ptr = PyUnicode_InternFromString("data_ptr");
    s_is_contiguous = PyUnicode_InternFromString("is_contiguous");
    return s_data_ptr && s_is_contiguous ? PyModule_Create(&module) : NULL;
}
