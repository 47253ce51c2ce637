/* Call path from Python into the C ABI for the entry points that a serving loop calls per step: a CPython extension that
 * takes plain integers (addresses, sizes, a stream) and passes them on.  Marshalling only, like the ctypes binding beside
 * it, which costs 2.3 microseconds for the 17 arguments of a forward (and tens for the prefix sums of a packed batch)
 * where this takes a few tenths.  The library is not linked: the binding hands over the addresses of its functions.
 * As in ctypes, the interpreter lock is released around every call: a launch waits while the stream's queue is full, and the
 * table copy of a packed batch may wait for the stream, and neither may stop the other threads of a server. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>
#include <stdlib.h>

#include "efq.h"

typedef efq_status_t (*attention_fn)(const void*, const void*, const void*, float*, int, int, int, int64_t, int64_t, int, int,
                                     float, const efq_params_t*, void*, size_t, const efq_debug_t*, void*);
typedef efq_status_t (*etq_attention_fn)(const void*, const void*, const void*, float*, int, int, int, int64_t, int64_t, int, int,
                                         float, int, void*, size_t, const efq_debug_t*, void*);
typedef efq_status_t (*probgen_fn)(const float*, int64_t, const float*, int64_t, int64_t, float, const efq_params_t*, uint8_t*,
                                   uint8_t*, void*);
typedef efq_status_t (*etq_probgen_fn)(const float*, int64_t, const float*, int64_t, int64_t, float, int, uint8_t*, uint8_t*, void*);
typedef efq_status_t (*varlen_fn)(const void*, const void*, const void*, float*, const int64_t*, const int64_t*, int, int, int, int,
                                  int, float, int, const efq_params_t*, void*, size_t, void*);
typedef size_t (*varlen_bytes_fn)(const int64_t*, const int64_t*, int, int, int, int);

static struct {
    attention_fn attention;
    etq_attention_fn etq_attention;
    probgen_fn probgen;
    etq_probgen_fn etq_probgen;
    varlen_fn varlen;
    varlen_bytes_fn varlen_bytes;
} fn;

/* The call without the interpreter lock; its arguments are plain C values by then. */
#define UNLOCKED(type, call) type st; Py_BEGIN_ALLOW_THREADS st = call; Py_END_ALLOW_THREADS

/* Arguments are converted first and errors looked at once: a conversion that fails leaves the exception set. */
static void* ptr(PyObject* o) { return o == Py_None ? NULL : (void*)(uintptr_t)PyLong_AsUnsignedLongLong(o); }
static int64_t i64(PyObject* o) { return PyLong_AsLongLong(o); }
static int i32(PyObject* o) { return (int)PyLong_AsLong(o); }
static float f32(PyObject* o) { return (float)PyFloat_AsDouble(o); }

static int want(Py_ssize_t got, Py_ssize_t n)
{
    if (fn.attention == NULL) { PyErr_SetString(PyExc_RuntimeError, "efq_fastcall: the library's functions have not been set"); return 0; }
    if (got != n) { PyErr_Format(PyExc_TypeError, "efq_fastcall: %zd arguments expected, got %zd", n, got); return 0; }
    return 1;
}

static PyObject* set_functions(PyObject* self, PyObject* const* a, Py_ssize_t n)
{
    (void)self;
    if (n != 6) { PyErr_SetString(PyExc_TypeError, "efq_fastcall.set_functions: six addresses expected"); return NULL; }
    fn.attention = (attention_fn)ptr(a[0]);
    fn.etq_attention = (etq_attention_fn)ptr(a[1]);
    fn.probgen = (probgen_fn)ptr(a[2]);
    fn.etq_probgen = (etq_probgen_fn)ptr(a[3]);
    fn.varlen = (varlen_fn)ptr(a[4]);
    fn.varlen_bytes = (varlen_bytes_fn)ptr(a[5]);
    if (PyErr_Occurred()) return NULL;
    Py_RETURN_NONE;
}

/* q, k, v, o, B, Hq, Hkv, Sq, Sk, d, causal, scale, params or scale mode, workspace, bytes, debug, stream */
static PyObject* attention(PyObject* self, PyObject* const* a, Py_ssize_t n)
{
    (void)self;
    if (!want(n, 17)) return NULL;
    void *q = ptr(a[0]), *k = ptr(a[1]), *v = ptr(a[2]), *o = ptr(a[3]);
    const int B = i32(a[4]), Hq = i32(a[5]), Hkv = i32(a[6]), d = i32(a[9]), causal = i32(a[10]);
    const int64_t Sq = i64(a[7]), Sk = i64(a[8]), bytes = i64(a[14]);
    const float scale = f32(a[11]);
    void *params = ptr(a[12]), *ws = ptr(a[13]), *debug = ptr(a[15]), *stream = ptr(a[16]);
    if (PyErr_Occurred()) return NULL;
    UNLOCKED(efq_status_t, fn.attention(q, k, v, o, B, Hq, Hkv, Sq, Sk, d, causal, scale, params, ws, (size_t)bytes, debug, stream))
    return PyLong_FromLong(st);
}

static PyObject* etq_attention(PyObject* self, PyObject* const* a, Py_ssize_t n)
{
    (void)self;
    if (!want(n, 17)) return NULL;
    void *q = ptr(a[0]), *k = ptr(a[1]), *v = ptr(a[2]), *o = ptr(a[3]);
    const int B = i32(a[4]), Hq = i32(a[5]), Hkv = i32(a[6]), d = i32(a[9]), causal = i32(a[10]), mode = i32(a[12]);
    const int64_t Sq = i64(a[7]), Sk = i64(a[8]), bytes = i64(a[14]);
    const float scale = f32(a[11]);
    void *ws = ptr(a[13]), *debug = ptr(a[15]), *stream = ptr(a[16]);
    if (PyErr_Occurred()) return NULL;
    UNLOCKED(efq_status_t, fn.etq_attention(q, k, v, o, B, Hq, Hkv, Sq, Sk, d, causal, scale, mode, ws, (size_t)bytes, debug, stream))
    return PyLong_FromLong(st);
}

/* scores, ld, row_max, rows, cols, scale, params or scale mode, codes, scales, stream */
static PyObject* probgen(PyObject* self, PyObject* const* a, Py_ssize_t n)
{
    (void)self;
    if (!want(n, 10)) return NULL;
    void *scores = ptr(a[0]), *row_max = ptr(a[2]), *params = ptr(a[6]), *codes = ptr(a[7]), *scales = ptr(a[8]), *stream = ptr(a[9]);
    const int64_t ld = i64(a[1]), rows = i64(a[3]), cols = i64(a[4]);
    const float scale = f32(a[5]);
    if (PyErr_Occurred()) return NULL;
    UNLOCKED(efq_status_t, fn.probgen(scores, ld, row_max, rows, cols, scale, params, codes, scales, stream))
    return PyLong_FromLong(st);
}

static PyObject* etq_probgen(PyObject* self, PyObject* const* a, Py_ssize_t n)
{
    (void)self;
    if (!want(n, 10)) return NULL;
    void *scores = ptr(a[0]), *row_max = ptr(a[2]), *codes = ptr(a[7]), *scales = ptr(a[8]), *stream = ptr(a[9]);
    const int64_t ld = i64(a[1]), rows = i64(a[3]), cols = i64(a[4]);
    const float scale = f32(a[5]);
    const int mode = i32(a[6]);
    if (PyErr_Occurred()) return NULL;
    UNLOCKED(efq_status_t, fn.etq_probgen(scores, ld, row_max, rows, cols, scale, mode, codes, scales, stream))
    return PyLong_FromLong(st);
}

/* A sequence of integers as a C array; NULL with an exception set on failure. */
static int64_t* to_array(PyObject* o, Py_ssize_t* n)
{
    PyObject* s = PySequence_Fast(o, "prefix sums have to be a sequence of integers");
    if (s == NULL) return NULL;
    *n = PySequence_Fast_GET_SIZE(s);
    int64_t* out = malloc(sizeof(int64_t) * (size_t)(*n > 0 ? *n : 1));
    if (out == NULL) { Py_DECREF(s); PyErr_NoMemory(); return NULL; }
    PyObject** items = PySequence_Fast_ITEMS(s);
    for (Py_ssize_t i = 0; i < *n; ++i) {
        if (PyLong_CheckExact(items[i])) {
            out[i] = PyLong_AsLongLong(items[i]);
        } else {                                     /* numpy and torch integers */
            PyObject* x = PyNumber_Long(items[i]);
            out[i] = x == NULL ? -1 : PyLong_AsLongLong(x);
            Py_XDECREF(x);
        }
        if (out[i] == -1 && PyErr_Occurred()) { free(out); Py_DECREF(s); return NULL; }
    }
    Py_DECREF(s);
    return out;
}

/* cu_q, cu_k, total_q, total_k, Hq, Hkv, d, q, k, v, o, causal, scale, producer, params, workspace, bytes, stream
 * -> status, or -1 if the prefix sums do not fit the tensors.  With q None: the bytes the workspace has to have. */
static PyObject* varlen(PyObject* self, PyObject* const* a, Py_ssize_t n)
{
    (void)self;
    if (!want(n, 18)) return NULL;
    Py_ssize_t nq = 0, nk = 0;
    int64_t* cq = to_array(a[0], &nq);
    if (cq == NULL) return NULL;
    int64_t* ck = to_array(a[1], &nk);
    if (ck == NULL) { free(cq); return NULL; }
    const int64_t total_q = i64(a[2]), total_k = i64(a[3]), bytes = i64(a[16]);
    const int Hq = i32(a[4]), Hkv = i32(a[5]), d = i32(a[6]), causal = i32(a[11]), producer = i32(a[13]);
    void *q = ptr(a[7]), *k = ptr(a[8]), *v = ptr(a[9]), *o = ptr(a[10]), *params = ptr(a[14]), *ws = ptr(a[15]), *stream = ptr(a[17]);
    const float scale = f32(a[12]);
    PyObject* result = NULL;
    if (!PyErr_Occurred()) {
        if (nq < 1 || nk != nq || cq[nq - 1] != total_q || ck[nk - 1] != total_k) {
            result = PyLong_FromLong(-1);
        } else if (a[7] == Py_None) {
            UNLOCKED(size_t, fn.varlen_bytes(cq, ck, (int)(nq - 1), Hq, Hkv, d))
            result = PyLong_FromSize_t(st);
        } else {
            UNLOCKED(efq_status_t, fn.varlen(q, k, v, o, cq, ck, (int)(nq - 1), Hq, Hkv, d, causal, scale, producer, params, ws, (size_t)bytes, stream))
            result = PyLong_FromLong(st);
        }
    }
    free(cq);
    free(ck);
    return result;
}

static PyMethodDef methods[] = {
    {"set_functions", (PyCFunction)(void (*)(void))set_functions, METH_FASTCALL, NULL},
    {"attention", (PyCFunction)(void (*)(void))attention, METH_FASTCALL, NULL},
    {"etq_attention", (PyCFunction)(void (*)(void))etq_attention, METH_FASTCALL, NULL},
    {"probgen", (PyCFunction)(void (*)(void))probgen, METH_FASTCALL, NULL},
    {"etq_probgen", (PyCFunction)(void (*)(void))etq_probgen, METH_FASTCALL, NULL},
    {"varlen", (PyCFunction)(void (*)(void))varlen, METH_FASTCALL, NULL},
    {NULL, NULL, 0, NULL},
};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "efq_fastcall", NULL, -1, methods, NULL, NULL, NULL, NULL};
PyMODINIT_FUNC PyInit_efq_fastcall(void) { return PyModule_Create(&module); }
