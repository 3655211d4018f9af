/*
 * Argument marshalling of thc.Context in C: tensors -> device addresses, then the C ABI of
 * include/thc.h.  A round is four calls with up to 2 n + 4 addresses each; collected in Python
 * (a ctypes array per pointer list) that took longer than the kernels of a small round.
 *
 * Every function takes the context handle as an integer (0 where the call has none) and returns
 * the library's return code.  A tensor argument is anything with data_ptr(), a raw address as int,
 * or None (NULL).  A stream is None (the current stream of the current device), a raw handle as
 * int, or anything with cuda_stream.
 */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>

#include "../../include/thc.h"

static PyObject *s_data_ptr, *s_nbytes, *s_cuda_stream;   /* interned names */
static PyObject *get_device, *get_raw_stream;             /* torch._C, looked up on first use */

/* Address of one argument; -1 with an exception set on failure. */
static int address(PyObject *o, void **p)
{
    if (o == Py_None) { *p = NULL; return 0; }
    if (PyLong_Check(o)) {
        *p = PyLong_AsVoidPtr(o);
        return PyErr_Occurred() ? -1 : 0;
    }
    PyObject *v = PyObject_CallMethodNoArgs(o, s_data_ptr);
    if (v == NULL) return -1;
    *p = PyLong_AsVoidPtr(v);
    Py_DECREF(v);
    return PyErr_Occurred() ? -1 : 0;
}

/* A list of addresses.  Longer lists than the library serves (THC_MAX_WORKERS) keep their length,
 * which the library refuses before it reads the array. */
typedef struct { void *p[THC_MAX_WORKERS]; uint32_t n; int given; } list_t;

static int addresses(PyObject *o, list_t *out)
{
    out->n = 0;
    out->given = o != Py_None;
    if (!out->given) return 0;
    PyObject *seq = PySequence_Fast(o, "a sequence of tensors is expected");
    if (seq == NULL) return -1;
    const Py_ssize_t n = PySequence_Fast_GET_SIZE(seq);
    int rc = 0;
    for (Py_ssize_t i = 0; rc == 0 && i < n && i < (Py_ssize_t)THC_MAX_WORKERS; ++i)
        rc = address(PySequence_Fast_GET_ITEM(seq, i), &out->p[i]);
    out->n = (uint32_t)n;
    Py_DECREF(seq);
    return rc;
}

static void **array_of(list_t *l) { return l->given ? l->p : NULL; }

/* Another list (packed, rotated, ...) has to have an entry for each of the first one's n. */
static int same_length(const list_t *a, const list_t *b)
{
    if (!b->given || b->n >= a->n) return 0;
    PyErr_SetString(PyExc_ValueError, "the lists of per-worker tensors differ in length");
    return -1;
}

static int number(PyObject *o, uint64_t *v)
{
    *v = PyLong_AsUnsignedLongLong(o);
    return *v == (uint64_t)-1 && PyErr_Occurred() ? -1 : 0;
}

static int number32(PyObject *o, uint32_t *v)
{
    const unsigned long long x = PyLong_AsUnsignedLongLongMask(o);
    if (x == (unsigned long long)-1 && PyErr_Occurred()) return -1;
    *v = (uint32_t)x;
    return 0;
}

/* Workspace: its address and its size in bytes (None: no workspace). */
static int workspace(PyObject *o, void **p, uint64_t *bytes)
{
    *bytes = 0;
    if (address(o, p) != 0) return -1;
    if (o == Py_None) return 0;
    PyObject *v = PyObject_GetAttr(o, s_nbytes);
    if (v == NULL) return -1;
    const int rc = number(v, bytes);
    Py_DECREF(v);
    return rc;
}

static int stream_of(PyObject *o, void **st)
{
    PyObject *v;
    if (PyLong_Check(o)) {
        *st = PyLong_AsVoidPtr(o);
        return PyErr_Occurred() ? -1 : 0;
    }
    if (o == Py_None) {
        if (get_raw_stream == NULL) {
            PyObject *c = PyImport_ImportModule("torch._C");
            if (c == NULL) return -1;
            get_device = PyObject_GetAttrString(c, "_cuda_getDevice");
            get_raw_stream = get_device ? PyObject_GetAttrString(c, "_cuda_getCurrentRawStream") : NULL;
            Py_DECREF(c);
            if (get_raw_stream == NULL) return -1;
        }
        PyObject *dev = PyObject_CallNoArgs(get_device);
        if (dev == NULL) return -1;
        v = PyObject_CallOneArg(get_raw_stream, dev);
        Py_DECREF(dev);
    } else {
        v = PyObject_GetAttr(o, s_cuda_stream);
    }
    if (v == NULL) return -1;
    *st = PyLong_AsVoidPtr(v);
    Py_DECREF(v);
    return PyErr_Occurred() ? -1 : 0;
}

static int want(Py_ssize_t got, Py_ssize_t n)
{
    if (got == n) return 0;
    PyErr_Format(PyExc_TypeError, "%zd arguments are expected, got %zd", n, got);
    return -1;
}

#define ARGS PyObject *self, PyObject *const *a, Py_ssize_t na
#define BEGIN(count)                                                            \
    void *ctx_p, *st;                                                           \
    (void)self;                                                                 \
    if (want(na, count) || address(a[0], &ctx_p) || stream_of(a[na - 1], &st)) return NULL; \
    thc_ctx *ctx = (thc_ctx *)ctx_p;                                            \
    (void)ctx;                                                                  \
    int rc
#define CALL(expr)                                                              \
    Py_BEGIN_ALLOW_THREADS                                                      \
    rc = (expr);                                                                \
    Py_END_ALLOW_THREADS                                                        \
    return PyLong_FromLong(rc)

typedef const void *const *in_t;
typedef float *const *rot_t;

/* (handle, grads, d, scales, workspace, stream) */
static PyObject *b_prepare(ARGS)
{
    BEGIN(6);
    list_t g;
    uint64_t d, wb;
    void *scales, *ws;
    if (addresses(a[1], &g) || number(a[2], &d) || address(a[3], &scales) || workspace(a[4], &ws, &wb)) return NULL;
    CALL(thc_prepare(ctx, (in_t)g.p, g.n, d, scales, ws, wb, st));
}

/* (handle, grads, d, round, scales, rotated, workspace, stream) */
static PyObject *b_prepare_minmax(ARGS)
{
    BEGIN(8);
    list_t g, r;
    uint64_t d, wb;
    uint32_t rnd;
    void *scales, *ws;
    if (addresses(a[1], &g) || number(a[2], &d) || number32(a[3], &rnd) || address(a[4], &scales) ||
        addresses(a[5], &r) || same_length(&g, &r) || workspace(a[6], &ws, &wb)) return NULL;
    CALL(thc_prepare_minmax(ctx, (in_t)g.p, g.n, d, rnd, scales, (rot_t)array_of(&r), ws, wb, st));
}

/* (handle, grads, worker_base, d, round, scales, packed, rotated, workspace, stream) */
static PyObject *compress(ARGS, int with_scales)
{
    BEGIN(10);
    list_t g, p, r;
    uint64_t d, wb;
    uint32_t base, rnd;
    void *scales, *ws;
    if (addresses(a[1], &g) || number32(a[2], &base) || number(a[3], &d) || number32(a[4], &rnd) ||
        address(a[5], &scales) || addresses(a[6], &p) || addresses(a[7], &r) || same_length(&g, &p) ||
        same_length(&g, &r) || workspace(a[8], &ws, &wb)) return NULL;
    CALL(with_scales ? thc_prepare_compress(ctx, (in_t)g.p, g.n, base, d, rnd, scales, p.p, (rot_t)array_of(&r), ws, wb, st)
                     : thc_compress(ctx, (in_t)g.p, g.n, base, d, rnd, scales, p.p, (rot_t)array_of(&r), ws, wb, st));
}
static PyObject *b_compress(ARGS) { return compress(self, a, na, 0); }
static PyObject *b_prepare_compress(ARGS) { return compress(self, a, na, 1); }

/* (handle, rotated, worker_base, d, round, scales, packed, stream) */
static PyObject *b_quantize_rotated(ARGS)
{
    BEGIN(8);
    list_t r, p;
    uint64_t d;
    uint32_t base, rnd;
    void *scales;
    if (addresses(a[1], &r) || number32(a[2], &base) || number(a[3], &d) || number32(a[4], &rnd) ||
        address(a[5], &scales) || addresses(a[6], &p) || same_length(&r, &p)) return NULL;
    CALL(thc_quantize_rotated(ctx, (const float *const *)r.p, r.n, base, d, rnd, scales, p.p, st));
}

/* (handle, packed, d, total, stream) */
static PyObject *b_aggregate(ARGS)
{
    BEGIN(5);
    list_t p;
    uint64_t d;
    void *total;
    if (addresses(a[1], &p) || number(a[2], &d) || address(a[3], &total)) return NULL;
    CALL(thc_aggregate(ctx, (in_t)p.p, p.n, d, total, st));
}

/* (handle, total, divisor, d, round, scales, out, workspace, stream) */
static PyObject *b_decompress(ARGS)
{
    BEGIN(9);
    uint64_t d, wb;
    uint32_t divisor, rnd;
    void *total, *scales, *out, *ws;
    if (address(a[1], &total) || number32(a[2], &divisor) || number(a[3], &d) || number32(a[4], &rnd) ||
        address(a[5], &scales) || address(a[6], &out) || workspace(a[7], &ws, &wb)) return NULL;
    CALL(thc_decompress(ctx, total, divisor, d, rnd, scales, out, ws, wb, st));
}

/* (handle, packed, d, round, scales, out, total, workspace, stream) */
static PyObject *b_aggregate_decompress(ARGS)
{
    BEGIN(9);
    list_t p;
    uint64_t d, wb;
    uint32_t rnd;
    void *scales, *out, *total, *ws;
    if (addresses(a[1], &p) || number(a[2], &d) || number32(a[3], &rnd) || address(a[4], &scales) ||
        address(a[5], &out) || address(a[6], &total) || workspace(a[7], &ws, &wb)) return NULL;
    CALL(thc_aggregate_decompress(ctx, (in_t)p.p, p.n, d, rnd, scales, out, total, ws, wb, st));
}

/* (handle, grads, packed, d, round, scales, ef, workspace, stream) */
static PyObject *b_error_feedback(ARGS)
{
    BEGIN(9);
    list_t g, p, e;
    uint64_t d, wb;
    uint32_t rnd;
    void *scales, *ws;
    if (addresses(a[1], &g) || addresses(a[2], &p) || number(a[3], &d) || number32(a[4], &rnd) ||
        address(a[5], &scales) || addresses(a[6], &e) || same_length(&g, &p) || same_length(&g, &e) ||
        workspace(a[7], &ws, &wb)) return NULL;
    CALL(thc_error_feedback(ctx, (in_t)g.p, (in_t)p.p, g.n, d, rnd, scales, (rot_t)e.p, ws, wb, st));
}

/* (handle, grads, ef, d, stream) */
static PyObject *b_accumulate_error(ARGS)
{
    BEGIN(5);
    list_t g, e;
    uint64_t d;
    if (addresses(a[1], &g) || addresses(a[2], &e) || same_length(&g, &e) || number(a[3], &d)) return NULL;
    CALL(thc_accumulate_error(ctx, (rot_t)g.p, (const float *const *)e.p, g.n, d, st));
}

/* (0, grads, d, log2_block, in_dtype, t_p, scales, status, stream) */
static PyObject *b_prepare_noalloc(ARGS)
{
    BEGIN(9);
    list_t g;
    uint64_t d;
    uint32_t k, dtype;
    void *scales, *status;
    const double t_p = na > 5 ? PyFloat_AsDouble(a[5]) : 0.0;
    if (PyErr_Occurred()) return NULL;
    if (addresses(a[1], &g) || number(a[2], &d) || number32(a[3], &k) || number32(a[4], &dtype) ||
        address(a[6], &scales) || address(a[7], &status)) return NULL;
    CALL(thc_prepare_noalloc((in_t)g.p, g.n, d, k, dtype, t_p, scales, status, st));
}

#define ENTRY(name) {#name, (PyCFunction)(void (*)(void))b_##name, METH_FASTCALL, NULL}
static PyMethodDef methods[] = {
    ENTRY(prepare), ENTRY(prepare_minmax), ENTRY(compress), ENTRY(prepare_compress), ENTRY(quantize_rotated),
    ENTRY(aggregate), ENTRY(decompress), ENTRY(aggregate_decompress), ENTRY(error_feedback),
    ENTRY(accumulate_error), ENTRY(prepare_noalloc), {NULL, NULL, 0, NULL}};

static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_binding", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__binding(void)
{
    s_data_ptr = PyUnicode_InternFromString("data_ptr");
    s_nbytes = PyUnicode_InternFromString("nbytes");
    s_cuda_stream = PyUnicode_InternFromString("cuda_stream");
    if (s_data_ptr == NULL || s_nbytes == NULL || s_cuda_stream == NULL) return NULL;
    return PyModule_Create(&module);
}
