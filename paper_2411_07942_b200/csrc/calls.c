/* The calls of a synchronisation step as functions of a Python extension module: what binding.py otherwise does through
 * ctypes, with the arguments converted here.  A call of the library costs the host a launch (1.9 us) and its own checks;
 * ctypes added 0.9 to 1.9 us of argument conversion on top: a batched quantisation of 8 shards 4.85 -> 3.1 us, a reduction of 8
 * payloads 4.5 -> 3.2, one token's step over 8 devices, which nothing but the host bounds, 9.65 -> 6.7, a decode layer 8.4 -> 7.2.
 *
 * Every function takes positional arguments in the form that programs pass in earnest -- plain integers, lists or tuples of
 * plain integers -- and returns the library's status.  It returns None without calling anything where an argument has
 * another form or does not fit its C type: binding.py then makes the call through ctypes, which accepts or refuses it as
 * it always has.  The interpreter lock is released during a call, as ctypes does. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>

#include "tpq.h"

enum { MOST = 64 }; /* pointers of a list (a context has at most 64 devices) */

/* the library's entry points, by the order of bind()'s argument */
static struct {
    tpq_status (*calibrate)(tpq_ctx *, int, const void *, int64_t, int64_t, int64_t, void *);
    tpq_status (*pack)(tpq_ctx *, int, const void *, int64_t, int64_t, void *, size_t, void *);
    tpq_status (*batch)(tpq_ctx *, int, int, const void *const *, int64_t, int64_t, void *const *, size_t, void *);
    tpq_status (*reduce)(tpq_ctx *, const void *const *, int, int64_t, void *, tpq_out_dtype, int64_t, void *);
    tpq_status (*reduce_bias)(tpq_ctx *, const void *const *, int, int64_t, void *, tpq_out_dtype, int64_t, const float *, void *);
    tpq_status (*reduce_arrivals)(tpq_ctx *, const void *const *, int, int64_t, void *, tpq_out_dtype, int64_t, const float *,
                                  const uint32_t *, uint32_t, uint64_t, void *);
    tpq_status (*push)(tpq_ctx *, int, const void *, int64_t, int64_t, void *const *, uint32_t *const *, int, size_t, uint32_t, void *);
    tpq_status (*linear)(tpq_ctx *, int, const void *, const void *, int64_t, int64_t, void *, size_t, void *, void *);
} lib;

/* conversions: 1, or 0 where the argument is not of the plain form (no exception is left set) */
static int as_i64(PyObject *o, int64_t *v)
{
    int over;
    if (!PyLong_CheckExact(o)) return 0;
    *v = PyLong_AsLongLongAndOverflow(o, &over);
    return !over;
}
static int as_int(PyObject *o, int *v)
{
    int64_t x;
    if (!as_i64(o, &x) || x != (int)x) return 0;
    *v = (int)x;
    return 1;
}
static int as_u64(PyObject *o, uint64_t *v)
{
    if (!PyLong_CheckExact(o)) return 0;
    *v = PyLong_AsUnsignedLongLong(o);
    if (*v == (uint64_t)-1 && PyErr_Occurred()) { /* negative or above 64 bits */
        PyErr_Clear();
        return 0;
    }
    return 1;
}
static int as_ptr(PyObject *o, void **v)
{
    uint64_t x;
    if (!as_u64(o, &x)) return 0;
    *v = (void *)(uintptr_t)x;
    return 1;
}
static int as_ptr_or_none(PyObject *o, void **v)
{
    *v = NULL;
    return o == Py_None || as_ptr(o, v);
}
static int as_ptrs(PyObject *o, void **v, int *n)
{
    if (!PyList_CheckExact(o) && !PyTuple_CheckExact(o)) return 0;
    const Py_ssize_t len = PySequence_Fast_GET_SIZE(o);
    if (len > MOST) return 0;
    for (Py_ssize_t i = 0; i < len; ++i)
        if (!as_ptr(PySequence_Fast_GET_ITEM(o, i), &v[i])) return 0;
    *n = (int)len;
    return 1;
}
static PyObject *status(tpq_status st) { return PyLong_FromLong((long)st); }

#define CALL(n, conversions, call)                     \
    tpq_status st;                                     \
    void *ctx;                                         \
    if (n_args != n || !as_ptr(a[0], &ctx) || !(conversions)) Py_RETURN_NONE; \
    Py_BEGIN_ALLOW_THREADS                             \
    st = call;                                         \
    Py_END_ALLOW_THREADS                               \
    return status(st)

static PyObject *calibrate_ranges(PyObject *self, PyObject *const *a, Py_ssize_t n_args)
{
    int shard;
    int64_t n_seq, S, stride;
    void *y, *stream;
    CALL(7, as_int(a[1], &shard) && as_ptr(a[2], &y) && as_i64(a[3], &n_seq) && as_i64(a[4], &S) && as_i64(a[5], &stride) && as_ptr(a[6], &stream),
         lib.calibrate(ctx, shard, y, n_seq, S, stride, stream));
}

static PyObject *quantize_pack(PyObject *self, PyObject *const *a, Py_ssize_t n_args)
{
    int shard;
    int64_t T, stride;
    uint64_t cap;
    void *y, *payload, *stream;
    CALL(8, as_int(a[1], &shard) && as_ptr(a[2], &y) && as_i64(a[3], &T) && as_i64(a[4], &stride) && as_ptr(a[5], &payload) && as_u64(a[6], &cap) &&
            as_ptr(a[7], &stream),
         lib.pack(ctx, shard, y, T, stride, payload, cap, stream));
}

static PyObject *quantize_pack_batch(PyObject *self, PyObject *const *a, Py_ssize_t n_args)
{
    int first, n, np;
    int64_t T, stride;
    uint64_t cap;
    void *ys[MOST], *payloads[MOST], *stream;
    CALL(8, as_int(a[1], &first) && as_ptrs(a[2], ys, &n) && as_i64(a[3], &T) && as_i64(a[4], &stride) && as_ptrs(a[5], payloads, &np) && n == np &&
            as_u64(a[6], &cap) && as_ptr(a[7], &stream),
         lib.batch(ctx, first, n, (const void *const *)ys, T, stride, payloads, cap, stream));
}

static PyObject *dequant_reduce(PyObject *self, PyObject *const *a, Py_ssize_t n_args)
{
    int n, dtype;
    int64_t T, stride;
    void *payloads[MOST], *out, *bias, *stream;
    CALL(8, as_ptrs(a[1], payloads, &n) && as_i64(a[2], &T) && as_ptr(a[3], &out) && as_int(a[4], &dtype) && as_i64(a[5], &stride) &&
            as_ptr_or_none(a[6], &bias) && as_ptr(a[7], &stream),
         a[6] == Py_None ? lib.reduce(ctx, (const void *const *)payloads, n, T, out, (tpq_out_dtype)dtype, stride, stream)
                         : lib.reduce_bias(ctx, (const void *const *)payloads, n, T, out, (tpq_out_dtype)dtype, stride, bias, stream));
}

static PyObject *dequant_reduce_arrivals(PyObject *self, PyObject *const *a, Py_ssize_t n_args)
{
    int n, dtype;
    int64_t T, stride;
    uint64_t epoch, timeout;
    void *payloads[MOST], *out, *bias, *arrived, *stream;
    CALL(11, as_ptrs(a[1], payloads, &n) && as_i64(a[2], &T) && as_ptr(a[3], &out) && as_int(a[4], &dtype) && as_i64(a[5], &stride) &&
             as_ptr_or_none(a[6], &bias) && as_ptr(a[7], &arrived) && as_u64(a[8], &epoch) && as_u64(a[9], &timeout) && as_ptr(a[10], &stream),
         lib.reduce_arrivals(ctx, (const void *const *)payloads, n, T, out, (tpq_out_dtype)dtype, stride, bias, arrived, (uint32_t)epoch, timeout, stream));
}

static PyObject *quantize_pack_push(PyObject *self, PyObject *const *a, Py_ssize_t n_args)
{
    int shard, n, na;
    int64_t T, stride;
    uint64_t cap, epoch;
    void *y, *dst[MOST], *arrived[MOST], *stream;
    CALL(10, as_int(a[1], &shard) && as_ptr(a[2], &y) && as_i64(a[3], &T) && as_i64(a[4], &stride) && as_ptrs(a[5], dst, &n) &&
             as_ptrs(a[6], arrived, &na) && n == na && as_u64(a[7], &cap) && as_u64(a[8], &epoch) && as_ptr(a[9], &stream),
         lib.push(ctx, shard, y, T, stride, dst, (uint32_t *const *)arrived, n, cap, (uint32_t)epoch, stream));
}

static PyObject *linear_quantize_pack(PyObject *self, PyObject *const *a, Py_ssize_t n_args)
{
    int shard;
    int64_t T, K;
    uint64_t cap;
    void *x, *w, *payload, *y_slots, *stream;
    CALL(10, as_int(a[1], &shard) && as_ptr(a[2], &x) && as_ptr(a[3], &w) && as_i64(a[4], &T) && as_i64(a[5], &K) && as_ptr(a[6], &payload) &&
             as_u64(a[7], &cap) && as_ptr_or_none(a[8], &y_slots) && as_ptr(a[9], &stream),
         lib.linear(ctx, shard, x, w, T, K, payload, cap, y_slots, stream));
}

/* bind(addresses): the entry points of the loaded library, in the order of `lib` */
static PyObject *bind(PyObject *self, PyObject *addresses)
{
    void *p[MOST];
    int n;
    if (!as_ptrs(addresses, p, &n) || n != (int)(sizeof lib / sizeof p[0])) {
        PyErr_SetString(PyExc_ValueError, "bind() takes a list of the entry points' addresses");
        return NULL;
    }
    memcpy(&lib, p, sizeof lib);
    Py_RETURN_NONE;
}

static PyMethodDef methods[] = {
    {"bind", bind, METH_O, NULL},
#define METHOD(f) {#f, (PyCFunction)(void (*)(void))f, METH_FASTCALL, NULL}
    METHOD(calibrate_ranges), METHOD(quantize_pack), METHOD(quantize_pack_batch), METHOD(dequant_reduce),
    METHOD(dequant_reduce_arrivals), METHOD(quantize_pack_push), METHOD(linear_quantize_pack),
    {NULL, NULL, 0, NULL}};

static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_calls", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__calls(void) { return PyModule_Create(&module); }
