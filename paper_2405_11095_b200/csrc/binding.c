/* Native half of the Python binding: turns torch tensors and numbers into the arguments of the C-ABI.
 *
 * A call on a short vector is bound by the host, and of the 8 us that an encode of 2^16 coordinates took there (two
 * launches of 2.3 us each) 3.3 us were Python and ctypes marshalling; here the same conversions take about 1 us.
 * Nothing is computed: every function reads tensor attributes, calls the library function of the same name with
 * the GIL released, and returns its status.  The library is the one that the package has loaded: bind() receives the
 * functions' addresses. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <stdint.h>

#include "../../include/fosgd.h"

enum { FN_ENCODE, FN_FLATTEN, FN_DECODE, FN_AGGREGATE, FN_DOWN_DECODE, FN_AMPLITUDES, FN_ENCODE_DEV, FN_AGGREGATE_DEV,
       FN_DOWN_DECODE_DEV, FN_DOWN_ENCODE, FN_DOWN_APPLY, FN_ENCODE_MEASURED, FN_ENCODE_MEASURED_BLOCKS, FN_COUNT };

static void* g_fn[FN_COUNT];
static PyObject *g_get_device, *g_get_stream, *g_float32, *g_bfloat16;
static PyObject *s_data_ptr, *s_numel, *s_element_size, *s_dim, *s_size, *s_stride, *s_dtype, *g_zero;

/* One call's conversions; `bad` is set (and a Python exception pending) as soon as one of them failed. */
typedef struct { PyObject* const* a; int bad; } Args;

static int64_t as_int(Args* c, PyObject* o)
{
    if (c->bad) return 0;
    const uint64_t v = (uint64_t)PyLong_AsUnsignedLongLongMask(o);   /* wraps, as the C types do */
    if (v == (uint64_t)-1 && PyErr_Occurred()) c->bad = 1;
    return (int64_t)v;
}

static double as_double(Args* c, PyObject* o)
{
    if (c->bad) return 0.0;
    const double v = PyFloat_AsDouble(o);
    if (v == -1.0 && PyErr_Occurred()) c->bad = 1;
    return v;
}

/* an int returned by a call that may have failed; steals the reference */
static int64_t taken(Args* c, PyObject* r)
{
    if (r == NULL) { c->bad = 1; return 0; }
    const int64_t v = as_int(c, r);
    Py_DECREF(r);
    return v;
}

/* whatever int(o) and float(o) take: numpy's truth values for a switch, say */
static int64_t made_int(Args* c, PyObject* o) { return c->bad ? 0 : PyLong_Check(o) ? as_int(c, o) : taken(c, PyNumber_Long(o)); }
static double made_double(Args* c, PyObject* o)
{
    if (c->bad) return 0.0;
    PyObject* const r = PyNumber_Float(o);
    if (r == NULL) { c->bad = 1; return 0.0; }
    const double v = PyFloat_AS_DOUBLE(r);
    Py_DECREF(r);
    return v;
}

static int64_t method0(Args* c, PyObject* t, PyObject* name) { return c->bad ? 0 : taken(c, PyObject_CallMethodNoArgs(t, name)); }
static int64_t method_of_0(Args* c, PyObject* t, PyObject* name) { return c->bad ? 0 : taken(c, PyObject_CallMethodOneArg(t, name, g_zero)); }

static void* ptr(Args* c, PyObject* t) { return t == Py_None ? NULL : (void*)(uintptr_t)method0(c, t, s_data_ptr); }

static size_t nbytes(Args* c, PyObject* t)
{
    return t == Py_None ? 0 : (size_t)method0(c, t, s_numel) * (size_t)method0(c, t, s_element_size);
}

static fosgd_stream stream(Args* c)
{
    if (c->bad) return NULL;
    PyObject* const dev = PyObject_CallNoArgs(g_get_device);
    if (dev == NULL) { c->bad = 1; return NULL; }
    PyObject* const r = PyObject_CallOneArg(g_get_stream, dev);
    Py_DECREF(dev);
    return (fosgd_stream)(uintptr_t)taken(c, r);
}

static int rows(Args* c, PyObject* t) { return method0(c, t, s_dim) == 2 ? (int)method_of_0(c, t, s_size) : 1; }

/* gradients: pointer, type, worker count, stride between rows in elements (an int, or None: the tensor's own) */
typedef struct { const void* p; int dtype, M; int64_t stride; } Grads;

static Grads grads(Args* c, PyObject* t, PyObject* stride, int64_t d)
{
    Grads g = {NULL, -1, 1, d};
    g.M = rows(c, t);
    if (stride != Py_None) g.stride = as_int(c, stride);
    else if (!c->bad && method0(c, t, s_dim) == 2) g.stride = method_of_0(c, t, s_stride);
    g.p = ptr(c, t);
    if (c->bad) return g;
    PyObject* const dt = PyObject_GetAttr(t, s_dtype);
    if (dt == NULL) { c->bad = 1; return g; }
    g.dtype = dt == g_float32 ? FOSGD_F32 : dt == g_bfloat16 ? FOSGD_BF16 : -1;
    Py_DECREF(dt);
    return g;
}

/* an amplitude given as a number, or as a device tensor */
static const float* device_amplitude(Args* c, PyObject* o, float* value)
{
    *value = 0.f;
    if (PyFloat_Check(o) || PyLong_Check(o)) { *value = (float)as_double(c, o); return NULL; }
    return (const float*)ptr(c, o);
}

#define ENTER(COUNT)                                                                                    \
    if (n != (COUNT)) { PyErr_SetString(PyExc_TypeError, "wrong number of arguments"); return NULL; }   \
    Args ctx = {a, 0}, *const c = &ctx;                                                                 \
    int st;
#define I32(K) ((int)as_int(c, a[K]))
#define U32(K) ((uint32_t)as_int(c, a[K]))
#define I64(K) (as_int(c, a[K]))
#define U64(K) ((uint64_t)as_int(c, a[K]))
#define F32(K) ((float)as_double(c, a[K]))
#define F64(K) (as_double(c, a[K]))
#define SWITCH(K) ((int)made_int(c, a[K]))
#define PTR(K) (ptr(c, a[K]))
#define CALL(EXPR)                       \
    if (c->bad) return NULL;             \
    Py_BEGIN_ALLOW_THREADS st = (EXPR);  \
    Py_END_ALLOW_THREADS return PyLong_FromLong(st);
#define FN(K, NAME) ((__typeof__(&NAME))g_fn[K])
#define CALLABLE(NAME) static PyObject* NAME(PyObject* self, PyObject* const* a, Py_ssize_t n)

/* grads d bits lam seed step worker_id0 block_log2 ws worker_stride */
CALLABLE(encode)
{
    ENTER(10)
    const int64_t d = I64(1);
    const Grads g = grads(c, a[0], a[9], d);
    uint32_t* const bits = PTR(2);
    const float lam = F32(3);
    const uint64_t seed = U64(4), step = U64(5);
    const uint32_t id0 = U32(6);
    const int b = I32(7);
    void* const ws = PTR(8);
    const size_t wsn = nbytes(c, a[8]);
    const fosgd_stream s = stream(c);
    CALL(FN(FN_ENCODE, fosgd_encode)(g.p, g.dtype, d, g.stride, g.M, id0, seed, step, lam, b, bits, ws, wsn, s))
}

/* grads d out seed step worker_id0 block_log2 ws worker_stride */
CALLABLE(flatten)
{
    ENTER(9)
    const int64_t d = I64(1);
    const Grads g = grads(c, a[0], a[8], d);
    float* const out = PTR(2);
    const uint64_t seed = U64(3), step = U64(4);
    const uint32_t id0 = U32(5);
    const int b = I32(6);
    void* const ws = PTR(7);
    const size_t wsn = nbytes(c, a[7]);
    const fosgd_stream s = stream(c);
    CALL(FN(FN_FLATTEN, fosgd_flatten)(g.p, g.dtype, d, g.stride, g.M, id0, seed, step, b, out, ws, wsn, s))
}

/* bits d out lam seed step worker_id block_log2 ws */
CALLABLE(decode)
{
    ENTER(9)
    const uint32_t* const bits = PTR(0);
    const int64_t d = I64(1);
    float* const out = PTR(2);
    const float lam = F32(3);
    const uint64_t seed = U64(4), step = U64(5);
    const uint32_t id = U32(6);
    const int b = I32(7);
    void* const ws = PTR(8);
    const size_t wsn = nbytes(c, a[8]);
    const fosgd_stream s = stream(c);
    CALL(FN(FN_DECODE, fosgd_decode)(bits, d, id, seed, step, lam, b, out, ws, wsn, s))
}

/* bits d acc lam seed step N_total worker_id0 flags lam_s K down_bits block_log2 ws */
CALLABLE(server_aggregate)
{
    ENTER(14)
    const uint32_t* const bits = PTR(0);
    const int M = rows(c, a[0]);
    const int64_t d = I64(1);
    float* const acc = PTR(2);
    const float lam = F32(3);
    const uint64_t seed = U64(4), step = U64(5);
    const int total = a[6] == Py_None ? M : I32(6);
    const uint32_t id0 = U32(7);
    const int flags = I32(8);
    const float lam_s = F32(9);
    const int K = I32(10);
    uint32_t* const down = PTR(11);
    const int b = I32(12);
    void* const ws = PTR(13);
    const size_t wsn = nbytes(c, a[13]);
    const fosgd_stream s = stream(c);
    CALL(FN(FN_AGGREGATE, fosgd_server_aggregate)(bits, d, M, id0, total, seed, step, lam, b, acc, flags, lam_s, K, down, ws, wsn, s))
}

/* bits d acc lam seed step N_total worker_id0 flags lam_s K down_bits block_log2 per_block ws */
CALLABLE(server_aggregate_dev)
{
    ENTER(15)
    const uint32_t* const bits = PTR(0);
    const int M = rows(c, a[0]);
    const int64_t d = I64(1);
    float* const acc = PTR(2);
    const float* const lam = PTR(3);
    const uint64_t seed = U64(4), step = U64(5);
    const int total = a[6] == Py_None ? M : I32(6);
    const uint32_t id0 = U32(7);
    const int flags = I32(8);
    const float* const lam_s = PTR(9);
    const int K = I32(10);
    uint32_t* const down = PTR(11);
    const int b = I32(12), pb = SWITCH(13);
    void* const ws = PTR(14);
    const size_t wsn = nbytes(c, a[14]);
    const fosgd_stream s = stream(c);
    CALL(FN(FN_AGGREGATE_DEV, fosgd_server_aggregate_dev)(bits, d, M, id0, total, seed, step, lam, lam_s, pb, b, acc, flags, K, down, ws, wsn, s))
}

/* down_bits d out lam_s seed step K block_log2 ws */
CALLABLE(downlink_decode)
{
    ENTER(9)
    const uint32_t* const down = PTR(0);
    const int64_t d = I64(1);
    float* const out = PTR(2);
    const float lam_s = F32(3);
    const uint64_t seed = U64(4), step = U64(5);
    const int K = I32(6), b = I32(7);
    void* const ws = PTR(8);
    const size_t wsn = nbytes(c, a[8]);
    const fosgd_stream s = stream(c);
    CALL(FN(FN_DOWN_DECODE, fosgd_downlink_decode)(down, d, seed, step, lam_s, K, b, out, ws, wsn, s))
}

/* down_bits d out lam_s seed step K block_log2 per_block ws */
CALLABLE(downlink_decode_dev)
{
    ENTER(10)
    const uint32_t* const down = PTR(0);
    const int64_t d = I64(1);
    float* const out = PTR(2);
    const float* const lam_s = PTR(3);
    const uint64_t seed = U64(4), step = U64(5);
    const int K = I32(6), b = I32(7), pb = SWITCH(8);
    void* const ws = PTR(9);
    const size_t wsn = nbytes(c, a[9]);
    const fosgd_stream s = stream(c);
    CALL(FN(FN_DOWN_DECODE_DEV, fosgd_downlink_decode_dev)(down, d, seed, step, lam_s, pb, K, b, out, ws, wsn, s))
}

/* gbar d down_bits lam_s seed step K block_log2 per_block ws */
CALLABLE(downlink_encode)
{
    ENTER(10)
    const float* const gbar = PTR(0);
    const int64_t d = I64(1);
    uint32_t* const down = PTR(2);
    float value;
    const float* const dev = device_amplitude(c, a[3], &value);
    const uint64_t seed = U64(4), step = U64(5);
    const int K = I32(6), b = I32(7), pb = SWITCH(8);
    void* const ws = PTR(9);
    const size_t wsn = nbytes(c, a[9]);
    const fosgd_stream s = stream(c);
    CALL(FN(FN_DOWN_ENCODE, fosgd_downlink_encode)(gbar, d, seed, step, value, dev, pb, K, b, down, ws, wsn, s))
}

/* down_bits d x lam_s seed step step_size K block_log2 per_block ws */
CALLABLE(downlink_apply)
{
    ENTER(11)
    const uint32_t* const down = PTR(0);
    const int64_t d = I64(1);
    float* const x = PTR(2);
    float value;
    const float* const dev = device_amplitude(c, a[3], &value);
    const uint64_t seed = U64(4), step = U64(5);
    const float step_size = (float)made_double(c, a[6]);
    const int K = I32(7), b = I32(8), pb = SWITCH(9);
    void* const ws = PTR(10);
    const size_t wsn = nbytes(c, a[10]);
    const fosgd_stream s = stream(c);
    CALL(FN(FN_DOWN_APPLY, fosgd_downlink_apply)(down, d, seed, step, value, dev, pb, K, b, step_size, x, ws, wsn, s))
}

/* grads d lam lam_s alpha alpha_s block_log2 per_block ws worker_stride */
CALLABLE(amplitudes)
{
    ENTER(10)
    const int64_t d = I64(1);
    const Grads g = grads(c, a[0], a[9], d);
    float* const lam = PTR(2);
    float* const lam_s = PTR(3);
    const double alpha = F64(4), alpha_s = F64(5);
    const int b = I32(6), pb = SWITCH(7);
    void* const ws = PTR(8);
    const size_t wsn = nbytes(c, a[8]);
    const fosgd_stream s = stream(c);
    CALL(FN(FN_AMPLITUDES, fosgd_amplitudes)(g.p, g.dtype, d, g.stride, g.M, alpha, alpha_s, b, pb, lam, lam_s, ws, wsn, s))
}

/* grads d bits lam seed step worker_id0 block_log2 per_block ws worker_stride */
CALLABLE(encode_dev)
{
    ENTER(11)
    const int64_t d = I64(1);
    const Grads g = grads(c, a[0], a[10], d);
    uint32_t* const bits = PTR(2);
    const float* const lam = PTR(3);
    const uint64_t seed = U64(4), step = U64(5);
    const uint32_t id0 = U32(6);
    const int b = I32(7), pb = SWITCH(8);
    void* const ws = PTR(9);
    const size_t wsn = nbytes(c, a[9]);
    const fosgd_stream s = stream(c);
    CALL(FN(FN_ENCODE_DEV, fosgd_encode_dev)(g.p, g.dtype, d, g.stride, g.M, id0, seed, step, lam, pb, b, bits, ws, wsn, s))
}

/* grads d bits lam lam_s seed step alpha alpha_s worker_id0 block_log2 ws amp_ws worker_stride */
static PyObject* measured(PyObject* const* a, Py_ssize_t n, int fn)
{
    ENTER(14)
    const int64_t d = I64(1);
    const Grads g = grads(c, a[0], a[13], d);
    uint32_t* const bits = PTR(2);
    float* const lam = PTR(3);
    float* const lam_s = PTR(4);
    const uint64_t seed = U64(5), step = U64(6);
    const double alpha = F64(7), alpha_s = F64(8);
    const uint32_t id0 = U32(9);
    const int b = I32(10);
    void* const ws = PTR(11);
    const size_t wsn = nbytes(c, a[11]);
    void* const aws = PTR(12);
    const size_t awsn = nbytes(c, a[12]);
    const fosgd_stream s = stream(c);
    CALL(FN(fn, fosgd_encode_measured)(g.p, g.dtype, d, g.stride, g.M, id0, seed, step, alpha, alpha_s, b, lam, lam_s, bits, ws, wsn, aws, awsn, s))
}

CALLABLE(encode_measured) { return measured(a, n, FN_ENCODE_MEASURED); }
CALLABLE(encode_measured_blocks) { return measured(a, n, FN_ENCODE_MEASURED_BLOCKS); }

/* addresses (a tuple in the order of FN_*), current-device function, current-stream function, float32, bfloat16 */
CALLABLE(bind)
{
    if (n != 5 || !PyTuple_Check(a[0]) || PyTuple_GET_SIZE(a[0]) != FN_COUNT) {
        PyErr_SetString(PyExc_TypeError, "bind(addresses, get_device, get_stream, float32, bfloat16)");
        return NULL;
    }
    for (int k = 0; k < FN_COUNT; ++k) {
        void* const f = PyLong_AsVoidPtr(PyTuple_GET_ITEM(a[0], k));
        if (f == NULL) {
            if (!PyErr_Occurred()) PyErr_SetString(PyExc_ValueError, "null function address");
            return NULL;
        }
        g_fn[k] = f;
    }
    PyObject** const kept[4] = {&g_get_device, &g_get_stream, &g_float32, &g_bfloat16};
    for (int k = 0; k < 4; ++k) {
        Py_INCREF(a[k + 1]);
        Py_XSETREF(*kept[k], a[k + 1]);
    }
    Py_RETURN_NONE;
}

#define METHOD(NAME) {#NAME, (PyCFunction)(void (*)(void))NAME, METH_FASTCALL, NULL}
static PyMethodDef methods[] = {METHOD(bind), METHOD(encode), METHOD(flatten), METHOD(decode), METHOD(server_aggregate),
                                METHOD(server_aggregate_dev), METHOD(downlink_decode), METHOD(downlink_decode_dev),
                                METHOD(downlink_encode), METHOD(downlink_apply), METHOD(amplitudes), METHOD(encode_dev),
                                METHOD(encode_measured), METHOD(encode_measured_blocks), {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__native(void)
{
    s_data_ptr = PyUnicode_InternFromString("data_ptr");
    s_numel = PyUnicode_InternFromString("numel");
    s_element_size = PyUnicode_InternFromString("element_size");
    s_dim = PyUnicode_InternFromString("dim");
    s_size = PyUnicode_InternFromString("size");
    s_stride = PyUnicode_InternFromString("stride");
    s_dtype = PyUnicode_InternFromString("dtype");
    g_zero = PyLong_FromLong(0);
    if (!s_data_ptr || !s_numel || !s_element_size || !s_dim || !s_size || !s_stride || !s_dtype || !g_zero) return NULL;
    return PyModule_Create(&module);
}
