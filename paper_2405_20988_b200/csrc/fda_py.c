/*
 * CPython module _native: the calls of a monitoring step from Python to libfda.
 *
 * Bound: host time.  On small models the kernels of a step take less than the Python that launches
 * them: marshalling one call in Python (tensor attributes, ctypes conversions, the current stream)
 * took 5-7 us, this module takes about 1.  It checks what the Python wrappers checked, passes
 * data pointers and the stream through and returns the status; it computes nothing.
 */
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include "../../include/fda.h"

static PyObject *s_is_cuda, *s_dtype, *s_data_ptr, *s_shape, *s_stride, *s_cuda_stream, *s_get_device,
    *s_is_contiguous;
static PyObject *g_float32, *g_uint8, *g_raw_stream, *g_get_device;

/* init(torch.float32, torch.uint8, raw stream of a device, current device) */
static PyObject *py_init(PyObject *self, PyObject *const *args, Py_ssize_t n)
{
    if (n != 4) { PyErr_SetString(PyExc_TypeError, "init takes 4 arguments"); return NULL; }
    PyObject **slot[4] = {&g_float32, &g_uint8, &g_raw_stream, &g_get_device};
    for (int i = 0; i < 4; ++i) { Py_INCREF(args[i]); Py_XSETREF(*slot[i], args[i]); }
    Py_RETURN_NONE;
}

static int as_i64(PyObject *o, int64_t *out)
{
    *out = (int64_t)PyLong_AsLongLong(o);
    return *out == -1 && PyErr_Occurred() ? -1 : 0;
}
static int call_i64(PyObject *t, PyObject *method, int64_t *out)
{
    PyObject *r = PyObject_CallMethodNoArgs(t, method);
    if (!r) return -1;
    const int st = as_i64(r, out);
    Py_DECREF(r);
    return st;
}
static int call_ptr(PyObject *t, PyObject *method, void **out)
{
    PyObject *r = PyObject_CallMethodNoArgs(t, method);
    if (!r) return -1;
    *out = PyLong_AsVoidPtr(r);
    Py_DECREF(r);
    return *out == NULL && PyErr_Occurred() ? -1 : 0;
}

/* device pointer of a CUDA tensor of the given type (None: NULL) */
static int dev_ptr(PyObject *t, PyObject *dtype, const char *name, void **out)
{
    *out = NULL;
    if (t == Py_None) return 0;
    PyObject *v = PyObject_GetAttr(t, s_is_cuda);
    if (!v) return -1;
    const int cuda = PyObject_IsTrue(v);
    Py_DECREF(v);
    if (cuda < 0) return -1;
    if (!cuda) { PyErr_Format(PyExc_ValueError, "%s must be a CUDA tensor", name); return -1; }
    v = PyObject_GetAttr(t, s_dtype);
    if (!v) return -1;
    const int same = v == dtype;
    Py_DECREF(v);
    if (!same) { PyErr_Format(PyExc_ValueError, "%s must have dtype %S", name, dtype); return -1; }
    return call_ptr(t, s_data_ptr, out);
}

/* pointer, pitch, rows and columns of a 2-D float32 tensor whose rows are contiguous */
static int rows_of(PyObject *w, void **ptr, int64_t *pitch, int64_t *K, int64_t *d)
{
    PyObject *shape = PyObject_GetAttr(w, s_shape), *stride = NULL;
    int ok = 0;
    if (!shape) return -1;
    stride = PyObject_CallMethodNoArgs(w, s_stride);
    if (stride && PyTuple_Check(shape) && PyTuple_Check(stride) && PyTuple_GET_SIZE(shape) == 2 &&
        PyTuple_GET_SIZE(stride) == 2) {
        int64_t s0 = 0, s1 = 0;
        ok = as_i64(PyTuple_GET_ITEM(shape, 0), K) == 0 && as_i64(PyTuple_GET_ITEM(shape, 1), d) == 0 &&
             as_i64(PyTuple_GET_ITEM(stride, 0), &s0) == 0 && as_i64(PyTuple_GET_ITEM(stride, 1), &s1) == 0 &&
             (*d <= 1 || s1 == 1);
        *pitch = *K > 1 || s0 > *d ? s0 : *d;
    }
    Py_DECREF(shape);
    Py_XDECREF(stride);
    if (!ok) {
        if (!PyErr_Occurred()) PyErr_SetString(PyExc_ValueError, "w must be 2-D with contiguous rows");
        return -1;
    }
    return dev_ptr(w, g_float32, "w", ptr);
}

/* cudaStream_t of a torch stream, or of the current one (None) */
static int stream_ptr(PyObject *stream, void **out)
{
    PyObject *r;
    if (stream == Py_None) {
        PyObject *dev = PyObject_CallNoArgs(g_get_device);
        if (!dev) return -1;
        r = PyObject_CallOneArg(g_raw_stream, dev);
        Py_DECREF(dev);
    } else {
        r = PyObject_GetAttr(stream, s_cuda_stream);
    }
    if (!r) return -1;
    *out = PyLong_AsVoidPtr(r);
    Py_DECREF(r);
    return *out == NULL && PyErr_Occurred() ? -1 : 0;
}

static int handle_of(PyObject *o, fda_ctx **ctx)
{
    *ctx = NULL;
    if (o == Py_None) return 0;
    *ctx = (fda_ctx *)PyLong_AsVoidPtr(o);
    return *ctx == NULL && PyErr_Occurred() ? -1 : 0;
}
static int expect(Py_ssize_t n, Py_ssize_t want)
{
    if (n == want) return 0;
    PyErr_Format(PyExc_TypeError, "%zd arguments expected, %zd given", want, n);
    return -1;
}

typedef fda_status (*state_fn)(fda_ctx *, const float *, int64_t, int, int64_t, const float *, const float *, uint32_t,
                               float *, void *);

/* (handle, w, w_t0, xi, flags, states, stream) */
static PyObject *state_call(PyObject *const *a, Py_ssize_t n, state_fn fn, const char *out_name)
{
    fda_ctx *ctx;
    void *w, *w0, *xi, *out, *stream;
    int64_t pitch, K, d;
    if (expect(n, 7) || handle_of(a[0], &ctx) || rows_of(a[1], &w, &pitch, &K, &d) || dev_ptr(a[2], g_float32, "w_t0", &w0) ||
        dev_ptr(a[3], g_float32, "xi", &xi) || dev_ptr(a[5], g_float32, out_name, &out) || stream_ptr(a[6], &stream))
        return NULL;
    const uint32_t flags = (uint32_t)PyLong_AsUnsignedLongMask(a[4]);
    if (PyErr_Occurred()) return NULL;
    fda_status st;
    Py_BEGIN_ALLOW_THREADS
    st = fn(ctx, w, pitch, (int)K, d, w0, xi, flags, out, stream);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong((long)st);
}
static PyObject *py_local_state(PyObject *self, PyObject *const *a, Py_ssize_t n) { return state_call(a, n, fda_local_state, "states"); }
static PyObject *py_mean_state(PyObject *self, PyObject *const *a, Py_ssize_t n) { return state_call(a, n, fda_mean_state, "mean_state"); }

/* (handle, states, K, variant, epsilon, theta, est_dev, address of a host fda_estimate or 0, stream) */
static PyObject *py_combine_estimate(PyObject *self, PyObject *const *a, Py_ssize_t n)
{
    fda_ctx *ctx;
    void *states, *est, *stream;
    if (expect(n, 9) || handle_of(a[0], &ctx) || dev_ptr(a[1], g_float32, "states", &states) ||
        dev_ptr(a[6], g_uint8, "est_dev", &est) || stream_ptr(a[8], &stream))
        return NULL;
    const int K = (int)PyLong_AsLong(a[2]), variant = (int)PyLong_AsLong(a[3]);
    if (PyErr_Occurred()) return NULL;
    const float epsilon = (float)PyFloat_AsDouble(a[4]), theta = (float)PyFloat_AsDouble(a[5]);
    void *host = PyLong_AsVoidPtr(a[7]);
    if (PyErr_Occurred()) return NULL;
    fda_status st;
    Py_BEGIN_ALLOW_THREADS
    st = fda_combine_estimate(ctx, states, K, variant, epsilon, theta, est, host, stream);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong((long)st);
}

/* (handle, w, w_t0, est_dev, flags, stream) */
static PyObject *py_average_models(PyObject *self, PyObject *const *a, Py_ssize_t n)
{
    fda_ctx *ctx;
    void *w, *w0, *est, *stream;
    int64_t pitch, K, d;
    if (expect(n, 6) || handle_of(a[0], &ctx) || rows_of(a[1], &w, &pitch, &K, &d) || dev_ptr(a[2], g_float32, "w_t0", &w0) ||
        dev_ptr(a[3], g_uint8, "est_dev", &est) || stream_ptr(a[5], &stream))
        return NULL;
    const uint32_t flags = (uint32_t)PyLong_AsUnsignedLongMask(a[4]);
    if (PyErr_Occurred()) return NULL;
    fda_status st;
    Py_BEGIN_ALLOW_THREADS
    st = fda_average_models(ctx, w, pitch, (int)K, d, w0, est, flags, stream);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong((long)st);
}

/* (handle, w, w_t0, xi_out, est_dev, flags, stream) */
static PyObject *py_average_models_xi(PyObject *self, PyObject *const *a, Py_ssize_t n)
{
    fda_ctx *ctx;
    void *w, *w0, *xi, *est, *stream;
    int64_t pitch, K, d;
    if (expect(n, 7) || handle_of(a[0], &ctx) || rows_of(a[1], &w, &pitch, &K, &d) || dev_ptr(a[2], g_float32, "w_t0", &w0) ||
        dev_ptr(a[3], g_float32, "xi_out", &xi) || dev_ptr(a[4], g_uint8, "est_dev", &est) || stream_ptr(a[6], &stream))
        return NULL;
    const uint32_t flags = (uint32_t)PyLong_AsUnsignedLongMask(a[5]);
    if (PyErr_Occurred()) return NULL;
    fda_status st;
    Py_BEGIN_ALLOW_THREADS
    st = fda_average_models_xi(ctx, w, pitch, (int)K, d, w0, xi, est, flags, stream);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong((long)st);
}

/* (w, w_t0, xi, flags, states, stream) */
static PyObject *py_local_state_linear_noalloc(PyObject *self, PyObject *const *a, Py_ssize_t n)
{
    void *w, *w0, *xi, *out, *stream;
    int64_t pitch, K, d, device, rows = 0, cols = 0;
    if (expect(n, 6) || rows_of(a[0], &w, &pitch, &K, &d)) return NULL;
    PyObject *shape = PyObject_GetAttr(a[4], s_shape);
    if (!shape) return NULL;
    if (PyTuple_Check(shape) && PyTuple_GET_SIZE(shape) == 2 &&
        (as_i64(PyTuple_GET_ITEM(shape, 0), &rows) || as_i64(PyTuple_GET_ITEM(shape, 1), &cols))) {
        Py_DECREF(shape);
        return NULL;
    }
    Py_DECREF(shape);
    PyObject *c = PyObject_CallMethodNoArgs(a[4], s_is_contiguous);
    if (!c) return NULL;
    const int contiguous = PyObject_IsTrue(c);
    Py_DECREF(c);
    if (rows != K || cols != 2 || contiguous != 1) {
        PyErr_SetString(PyExc_ValueError, "states must be a contiguous K x 2 tensor");
        return NULL;
    }
    if (call_i64(a[0], s_get_device, &device) || dev_ptr(a[1], g_float32, "w_t0", &w0) ||
        dev_ptr(a[2], g_float32, "xi", &xi) || dev_ptr(a[4], g_float32, "states", &out) || stream_ptr(a[5], &stream))
        return NULL;
    const uint32_t flags = (uint32_t)PyLong_AsUnsignedLongMask(a[3]);
    if (PyErr_Occurred()) return NULL;
    fda_status st;
    Py_BEGIN_ALLOW_THREADS
    st = fda_local_state_linear_noalloc((int)device, w, pitch, (int)K, d, w0, xi, flags, out, stream);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong((long)st);
}

#define FAST(name) {#name, (PyCFunction)(void (*)(void))py_##name, METH_FASTCALL, NULL}
static PyMethodDef methods[] = {FAST(init), FAST(local_state), FAST(mean_state), FAST(combine_estimate),
                                FAST(average_models), FAST(average_models_xi), FAST(local_state_linear_noalloc),
                                {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__native(void)
{
    struct { PyObject **slot; const char *text; } names[] = {
        {&s_is_cuda, "is_cuda"}, {&s_dtype, "dtype"}, {&s_data_ptr, "data_ptr"}, {&s_shape, "shape"},
        {&s_stride, "stride"}, {&s_cuda_stream, "cuda_stream"}, {&s_get_device, "get_device"},
        {&s_is_contiguous, "is_contiguous"}};
    for (size_t i = 0; i < sizeof(names) / sizeof(names[0]); ++i)
        if (!(*names[i].slot = PyUnicode_InternFromString(names[i].text))) return NULL;
    return PyModule_Create(&module);
}
