/* The binding's calls on the hot path as CPython functions: tensor pointers, shapes and parameters are taken from the
 * Python objects here and passed to libmuxq's entry points (whose addresses binding.py hands over once).
 *
 * Why: at decode shapes a layer takes the GPU less time than ctypes and torch's stream lookup take the host.  Per
 * muxq_linear call, host side, 16 x 768 -> 768: 20 us with ctypes (3.5 us of it the lookup of the current stream, 4 us
 * argument conversion). */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>

#include "../../include/muxq.h"

typedef int (*linear_fn)(const void *, int, int, int, const int8_t *, int, const float *, int, const muxq_params *, void *,
                         int, int, void *, size_t, int32_t *, void *);
typedef int (*linear_bias_fn)(const void *, int, int, int, const int8_t *, int, const float *, const float *, int,
                              const muxq_params *, void *, int, int, void *, size_t, int32_t *, void *);
typedef int (*quantize_fn)(const void *, int, int, int, const muxq_params *, int, const float *, const int32_t *,
                           const int32_t *, int8_t *, int, int8_t *, int, float *, void *, size_t, void *);

static linear_fn f_linear;
static linear_bias_fn f_linear_bias;
static quantize_fn f_quantize;
static PyObject *get_device, *raw_stream, *dt_f16, *dt_f32;
static PyObject *n_data_ptr, *n_shape, *n_stride, *n_dtype, *n_is_cuda, *n_numel, *n_is_contiguous;
static PyObject *n_threshold, *n_exp_factor, *n_act_bits, *n_w_bits, *n_gran, *n_aux_scale, *n_max_outliers;

static int tensor_ptr(PyObject *t, void **out) {
    PyObject *v = PyObject_CallMethodNoArgs(t, n_data_ptr);
    if (!v) return -1;
    *out = PyLong_AsVoidPtr(v);
    Py_DECREF(v);
    return PyErr_Occurred() ? -1 : 0;
}

static int as_int(PyObject *v, int *out) { /* takes the reference */
    if (!v) return -1;
    const long x = PyLong_AsLong(v);
    Py_DECREF(v);
    if (x == -1 && PyErr_Occurred()) return -1;
    if (x < INT32_MIN || x > INT32_MAX) {
        PyErr_SetString(PyExc_OverflowError, "value does not fit a C int");
        return -1;
    }
    *out = (int)x;
    return 0;
}

/* the first two entries of a tensor's shape / stride (*b: 0 where there is only one); *dim: number of dimensions */
static int pair_of(PyObject *tuple, int *a, int *b, int *dim) { /* takes the reference */
    if (!tuple) return -1;
    int rc = 0;
    *a = *b = 0;
    *dim = PyTuple_Check(tuple) ? (int)PyTuple_GET_SIZE(tuple) : 0;
    if (*dim >= 1) rc = as_int(Py_NewRef(PyTuple_GET_ITEM(tuple, 0)), a);
    else rc = (PyErr_SetString(PyExc_IndexError, "a tensor with at least one dimension is wanted"), -1);
    if (!rc && *dim >= 2) rc = as_int(Py_NewRef(PyTuple_GET_ITEM(tuple, 1)), b);
    Py_DECREF(tuple);
    return rc;
}
static int shape_of(PyObject *t, int *a, int *b, int *dim) { return pair_of(PyObject_GetAttr(t, n_shape), a, b, dim); }
static int stride_of(PyObject *t, int *a, int *b) {
    int dim;
    return pair_of(PyObject_CallMethodNoArgs(t, n_stride), a, b, &dim);
}
static int is_true(PyObject *t, PyObject *name) { /* 1, 0 or -1 */
    PyObject *v = PyObject_GetAttr(t, name);
    if (!v) return -1;
    const int r = PyObject_IsTrue(v);
    Py_DECREF(v);
    return r;
}
static int has_dtype(PyObject *t, PyObject *dt) {
    PyObject *v = PyObject_GetAttr(t, n_dtype);
    if (!v) return -1;
    const int r = v == dt;
    Py_DECREF(v);
    return r;
}
static int numel_of(PyObject *t, Py_ssize_t *out) {
    PyObject *v = PyObject_CallMethodNoArgs(t, n_numel);
    if (!v) return -1;
    *out = PyLong_AsSsize_t(v);
    Py_DECREF(v);
    return *out == -1 && PyErr_Occurred() ? -1 : 0;
}

static int params_of(PyObject *p, muxq_params *c) {
    PyObject *v = PyObject_GetAttr(p, n_threshold);
    if (!v) return -1;
    c->threshold = (float)PyFloat_AsDouble(v);
    Py_DECREF(v);
    if (PyErr_Occurred()) return -1;
    return as_int(PyObject_GetAttr(p, n_exp_factor), &c->exp_factor) || as_int(PyObject_GetAttr(p, n_act_bits), &c->act_bits) ||
                   as_int(PyObject_GetAttr(p, n_w_bits), &c->w_bits) || as_int(PyObject_GetAttr(p, n_gran), &c->gran) ||
                   as_int(PyObject_GetAttr(p, n_aux_scale), &c->aux_scale) ||
                   as_int(PyObject_GetAttr(p, n_max_outliers), &c->max_outliers)
               ? -1
               : 0;
}

/* the stream that is current for the calling thread on the current device */
static int current_stream(void **out) {
    PyObject *dev = PyObject_CallNoArgs(get_device);
    if (!dev) return -1;
    PyObject *s = PyObject_CallOneArg(raw_stream, dev);
    Py_DECREF(dev);
    if (!s) return -1;
    *out = PyLong_AsVoidPtr(s);
    Py_DECREF(s);
    return PyErr_Occurred() ? -1 : 0;
}

static PyObject *stream(PyObject *self, PyObject *unused) {
    void *s;
    if (current_stream(&s)) return NULL;
    return PyLong_FromVoidPtr(s);
}

/* X [M, K] fp16 on the device with unit column stride, as the entry points want it */
static int matrix_f16(PyObject *t, void **ptr, int *rows, int *cols, int *ld) {
    int dim, cs = 0, ok = is_true(t, n_is_cuda);
    if (ok > 0) ok = has_dtype(t, dt_f16);
    if (ok < 0 || (ok && (shape_of(t, rows, cols, &dim) || stride_of(t, ld, &cs)))) return -1;
    if (!ok || dim != 2 || cs != 1) { /* (dim is set where ok) */
        PyErr_SetString(PyExc_AssertionError, "a 2-D fp16 CUDA tensor with unit column stride is wanted");
        return -1;
    }
    return tensor_ptr(t, ptr);
}

/* linear(X, w_q, s_w, params, workspace, status, out_kind, Y, bias or None) -> status code */
static PyObject *linear(PyObject *self, PyObject *const *a, Py_ssize_t n) {
    if (n != 9) return PyErr_Format(PyExc_TypeError, "linear takes 9 arguments");
    muxq_params p;
    void *x, *w, *sw, *ws, *st, *y, *bias = NULL, *s;
    int M, K, ldx, N, wk, dim, ldw, ldy, unused, out_kind;
    Py_ssize_t ws_bytes;
    if (matrix_f16(a[0], &x, &M, &K, &ldx) || shape_of(a[1], &N, &wk, &dim) || stride_of(a[1], &ldw, &unused) ||
        stride_of(a[7], &ldy, &unused) || params_of(a[3], &p) || as_int(Py_NewRef(a[6]), &out_kind))
        return NULL;
    if (a[8] != Py_None) {
        int ok = is_true(a[8], n_is_cuda);
        Py_ssize_t len = 0;
        if (ok > 0) ok = has_dtype(a[8], dt_f32);
        if (ok > 0) {
            PyObject *v = PyObject_CallMethodNoArgs(a[8], n_is_contiguous);
            ok = v ? PyObject_IsTrue(v) : -1;
            Py_XDECREF(v);
        }
        if (ok < 0 || numel_of(a[8], &len)) return NULL;
        if (!ok || len != N) {
            PyErr_SetString(PyExc_AssertionError, "the bias is a contiguous fp32 CUDA tensor of N entries");
            return NULL;
        }
        if (tensor_ptr(a[8], &bias)) return NULL;
    }
    if (tensor_ptr(a[1], &w) || tensor_ptr(a[2], &sw) || tensor_ptr(a[4], &ws) || numel_of(a[4], &ws_bytes) ||
        tensor_ptr(a[5], &st) || tensor_ptr(a[7], &y) || current_stream(&s))
        return NULL;
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = a[8] != Py_None ? f_linear_bias(x, M, K, ldx, w, ldw, sw, bias, N, &p, y, ldy, out_kind, ws, (size_t)ws_bytes, st, s)
                         : f_linear(x, M, K, ldx, w, ldw, sw, N, &p, y, ldy, out_kind, ws, (size_t)ws_bytes, st, s);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

/* quantize_weight(W, params, W_q, scales, workspace) -> status code */
static PyObject *quantize_weight(PyObject *self, PyObject *const *a, Py_ssize_t n) {
    if (n != 5) return PyErr_Format(PyExc_TypeError, "quantize_weight takes 5 arguments");
    muxq_params p;
    void *w, *q, *sc, *ws, *s;
    int K, N, ld;
    Py_ssize_t ws_bytes;
    if (matrix_f16(a[0], &w, &K, &N, &ld) || params_of(a[1], &p) || tensor_ptr(a[2], &q) || tensor_ptr(a[3], &sc) ||
        tensor_ptr(a[4], &ws) || numel_of(a[4], &ws_bytes) || current_stream(&s))
        return NULL;
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = f_quantize(w, K, N, ld, &p, 1, NULL, NULL, NULL, q, K, NULL, 0, sc, ws, (size_t)ws_bytes, s);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

/* bind(muxq_linear, muxq_linear_bias, muxq_quantize, get_device, raw_stream, float16, float32) */
static PyObject *bind(PyObject *self, PyObject *const *a, Py_ssize_t n) {
    if (n != 7) return PyErr_Format(PyExc_TypeError, "bind takes 7 arguments");
    f_linear = (linear_fn)PyLong_AsVoidPtr(a[0]);
    f_linear_bias = (linear_bias_fn)PyLong_AsVoidPtr(a[1]);
    f_quantize = (quantize_fn)PyLong_AsVoidPtr(a[2]);
    if (PyErr_Occurred()) return NULL;
    Py_XSETREF(get_device, Py_NewRef(a[3]));
    Py_XSETREF(raw_stream, Py_NewRef(a[4]));
    Py_XSETREF(dt_f16, Py_NewRef(a[5]));
    Py_XSETREF(dt_f32, Py_NewRef(a[6]));
    Py_RETURN_NONE;
}

static PyMethodDef methods[] = {
    {"bind", (PyCFunction)(void (*)(void))bind, METH_FASTCALL, "addresses of the entry points, torch's stream lookup and dtypes"},
    {"linear", (PyCFunction)(void (*)(void))linear, METH_FASTCALL, "muxq_linear / muxq_linear_bias"},
    {"quantize_weight", (PyCFunction)(void (*)(void))quantize_weight, METH_FASTCALL, "muxq_quantize(is_weight = 1)"},
    {"stream", stream, METH_NOARGS, "handle of the current stream"},
    {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_calls", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__calls(void) {
    struct { PyObject **to; const char *name; } names[] = {
        {&n_data_ptr, "data_ptr"}, {&n_shape, "shape"}, {&n_stride, "stride"}, {&n_dtype, "dtype"}, {&n_is_cuda, "is_cuda"},
        {&n_numel, "numel"}, {&n_is_contiguous, "is_contiguous"}, {&n_threshold, "threshold"}, {&n_exp_factor, "exp_factor"}, {&n_act_bits, "act_bits"},
        {&n_w_bits, "w_bits"}, {&n_gran, "gran"}, {&n_aux_scale, "aux_scale"}, {&n_max_outliers, "max_outliers"}};
    for (size_t i = 0; i < sizeof names / sizeof *names; ++i)
        if (!*names[i].to && !(*names[i].to = PyUnicode_InternFromString(names[i].name))) return NULL;
    return PyModule_Create(&module);
}
