/* The fused layer calls of binding.py as native functions: a small layer's kernels are shorter than its marshalling through ctypes
 * (4.8 us on the host for the 19 arguments of a linear; 1.7 here).  The functions take what the Python ones take, ask a
 * tensor for its address, shape, pitch and type through its Python attributes, and call the C entry points, whose addresses
 * binding.py hands over (bind): nothing is linked against either library, and the GIL is released during the call. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>

#include "../../include/hq.h"

typedef hq_status (*qlinear_fn)(const void*, hq_dtype, int64_t, int64_t, int64_t, const hq_weight_desc*, const void*, const float*,
                                const float*, int, hq_scale_mode, const float*, void*, hq_dtype, int64_t, void*, size_t, int32_t*, void*);
typedef hq_status (*qconv_fn)(const void*, hq_dtype, int64_t, int64_t, int64_t, int64_t, const hq_weight_desc*, const void*, int, int, int,
                              int, const float*, const float*, int, hq_scale_mode, const float*, void*, hq_dtype, void*, size_t, int32_t*,
                              void*);
typedef hq_status (*ln_qlinear_fn)(const void*, hq_dtype, int64_t, int64_t, int64_t, const float*, const float*, int64_t, float,
                                   const hq_weight_desc*, const void*, const float*, const float*, int, void*, hq_dtype, int64_t, void*,
                                   size_t, int32_t*, void*);
typedef hq_status (*quant_fn)(const void*, hq_dtype, int64_t, int64_t, int64_t, int, int, hq_scale_mode, const float*, void*, hq_container,
                              int64_t, float*, void*);
static qlinear_fn f_qlinear;
static qconv_fn f_qconv;
static ln_qlinear_fn f_ln_qlinear;
static quant_fn f_quant;

static PyObject *s_data_ptr, *s_shape, *s_stride, *s_dtype, *s_nbytes, *s_desc, *s_blob_dev, *s_s_w_dev, *zero;
static PyObject* dtype_code;              /* binding.py's function, asked once per type */
static PyObject* known_dtype[2];
static int known_code[2];

static int address(PyObject* t, void** out) {
    *out = NULL;
    if (t == Py_None) return 0;
    PyObject* v = PyObject_CallMethodNoArgs(t, s_data_ptr);
    if (v == NULL) return -1;
    *out = PyLong_AsVoidPtr(v);
    Py_DECREF(v);
    return PyErr_Occurred() ? -1 : 0;
}
static int attr_address(PyObject* o, PyObject* name, void** out) {
    PyObject* t = PyObject_GetAttr(o, name);
    if (t == NULL) return -1;
    const int r = address(t, out);
    Py_DECREF(t);
    return r;
}
static int shape(PyObject* t, int n, int64_t* out) {
    PyObject* s = PyObject_GetAttr(t, s_shape);
    if (s == NULL) return -1;
    PyObject* f = PySequence_Fast(s, "a shape is a sequence");
    Py_DECREF(s);
    if (f == NULL) return -1;
    if (PySequence_Fast_GET_SIZE(f) != n) {
        PyErr_Format(PyExc_ValueError, "expected a tensor of %d dimensions, got %zd", n, PySequence_Fast_GET_SIZE(f));
        Py_DECREF(f);
        return -1;
    }
    for (int i = 0; i < n; ++i) out[i] = PyLong_AsLongLong(PySequence_Fast_GET_ITEM(f, i));
    Py_DECREF(f);
    return PyErr_Occurred() ? -1 : 0;
}
static int integer(PyObject* v, int64_t* out) {
    *out = PyLong_AsLongLong(v);
    return *out == -1 && PyErr_Occurred() ? -1 : 0;
}
static int small(PyObject* v, int* out) {
    const long r = PyLong_AsLong(v);
    if (r == -1 && PyErr_Occurred()) return -1;
    *out = (int)r;
    return 0;
}
static int pitch(PyObject* t, int64_t* out) {
    PyObject* v = PyObject_CallMethodOneArg(t, s_stride, zero);
    if (v == NULL) return -1;
    const int r = integer(v, out);
    Py_DECREF(v);
    return r;
}
static int dtype(PyObject* t, hq_dtype* out) {
    PyObject* d = PyObject_GetAttr(t, s_dtype);
    if (d == NULL) return -1;
    for (int i = 0; i < 2; ++i)
        if (d == known_dtype[i]) {
            Py_DECREF(d);
            *out = (hq_dtype)known_code[i];
            return 0;
        }
    PyObject* c = PyObject_CallOneArg(dtype_code, t);        /* raises for a type that is not taken */
    int code;
    if (c == NULL || small(c, &code) != 0) {
        Py_XDECREF(c);
        Py_DECREF(d);
        return -1;
    }
    Py_DECREF(c);
    const int slot = known_dtype[0] == NULL ? 0 : 1;
    if (known_dtype[slot] == NULL) {
        known_code[slot] = code;
        known_dtype[slot] = d;                               /* kept */
    } else {
        Py_DECREF(d);
    }
    *out = (hq_dtype)code;
    return 0;
}
static int bytes_of(PyObject* t, size_t* out) {
    PyObject* v = PyObject_GetAttr(t, s_nbytes);
    if (v == NULL) return -1;
    *out = PyLong_AsSize_t(v);
    Py_DECREF(v);
    return PyErr_Occurred() ? -1 : 0;
}
typedef struct { Py_buffer desc; void* blob; void* s_w; } weight;
static int weight_of(PyObject* pw, weight* w) {
    PyObject* d = PyObject_GetAttr(pw, s_desc);
    if (d == NULL) return -1;
    const int r = PyObject_GetBuffer(d, &w->desc, PyBUF_SIMPLE);
    Py_DECREF(d);
    if (r != 0) return -1;
    if ((size_t)w->desc.len >= sizeof(hq_weight_desc) && attr_address(pw, s_blob_dev, &w->blob) == 0 && attr_address(pw, s_s_w_dev, &w->s_w) == 0)
        return 0;
    PyBuffer_Release(&w->desc);
    if (!PyErr_Occurred()) PyErr_SetString(PyExc_TypeError, "not a weight descriptor");
    return -1;
}
static int arguments(Py_ssize_t n, Py_ssize_t want, const void* fn) {
    if (n == want && fn != NULL) return 0;
    PyErr_Format(PyExc_TypeError, fn == NULL ? "not bound" : "expected %zd arguments, got %zd", want, n);
    return -1;
}
#define MODE(o) ((o) == Py_None ? HQ_SCALE_PER_ROW : HQ_SCALE_STATIC)

/* qlinear(x, pw, bias, a_bits, y, workspace, static_scale, dev_status, stream) */
static PyObject* py_qlinear(PyObject* self, PyObject* const* a, Py_ssize_t n) {
    (void)self;
    void *x, *bias, *y, *ws, *ss, *status;
    int64_t dim[2], ldx, ldy, stream;
    hq_dtype xdt, ydt;
    size_t ws_bytes;
    int bits;
    weight w;
    if (arguments(n, 9, f_qlinear) || shape(a[0], 2, dim) || address(a[0], &x) || dtype(a[0], &xdt) || pitch(a[0], &ldx) ||
        address(a[2], &bias) || small(a[3], &bits) || address(a[4], &y) || dtype(a[4], &ydt) || pitch(a[4], &ldy) || address(a[5], &ws) ||
        bytes_of(a[5], &ws_bytes) || address(a[6], &ss) || address(a[7], &status) || integer(a[8], &stream) || weight_of(a[1], &w))
        return NULL;
    hq_status s;
    Py_BEGIN_ALLOW_THREADS
    s = f_qlinear(x, xdt, dim[0], dim[1], ldx, w.desc.buf, w.blob, w.s_w, bias, bits, MODE(a[6]), ss, y, ydt, ldy, ws, ws_bytes, status,
                  (void*)(intptr_t)stream);
    Py_END_ALLOW_THREADS
    PyBuffer_Release(&w.desc);
    return PyLong_FromLong(s);
}

/* qconv(x, pw, R, S, stride, pad, bias, a_bits, y, workspace, static_scale, dev_status, stream) */
static PyObject* py_qconv(PyObject* self, PyObject* const* a, Py_ssize_t n) {
    (void)self;
    void *x, *bias, *y, *ws, *ss, *status;
    int64_t dim[4], stream;
    hq_dtype xdt, ydt;
    size_t ws_bytes;
    int R, S, stride, pad, bits;
    weight w;
    if (arguments(n, 13, f_qconv) || shape(a[0], 4, dim) || address(a[0], &x) || dtype(a[0], &xdt) || small(a[2], &R) || small(a[3], &S) ||
        small(a[4], &stride) || small(a[5], &pad) || address(a[6], &bias) || small(a[7], &bits) || address(a[8], &y) || dtype(a[8], &ydt) ||
        address(a[9], &ws) || bytes_of(a[9], &ws_bytes) || address(a[10], &ss) || address(a[11], &status) || integer(a[12], &stream) ||
        weight_of(a[1], &w))
        return NULL;
    hq_status s;
    Py_BEGIN_ALLOW_THREADS
    s = f_qconv(x, xdt, dim[0], dim[1], dim[2], dim[3], w.desc.buf, w.blob, R, S, stride, pad, w.s_w, bias, bits, MODE(a[10]), ss, y, ydt, ws,
                ws_bytes, status, (void*)(intptr_t)stream);
    Py_END_ALLOW_THREADS
    PyBuffer_Release(&w.desc);
    return PyLong_FromLong(s);
}

/* ln_qlinear(x, ln_weight, ln_bias, rows_per_group, eps, pw, bias, a_bits, y, workspace, dev_status, stream) */
static PyObject* py_ln_qlinear(PyObject* self, PyObject* const* a, Py_ssize_t n) {
    (void)self;
    void *x, *lw, *lb, *bias, *y, *ws, *status;
    int64_t dim[2], ldx, ldy, group, stream;
    hq_dtype xdt, ydt;
    size_t ws_bytes;
    int bits;
    weight w;
    if (arguments(n, 12, f_ln_qlinear)) return NULL;
    const double eps = PyFloat_AsDouble(a[4]);
    if (PyErr_Occurred() || shape(a[0], 2, dim) || address(a[0], &x) || dtype(a[0], &xdt) || pitch(a[0], &ldx) || address(a[1], &lw) ||
        address(a[2], &lb) || integer(a[3], &group) || address(a[6], &bias) || small(a[7], &bits) || address(a[8], &y) || dtype(a[8], &ydt) ||
        pitch(a[8], &ldy) || address(a[9], &ws) || bytes_of(a[9], &ws_bytes) || address(a[10], &status) || integer(a[11], &stream) ||
        weight_of(a[5], &w))
        return NULL;
    hq_status s;
    Py_BEGIN_ALLOW_THREADS
    s = f_ln_qlinear(x, xdt, dim[0], dim[1], ldx, lw, lb, group, (float)eps, w.desc.buf, w.blob, w.s_w, bias, bits, y, ydt, ldy, ws, ws_bytes,
                     status, (void*)(intptr_t)stream);
    Py_END_ALLOW_THREADS
    PyBuffer_Release(&w.desc);
    return PyLong_FromLong(s);
}

/* hadamard_quant(x, had_block, bits, codes, container, scales, static_scale, stream) */
static PyObject* py_quant(PyObject* self, PyObject* const* a, Py_ssize_t n) {
    (void)self;
    void *x, *codes, *scales, *ss;
    int64_t dim[2], ldx, ldc, stream;
    hq_dtype xdt;
    int block, bits, cont;
    if (arguments(n, 8, f_quant) || shape(a[0], 2, dim) || address(a[0], &x) || dtype(a[0], &xdt) || pitch(a[0], &ldx) || small(a[1], &block) ||
        small(a[2], &bits) || address(a[3], &codes) || pitch(a[3], &ldc) || small(a[4], &cont) || address(a[5], &scales) || address(a[6], &ss) ||
        integer(a[7], &stream))
        return NULL;
    hq_status s;
    Py_BEGIN_ALLOW_THREADS
    s = f_quant(x, xdt, dim[0], dim[1], ldx, block, bits, MODE(a[6]), ss, codes, (hq_container)cont, ldc, scales, (void*)(intptr_t)stream);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(s);
}

/* bind(dtype_code, qlinear, qconv, ln_qlinear, hadamard_quant): the type lookup and the addresses of the entry points */
static PyObject* py_bind(PyObject* self, PyObject* args) {
    (void)self;
    PyObject* code;
    unsigned long long p[4];
    if (!PyArg_ParseTuple(args, "OKKKK", &code, &p[0], &p[1], &p[2], &p[3])) return NULL;
    Py_INCREF(code);
    Py_XSETREF(dtype_code, code);
    f_qlinear = (qlinear_fn)(uintptr_t)p[0];
    f_qconv = (qconv_fn)(uintptr_t)p[1];
    f_ln_qlinear = (ln_qlinear_fn)(uintptr_t)p[2];
    f_quant = (quant_fn)(uintptr_t)p[3];
    Py_RETURN_NONE;
}

static PyMethodDef methods[] = {
    {"bind", py_bind, METH_VARARGS, NULL},
    {"qlinear", (PyCFunction)(void (*)(void))py_qlinear, METH_FASTCALL, NULL},
    {"qconv", (PyCFunction)(void (*)(void))py_qconv, METH_FASTCALL, NULL},
    {"ln_qlinear", (PyCFunction)(void (*)(void))py_ln_qlinear, METH_FASTCALL, NULL},
    {"hadamard_quant", (PyCFunction)(void (*)(void))py_quant, METH_FASTCALL, NULL},
    {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_hqcall", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__hqcall(void) {
    s_data_ptr = PyUnicode_InternFromString("data_ptr");
    s_shape = PyUnicode_InternFromString("shape");
    s_stride = PyUnicode_InternFromString("stride");
    s_dtype = PyUnicode_InternFromString("dtype");
    s_nbytes = PyUnicode_InternFromString("nbytes");
    s_desc = PyUnicode_InternFromString("desc");
    s_blob_dev = PyUnicode_InternFromString("blob_dev");
    s_s_w_dev = PyUnicode_InternFromString("s_w_dev");
    zero = PyLong_FromLong(0);
    return PyModule_Create(&module);
}
