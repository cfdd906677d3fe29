/* The per-call entry points of the Python binding as a CPython extension: argument conversion only.
 *
 * A decode-sized mat-vec runs about 3 us on the GPU, less than ctypes and the lookup of the current stream took on
 * the host (q8_0 2048 x 2048, calls back to back: 8.7 us per call, of which the kernel 3.3).  Here an address costs one
 * method call, the stream one call of the raw-stream lookup, and the arguments no intermediate objects.
 *
 * The extension links against nothing of the library: the binding hands over the addresses of the C functions that it
 * has loaded (bind).  Every function returns the library's status code; the binding turns it into an exception. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>

typedef int (*matvec_fn)(int, const void*, int64_t, int64_t, const float*, float*, int, void*);
typedef int (*dequant_fn)(int, const void*, int64_t, float*, void*);
typedef int (*sequence_fn)(int, int, const void*, void*, int64_t, void*);
typedef int (*sequence_batch_fn)(int, int, const void*, int, void*);
typedef int (*attn_fn)(int, const void*, const void*, const float*, float*, int64_t, int64_t, int64_t, int64_t, float,
                       void*, int64_t, void*);

static matvec_fn p_matvec;
static dequant_fn p_dequant;
static sequence_fn p_sequence;
static sequence_batch_fn p_sequence_batch;
static attn_fn p_attn;

static PyObject *s_data_ptr, *s_ctypes, *s_data, *s_cuda_stream;
static PyObject *g_current_stream;      /* the binding's lookup: public torch API, any state of torch */
static PyObject *g_raw_stream, *g_get_device;   /* torch's raw lookups, used once torch's CUDA state is up; may be NULL */
static int g_cuda_up;

/* Raw address of a tensor (data_ptr), a numpy array or an integer; None is 0. */
static int to_addr(PyObject* o, void** out) {
    if (o == Py_None) {
        *out = NULL;
        return 0;
    }
    if (PyLong_Check(o)) {
        *out = PyLong_AsVoidPtr(o);
        return PyErr_Occurred() ? -1 : 0;
    }
    PyObject* v = PyObject_CallMethodNoArgs(o, s_data_ptr);
    if (!v && PyErr_ExceptionMatches(PyExc_AttributeError)) {
        PyErr_Clear();
        PyObject* c = PyObject_GetAttr(o, s_ctypes);
        if (!c) return -1;
        v = PyObject_GetAttr(c, s_data);
        Py_DECREF(c);
    }
    if (!v) return -1;
    *out = PyLong_AsVoidPtr(v);
    Py_DECREF(v);
    return PyErr_Occurred() ? -1 : 0;
}

static int to_i64(PyObject* o, int64_t* out) {
    *out = PyLong_AsLongLong(o);
    return *out == -1 && PyErr_Occurred() ? -1 : 0;
}

static int to_int(PyObject* o, int* out) {
    int64_t v;
    if (to_i64(o, &v)) return -1;
    *out = (int)v;
    return 0;
}

/* Handle of a stream object, an integer, or (None) the current stream of the current device. */
static int to_stream(PyObject* o, void** out) {
    PyObject* v;
    if (o == Py_None) {
        if (g_cuda_up && g_raw_stream) {
            PyObject* dev = PyObject_CallNoArgs(g_get_device);
            if (!dev) return -1;
            v = PyObject_CallOneArg(g_raw_stream, dev);
            Py_DECREF(dev);
        } else {
            v = PyObject_CallNoArgs(g_current_stream);
            if (v) g_cuda_up = 1;
        }
    } else if (PyLong_Check(o)) {
        Py_INCREF(o);
        v = o;
    } else {
        v = PyObject_GetAttr(o, s_cuda_stream);
    }
    if (!v) return -1;
    *out = PyLong_AsVoidPtr(v);
    Py_DECREF(v);
    return PyErr_Occurred() ? -1 : 0;
}

static int nargs_ok(Py_ssize_t n, Py_ssize_t want) {
    if (n == want) return 1;
    PyErr_Format(PyExc_TypeError, "%zd arguments expected, %zd given", want, n);
    return 0;
}

/* matvec(fmt, W, rows, cols, X, Y, batch, stream) */
static PyObject* py_matvec(PyObject* self, PyObject* const* a, Py_ssize_t n) {
    int fmt, batch, rc;
    int64_t rows, cols;
    void *w, *x, *y, *s;
    if (!nargs_ok(n, 8) || to_int(a[0], &fmt) || to_addr(a[1], &w) || to_i64(a[2], &rows) || to_i64(a[3], &cols) ||
        to_addr(a[4], &x) || to_addr(a[5], &y) || to_int(a[6], &batch) || to_stream(a[7], &s))
        return NULL;
    Py_BEGIN_ALLOW_THREADS
    rc = p_matvec(fmt, w, rows, cols, (const float*)x, (float*)y, batch, s);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

/* dequant(fmt, W, n, out, stream) */
static PyObject* py_dequant(PyObject* self, PyObject* const* a, Py_ssize_t n) {
    int fmt, rc;
    int64_t count;
    void *w, *o, *s;
    if (!nargs_ok(n, 5) || to_int(a[0], &fmt) || to_addr(a[1], &w) || to_i64(a[2], &count) || to_addr(a[3], &o) ||
        to_stream(a[4], &s))
        return NULL;
    Py_BEGIN_ALLOW_THREADS
    rc = p_dequant(fmt, w, count, (float*)o, s);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

/* sequence(fmt, n_items, items address, workspace, workspace bytes, stream) */
static PyObject* py_sequence(PyObject* self, PyObject* const* a, Py_ssize_t n) {
    int fmt, items_n, rc;
    int64_t bytes;
    void *items, *ws, *s;
    if (!nargs_ok(n, 6) || to_int(a[0], &fmt) || to_int(a[1], &items_n) || to_addr(a[2], &items) || to_addr(a[3], &ws) ||
        to_i64(a[4], &bytes) || to_stream(a[5], &s))
        return NULL;
    Py_BEGIN_ALLOW_THREADS
    rc = p_sequence(fmt, items_n, items, ws, bytes, s);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

/* sequence_batch(fmt, n_items, items address, batch, stream) */
static PyObject* py_sequence_batch(PyObject* self, PyObject* const* a, Py_ssize_t n) {
    int fmt, items_n, batch, rc;
    void *items, *s;
    if (!nargs_ok(n, 5) || to_int(a[0], &fmt) || to_int(a[1], &items_n) || to_addr(a[2], &items) || to_int(a[3], &batch) ||
        to_stream(a[4], &s))
        return NULL;
    Py_BEGIN_ALLOW_THREADS
    rc = p_sequence_batch(fmt, items_n, items, batch, s);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

/* attn_decode(fmt, K, V, q, out, n_head, n_kv_head, head_dim, n_pos, scale, workspace, workspace bytes, stream) */
static PyObject* py_attn_decode(PyObject* self, PyObject* const* a, Py_ssize_t n) {
    int fmt, rc;
    int64_t h, kv, d, pos, bytes;
    void *k, *v, *q, *o, *ws, *s;
    double scale;
    if (!nargs_ok(n, 13) || to_int(a[0], &fmt) || to_addr(a[1], &k) || to_addr(a[2], &v) || to_addr(a[3], &q) ||
        to_addr(a[4], &o) || to_i64(a[5], &h) || to_i64(a[6], &kv) || to_i64(a[7], &d) || to_i64(a[8], &pos))
        return NULL;
    scale = PyFloat_AsDouble(a[9]);
    if (scale == -1.0 && PyErr_Occurred()) return NULL;
    if (to_addr(a[10], &ws) || to_i64(a[11], &bytes) || to_stream(a[12], &s)) return NULL;
    Py_BEGIN_ALLOW_THREADS
    rc = p_attn(fmt, k, v, (const float*)q, (float*)o, h, kv, d, pos, (float)scale, ws, bytes, s);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

/* bind(matvec, dequant, sequence, sequence_batch, attn_decode, current_stream, raw_stream or None, get_device or None):
 * the addresses of the C functions and the ways to look up the current stream. */
static PyObject* py_bind(PyObject* self, PyObject* const* a, Py_ssize_t n) {
    void* f[5];
    if (!nargs_ok(n, 8)) return NULL;
    for (int i = 0; i < 5; ++i)
        if (to_addr(a[i], &f[i])) return NULL;
    p_matvec = (matvec_fn)f[0];
    p_dequant = (dequant_fn)f[1];
    p_sequence = (sequence_fn)f[2];
    p_sequence_batch = (sequence_batch_fn)f[3];
    p_attn = (attn_fn)f[4];
    Py_INCREF(a[5]);
    Py_XSETREF(g_current_stream, a[5]);
    if (a[6] != Py_None && a[7] != Py_None) {
        Py_INCREF(a[6]);
        Py_XSETREF(g_raw_stream, a[6]);
        Py_INCREF(a[7]);
        Py_XSETREF(g_get_device, a[7]);
    }
    Py_RETURN_NONE;
}

static PyMethodDef methods[] = {
    {"matvec", (PyCFunction)(void (*)(void))py_matvec, METH_FASTCALL, NULL},
    {"dequant", (PyCFunction)(void (*)(void))py_dequant, METH_FASTCALL, NULL},
    {"sequence", (PyCFunction)(void (*)(void))py_sequence, METH_FASTCALL, NULL},
    {"sequence_batch", (PyCFunction)(void (*)(void))py_sequence_batch, METH_FASTCALL, NULL},
    {"attn_decode", (PyCFunction)(void (*)(void))py_attn_decode, METH_FASTCALL, NULL},
    {"bind", (PyCFunction)(void (*)(void))py_bind, METH_FASTCALL, NULL},
    {NULL, NULL, 0, NULL}};

static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_lwcall", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__lwcall(void) {
    s_data_ptr = PyUnicode_InternFromString("data_ptr");
    s_ctypes = PyUnicode_InternFromString("ctypes");
    s_data = PyUnicode_InternFromString("data");
    s_cuda_stream = PyUnicode_InternFromString("cuda_stream");
    if (!s_data_ptr || !s_ctypes || !s_data || !s_cuda_stream) return NULL;
    return PyModule_Create(&module);
}
