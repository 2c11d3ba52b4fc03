/* Argument marshalling of the calls that a decode loop makes per layer and step (compression, append, query push, decode
 * attention) through CPython's C API.  The same rules as the ctypes binding beside it: a tensor crosses as its data pointer
 * and must be contiguous, an int or None is taken as it is, a missing stream means the current one.
 *
 * Bound by the interpreter: through ctypes such a call took 5-7 us, of which the library's own work is about 2. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <stdint.h>

typedef int (*push_fn)(const void *, void *, const void *, int32_t, int32_t, void *);
typedef int (*append_fn)(const void *, void *, void *, const void *, const void *, int32_t *, int32_t, int32_t, void *);
typedef int (*attend_fn)(const void *, const void *, const void *, const void *, const int32_t *, float *, int32_t, int32_t, void *);
typedef int (*stages_fn)(const void *, void *, void *, const void *, int32_t *, int32_t, int32_t, int32_t, float, int32_t *, void *,
                         uint32_t);

static push_fn g_push;
static append_fn g_append;
static attend_fn g_attend;
static stages_fn g_stages;
static PyObject *g_device, *g_raw_stream;    /* current device; its current stream's handle */
static PyObject *g_slow_stream;              /* the binding's own answer, asked until CUDA is initialised */
static PyObject *g_initialised;
static int g_ready;
static PyObject *g_desc_type;                /* the binding's descriptor structure, and its size */
static Py_ssize_t g_desc_size;
static PyObject *s_contiguous, *s_data_ptr, *s_cuda_stream;

static int get_ptr(PyObject *o, void **out)
{
    if (o == Py_None) {
        *out = NULL;
        return 0;
    }
    if (PyLong_Check(o)) {
        *out = (void *)(uintptr_t)PyLong_AsUnsignedLongLongMask(o);
        return PyErr_Occurred() ? -1 : 0;
    }
    PyObject *c = PyObject_CallMethodNoArgs(o, s_contiguous);
    if (!c) return -1;
    const int yes = PyObject_IsTrue(c);
    Py_DECREF(c);
    if (yes < 0) return -1;
    if (!yes) {
        PyErr_SetString(PyExc_AssertionError, "tensors must be contiguous");
        return -1;
    }
    PyObject *v = PyObject_CallMethodNoArgs(o, s_data_ptr);
    if (!v) return -1;
    *out = (void *)(uintptr_t)PyLong_AsUnsignedLongLongMask(v);
    Py_DECREF(v);
    return PyErr_Occurred() ? -1 : 0;
}

static int get_stream(PyObject *o, void **out)
{
    PyObject *v = NULL;
    if (o == Py_None) {
        if (!g_ready) {
            PyObject *i = PyObject_CallNoArgs(g_initialised);
            if (!i) return -1;
            g_ready = PyObject_IsTrue(i) > 0;
            Py_DECREF(i);
        }
        if (g_ready) {
            PyObject *d = PyObject_CallNoArgs(g_device);
            if (!d) return -1;
            v = PyObject_CallOneArg(g_raw_stream, d);
            Py_DECREF(d);
        } else {
            v = PyObject_CallNoArgs(g_slow_stream);
        }
        if (!v) return -1;
        if (v == Py_None) {
            Py_DECREF(v);
            *out = NULL;
            return 0;
        }
    } else if (PyLong_Check(o)) {
        v = Py_NewRef(o);
    } else {
        v = PyObject_GetAttr(o, s_cuda_stream);
        if (!v) {
            if (!PyErr_ExceptionMatches(PyExc_AttributeError)) return -1;
            PyErr_Clear();
            v = PyNumber_Long(o);
            if (!v) return -1;
        }
    }
    *out = (void *)(uintptr_t)PyLong_AsUnsignedLongLongMask(v);
    Py_DECREF(v);
    return PyErr_Occurred() ? -1 : 0;
}

static int get_int(PyObject *o, int32_t *out)
{
    *out = (int32_t)PyLong_AsUnsignedLongLongMask(o);
    return PyErr_Occurred() ? -1 : 0;
}

/* the descriptor (a ctypes structure of the binding's type, nothing else that has bytes) stays where it is while `view` is held */
static int get_desc(PyObject *o, Py_buffer *view)
{
    const int is = (PyObject *)Py_TYPE(o) == g_desc_type ? 1 : PyObject_IsInstance(o, g_desc_type);
    if (is < 0) return -1;
    if (!is) {
        PyErr_Format(PyExc_TypeError, "expected an RkvDesc, got %s", Py_TYPE(o)->tp_name);
        return -1;
    }
    if (PyObject_GetBuffer(o, view, PyBUF_SIMPLE)) return -1;
    if (view->len >= g_desc_size) return 0;
    PyBuffer_Release(view);
    PyErr_SetString(PyExc_TypeError, "the descriptor is too small");
    return -1;
}

static int want(Py_ssize_t n, Py_ssize_t expected)
{
    if (n == expected) return 0;
    PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", expected, n);
    return -1;
}

/* (desc, q_window, q_new, alpha, slot, stream) */
static PyObject *push_query(PyObject *self, PyObject *const *a, Py_ssize_t n)
{
    void *q, *x, *s;
    int32_t alpha, slot;
    Py_buffer d;
    int rc;
    if (want(n, 6) || get_ptr(a[1], &q) || get_ptr(a[2], &x) || get_int(a[3], &alpha) || get_int(a[4], &slot) || get_stream(a[5], &s) ||
        get_desc(a[0], &d))
        return NULL;
    Py_BEGIN_ALLOW_THREADS rc = g_push(d.buf, q, x, alpha, slot, s);
    Py_END_ALLOW_THREADS PyBuffer_Release(&d);
    return PyLong_FromLong(rc);
}

/* (desc, k_cache, v_cache, k_new, v_new, seq_lens, budget, buffer, stream) */
static PyObject *append(PyObject *self, PyObject *const *a, Py_ssize_t n)
{
    void *t[5], *s;
    int32_t budget, buffer;
    Py_buffer d;
    int rc;
    if (want(n, 9)) return NULL;
    for (int i = 0; i < 5; ++i)
        if (get_ptr(a[1 + i], &t[i])) return NULL;
    if (get_int(a[6], &budget) || get_int(a[7], &buffer) || get_stream(a[8], &s) || get_desc(a[0], &d)) return NULL;
    Py_BEGIN_ALLOW_THREADS rc = g_append(d.buf, t[0], t[1], t[2], t[3], t[4], budget, buffer, s);
    Py_END_ALLOW_THREADS PyBuffer_Release(&d);
    return PyLong_FromLong(rc);
}

/* (desc, k_cache, v_cache, q_new, seq_lens, out, budget, buffer, stream) */
static PyObject *decode_attention(PyObject *self, PyObject *const *a, Py_ssize_t n)
{
    void *t[5], *s;
    int32_t budget, buffer;
    Py_buffer d;
    int rc;
    if (want(n, 9)) return NULL;
    for (int i = 0; i < 5; ++i)
        if (get_ptr(a[1 + i], &t[i])) return NULL;
    if (get_int(a[6], &budget) || get_int(a[7], &buffer) || get_stream(a[8], &s) || get_desc(a[0], &d)) return NULL;
    Py_BEGIN_ALLOW_THREADS rc = g_attend(d.buf, t[0], t[1], t[2], t[3], t[4], budget, buffer, s);
    Py_END_ALLOW_THREADS PyBuffer_Release(&d);
    return PyLong_FromLong(rc);
}

/* (desc, k_cache, v_cache, q_window, seq_lens, budget, buffer, alpha, lambda, out_idx, stream, stage_mask) */
static PyObject *compress_stages(PyObject *self, PyObject *const *a, Py_ssize_t n)
{
    void *t[4], *idx, *s;
    int32_t budget, buffer, alpha, mask;
    Py_buffer d;
    int rc;
    if (want(n, 12)) return NULL;
    for (int i = 0; i < 4; ++i)
        if (get_ptr(a[1 + i], &t[i])) return NULL;
    const double lambda = PyFloat_AsDouble(a[8]);
    if (PyErr_Occurred() || get_int(a[5], &budget) || get_int(a[6], &buffer) || get_int(a[7], &alpha) || get_ptr(a[9], &idx) ||
        get_stream(a[10], &s) || get_int(a[11], &mask) || get_desc(a[0], &d))
        return NULL;
    Py_BEGIN_ALLOW_THREADS rc = g_stages(d.buf, t[0], t[1], t[2], t[3], budget, buffer, alpha, (float)lambda, idx, s, (uint32_t)mask);
    Py_END_ALLOW_THREADS PyBuffer_Release(&d);
    return PyLong_FromLong(rc);
}

/* (addresses of rkv_push_query, rkv_append, rkv_decode_attention, rkv_compress_stages; is_initialised, current_device,
 *  raw_stream(device), slow_stream; the descriptor's type and size) */
static PyObject *bind(PyObject *self, PyObject *args)
{
    unsigned long long f[4];
    PyObject *o[5];
    if (!PyArg_ParseTuple(args, "KKKKOOOOOn", &f[0], &f[1], &f[2], &f[3], &o[0], &o[1], &o[2], &o[3], &o[4], &g_desc_size)) return NULL;
    g_push = (push_fn)(uintptr_t)f[0];
    g_append = (append_fn)(uintptr_t)f[1];
    g_attend = (attend_fn)(uintptr_t)f[2];
    g_stages = (stages_fn)(uintptr_t)f[3];
    Py_XSETREF(g_initialised, Py_NewRef(o[0]));
    Py_XSETREF(g_device, Py_NewRef(o[1]));
    Py_XSETREF(g_raw_stream, Py_NewRef(o[2]));
    Py_XSETREF(g_slow_stream, Py_NewRef(o[3]));
    Py_XSETREF(g_desc_type, Py_NewRef(o[4]));
    Py_RETURN_NONE;
}

static PyMethodDef g_methods[] = {{"push_query", (PyCFunction)(void (*)(void))push_query, METH_FASTCALL, NULL},
                                  {"append", (PyCFunction)(void (*)(void))append, METH_FASTCALL, NULL},
                                  {"decode_attention", (PyCFunction)(void (*)(void))decode_attention, METH_FASTCALL, NULL},
                                  {"compress_stages", (PyCFunction)(void (*)(void))compress_stages, METH_FASTCALL, NULL},
                                  {"bind", bind, METH_VARARGS, NULL},
                                  {NULL, NULL, 0, NULL}};

static struct PyModuleDef g_module = {PyModuleDef_HEAD_INIT, "_rkv_call", NULL, -1, g_methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__rkv_call(void)
{
    s_contiguous = PyUnicode_InternFromString("is_contiguous");
    s_data_ptr = PyUnicode_InternFromString("data_ptr");
    s_cuda_stream = PyUnicode_InternFromString("cuda_stream");
    if (!s_contiguous || !s_data_ptr || !s_cuda_stream) return NULL;
    return PyModule_Create(&g_module);
}
