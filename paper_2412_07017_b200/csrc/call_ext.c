/* Argument marshalling of the calls that a serving step makes for every layer, as a CPython extension: the C ABI of
 * include/asynclm.h called with the addresses of tensors and arrays.  binding.py uses it where it has been built and the
 * arguments are of the ordinary kinds; everything else goes through ctypes there.
 *
 * Why: a step of few sequences is bound by the host.  Through ctypes, planning 4 sequences took 20.8 us (4.0 of them to turn the
 * four arrays into addresses) and a layer's call 4.2-4.4; so 13.8 (with the headers that such a plan no longer uploads) and
 * 3.6, of which the launch is 2.6.  A step of 4 sequences in one layer: 48.3 -> 29.0 us. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include "asynclm.h"

static int (*fn_plan)(const asynclm_shape*, const asynclm_plan_options*, const asynclm_batch*, void*, size_t, void*, size_t, void*,
                      asynclm_plan_t**);
static int (*fn_append)(const asynclm_plan_t*, const void*, const void*, void*, void*);
static int (*fn_append_rope)(const asynclm_plan_t*, const void*, const void*, void*, void*, double, void*);
static int (*fn_attn)(const asynclm_plan_t*, const void*, const void*, void*, float*, void*);
static int (*fn_step)(const asynclm_plan_t*, const void*, const void*, const void*, void*, void*, float*, void*);
static PyObject *current_device, *raw_stream;      /* callables: () -> device, (device) -> stream handle */
static PyObject *s_data_ptr, *s_numel, *s_cuda_stream, *s_num_q_heads, *s_num_kv_heads, *s_head_dim, *s_page_size;

/* (these return -1 with an exception set on failure) */
static int address(PyObject* tensor, void** out) {
    PyObject* v = PyObject_CallMethodNoArgs(tensor, s_data_ptr);
    if (!v) return -1;
    *out = PyLong_AsVoidPtr(v);
    Py_DECREF(v);
    return PyErr_Occurred() ? -1 : 0;
}

static int address_or_null(PyObject* tensor, void** out) {
    *out = NULL;
    return tensor == Py_None ? 0 : address(tensor, out);
}

static int handle_of(PyObject* v, void** out) {
    *out = v == Py_None ? NULL : PyLong_AsVoidPtr(v);
    return PyErr_Occurred() ? -1 : 0;
}

static int stream_of(PyObject* stream, void** out) {
    PyObject* v;
    if (stream == Py_None) {
        PyObject* device = PyObject_CallNoArgs(current_device);
        if (!device) return -1;
        v = PyObject_CallOneArg(raw_stream, device);
        Py_DECREF(device);
    } else {
        v = PyObject_GetAttr(stream, s_cuda_stream);
    }
    if (!v) return -1;
    *out = PyLong_AsVoidPtr(v);
    Py_DECREF(v);
    return PyErr_Occurred() ? -1 : 0;
}

/* (-1 without an exception where the value does not fit) */
static int int_attr(PyObject* obj, PyObject* name, int32_t* out) {
    PyObject* v = PyObject_GetAttr(obj, name);
    if (!v) return -1;
    const long x = PyLong_AsLong(v);
    Py_DECREF(v);
    *out = (int32_t)x;
    return (x == -1 && PyErr_Occurred()) || x != *out ? -1 : 0;
}

/* A one-dimensional contiguous array of 32-bit integers, held until released; 0 if `obj` is anything else. */
static int int32_array(PyObject* obj, Py_buffer* view) {
    if (PyObject_GetBuffer(obj, view, PyBUF_ND | PyBUF_FORMAT) != 0) {
        PyErr_Clear();
        return 0;
    }
    if (view->ndim == 1 && view->itemsize == 4 && view->format && view->format[0] == 'i' && view->format[1] == 0) return 1;
    PyBuffer_Release(view);
    return 0;
}

static PyObject* py_bind(PyObject* self, PyObject* args) {
    Py_ssize_t plan, append, rope, attn, step;
    PyObject *dev, *raw;
    if (!PyArg_ParseTuple(args, "nnnnnOO", &plan, &append, &rope, &attn, &step, &dev, &raw)) return NULL;
    fn_plan = (void*)plan;
    fn_append = (void*)append;
    fn_append_rope = (void*)rope;
    fn_attn = (void*)attn;
    fn_step = (void*)step;
    Py_XSETREF(current_device, Py_NewRef(dev));
    Py_XSETREF(raw_stream, Py_NewRef(raw));
    Py_RETURN_NONE;
}

/* plan(shape, num_pages, q_indptr, kv_len_before, page_indptr, page_indices, stream, sm_scale, host_ws, dev_ws)
 * -> (status, handle), or None where shape or arrays are not of the kind that needs no conversion. */
static PyObject* py_plan(PyObject* self, PyObject* const* a, Py_ssize_t n) {
    if (n != 10) return PyErr_Format(PyExc_TypeError, "10 arguments expected");
    asynclm_shape shape = {0};
    if (int_attr(a[0], s_num_q_heads, &shape.num_q_heads) || int_attr(a[0], s_num_kv_heads, &shape.num_kv_heads) ||
        int_attr(a[0], s_head_dim, &shape.head_dim) || int_attr(a[0], s_page_size, &shape.page_size)) {
        PyErr_Clear();
        Py_RETURN_NONE;
    }
    shape.num_pages = PyLong_AsLongLong(a[1]);
    if (shape.num_pages == -1 && PyErr_Occurred()) return NULL;
    const double scale = PyFloat_AsDouble(a[7]);
    if (scale == -1.0 && PyErr_Occurred()) return NULL;
    shape.sm_scale = (float)scale;
    void *host = NULL, *dev = NULL, *stream = NULL;
    size_t bytes[2];
    if (address(a[8], &host) || address(a[9], &dev) || stream_of(a[6], &stream)) return NULL;
    for (int k = 0; k < 2; ++k) {
        PyObject* v = PyObject_CallMethodNoArgs(a[8 + k], s_numel);
        if (!v) return NULL;
        bytes[k] = PyLong_AsSize_t(v);
        Py_DECREF(v);
        if (PyErr_Occurred()) return NULL;
    }
    Py_buffer view[4];
    int held = 0;
    while (held < 4 && int32_array(a[2 + held], &view[held])) ++held;
    PyObject* result = NULL;
    if (held < 4) {
        result = Py_NewRef(Py_None);
    } else {
        const asynclm_plan_options options = {0};
        const asynclm_batch batch = {(int32_t)view[1].shape[0], view[0].buf, view[1].buf, view[2].buf, view[3].buf};
        asynclm_plan_t* plan = NULL;
        int rc;
        Py_BEGIN_ALLOW_THREADS
        rc = fn_plan(&shape, &options, &batch, host, bytes[0], dev, bytes[1], stream, &plan);
        Py_END_ALLOW_THREADS
        result = Py_BuildValue("(iN)", rc, PyLong_FromVoidPtr(plan));
    }
    while (held > 0) PyBuffer_Release(&view[--held]);
    return result;
}

/* append(handle, k_new, v_new, kv_pool, stream) -> status, and the others alike */
static PyObject* py_append(PyObject* self, PyObject* const* a, Py_ssize_t n) {
    void *plan, *k, *v, *pool, *stream;
    if (n != 5) return PyErr_Format(PyExc_TypeError, "5 arguments expected");
    if (handle_of(a[0], &plan) || address(a[1], &k) || address(a[2], &v) || address(a[3], &pool) || stream_of(a[4], &stream)) return NULL;
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = fn_append(plan, k, v, pool, stream);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

static PyObject* py_append_rope(PyObject* self, PyObject* const* a, Py_ssize_t n) {
    void *plan, *k, *v, *pool, *q, *stream;
    if (n != 7) return PyErr_Format(PyExc_TypeError, "7 arguments expected");
    const double theta = PyFloat_AsDouble(a[5]);
    if (theta == -1.0 && PyErr_Occurred()) return NULL;
    if (handle_of(a[0], &plan) || address(a[1], &k) || address(a[2], &v) || address(a[3], &pool) || address_or_null(a[4], &q) || stream_of(a[6], &stream))
        return NULL;
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = fn_append_rope(plan, k, v, pool, q, theta, stream);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

static PyObject* py_attn(PyObject* self, PyObject* const* a, Py_ssize_t n) {
    void *plan, *q, *pool, *out, *lse, *stream;
    if (n != 6) return PyErr_Format(PyExc_TypeError, "6 arguments expected");
    if (handle_of(a[0], &plan) || address(a[1], &q) || address(a[2], &pool) || address(a[3], &out) || address_or_null(a[4], &lse) || stream_of(a[5], &stream))
        return NULL;
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = fn_attn(plan, q, pool, out, lse, stream);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

static PyObject* py_step(PyObject* self, PyObject* const* a, Py_ssize_t n) {
    void *plan, *q, *k, *v, *pool, *out, *lse, *stream;
    if (n != 8) return PyErr_Format(PyExc_TypeError, "8 arguments expected");
    if (handle_of(a[0], &plan) || address(a[1], &q) || address(a[2], &k) || address(a[3], &v) || address(a[4], &pool) || address(a[5], &out) ||
        address_or_null(a[6], &lse) || stream_of(a[7], &stream))
        return NULL;
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = fn_step(plan, q, k, v, pool, out, lse, stream);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

static PyMethodDef methods[] = {{"bind", py_bind, METH_VARARGS, "bind(plan, append, append_rope, attn, step, current_device, raw_stream)"},
                                {"plan", (PyCFunction)(void*)py_plan, METH_FASTCALL, NULL},
                                {"append", (PyCFunction)(void*)py_append, METH_FASTCALL, NULL},
                                {"append_rope", (PyCFunction)(void*)py_append_rope, METH_FASTCALL, NULL},
                                {"attn", (PyCFunction)(void*)py_attn, METH_FASTCALL, NULL},
                                {"step", (PyCFunction)(void*)py_step, METH_FASTCALL, NULL},
                                {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "call_ext", NULL, -1, methods};

PyMODINIT_FUNC PyInit_call_ext(void) {
    s_data_ptr = PyUnicode_InternFromString("data_ptr");
    s_numel = PyUnicode_InternFromString("numel");
    s_cuda_stream = PyUnicode_InternFromString("cuda_stream");
    s_num_q_heads = PyUnicode_InternFromString("num_q_heads");
    s_num_kv_heads = PyUnicode_InternFromString("num_kv_heads");
    s_head_dim = PyUnicode_InternFromString("head_dim");
    s_page_size = PyUnicode_InternFromString("page_size");
    if (!s_data_ptr || !s_numel || !s_cuda_stream || !s_num_q_heads || !s_num_kv_heads || !s_head_dim || !s_page_size) return NULL;
    return PyModule_Create(&module);
}
