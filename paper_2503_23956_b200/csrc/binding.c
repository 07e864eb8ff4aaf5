/* The marshalling of the two entry points that a decoder calls for every token (aircache_decode_attn and
 * aircache_decode_step), natively: a kernel of theirs may take 5 us, and through ctypes the arguments alone took 2.4 and
 * 3.1 us of host time; here 0.6 and 0.8.  Same arguments, same function in libaircache.so, same return code. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>

static PyObject *s_shape, *s_ragged;             /* the binding's structure types */
static PyObject *s_get_device, *s_get_stream;    /* torch's current device and its current stream's raw handle */
static PyObject *s_data_ptr, *s_numel, *s_element_size;

static int struct_address(PyObject *o, PyObject *type, int64_t *w) {
    if (!PyObject_TypeCheck(o, (PyTypeObject *)type)) {
        PyErr_Format(PyExc_TypeError, "expected %s, got %s", ((PyTypeObject *)type)->tp_name, Py_TYPE(o)->tp_name);
        return -1;
    }
    Py_buffer view;
    if (PyObject_GetBuffer(o, &view, PyBUF_SIMPLE)) return -1;
    *w = (int64_t)(intptr_t)view.buf;
    PyBuffer_Release(&view);   /* the caller's reference keeps the structure */
    return 0;
}

static int as_int(PyObject *o, int64_t *w) {
    *w = (int64_t)PyLong_AsUnsignedLongLongMask(o);
    return *w == -1 && PyErr_Occurred() ? -1 : 0;
}

/* None, an address, or an object with data_ptr() */
static int address(PyObject *o, int64_t *w) {
    if (o == Py_None) { *w = 0; return 0; }
    if (PyLong_Check(o)) return as_int(o, w);
    PyObject *r = PyObject_CallMethodNoArgs(o, s_data_ptr);
    if (!r) return -1;
    const int rc = as_int(r, w);
    Py_DECREF(r);
    return rc;
}

/* numel() * element_size(); 0 for None and a raw address */
static int size_of(PyObject *o, int64_t *w) {
    *w = 0;
    if (o == Py_None || PyLong_Check(o)) return 0;
    int64_t n = 0, e = 0;
    PyObject *r = PyObject_CallMethodNoArgs(o, s_numel);
    if (!r || as_int(r, &n)) { Py_XDECREF(r); return -1; }
    Py_DECREF(r);
    r = PyObject_CallMethodNoArgs(o, s_element_size);
    if (!r || as_int(r, &e)) { Py_XDECREF(r); return -1; }
    Py_DECREF(r);
    *w = n * e;
    return 0;
}

/* None (torch's current stream), a raw handle, or an object with cuda_stream */
static int stream_handle(PyObject *o, int64_t *w) {
    PyObject *r;
    if (o == Py_None) {
        PyObject *d = PyObject_CallNoArgs(s_get_device);
        if (!d) return -1;
        r = PyObject_CallOneArg(s_get_stream, d);
        Py_DECREF(d);
    } else if (PyLong_Check(o)) {
        return as_int(o, w);
    } else {
        r = PyObject_GetAttrString(o, "cuda_stream");
    }
    if (!r) return -1;
    const int rc = as_int(r, w);
    Py_DECREF(r);
    return rc;
}

static int tail(PyObject *workspace, PyObject *stream, int64_t *w) {
    return address(workspace, w) || size_of(workspace, w + 1) || stream_handle(stream, w + 2) ? -1 : 0;
}

/* decode_attn(function address, shape, cache, q, out, workspace, stream) */
static PyObject *decode_attn(PyObject *self, PyObject *const *a, Py_ssize_t n) {
    (void)self;
    int64_t f, w[7];
    if (n != 7) { PyErr_SetString(PyExc_TypeError, "decode_attn takes 7 arguments"); return NULL; }
    if (as_int(a[0], &f) || struct_address(a[1], s_shape, &w[0]) || struct_address(a[2], s_ragged, &w[1]) ||
        address(a[3], &w[2]) || address(a[4], &w[3]) || tail(a[5], a[6], &w[4]))
        return NULL;
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = ((int (*)(const void *, const void *, const void *, float *, void *, int64_t, void *))(intptr_t)f)(
        (const void *)w[0], (const void *)w[1], (const void *)w[2], (float *)w[3], (void *)w[4], w[5], (void *)w[6]);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

/* decode_step(function address, shape, cache, q, k_new, v_new, appended, out, workspace, stream) */
static PyObject *decode_step(PyObject *self, PyObject *const *a, Py_ssize_t n) {
    (void)self;
    int64_t f, w[10];
    if (n != 10) { PyErr_SetString(PyExc_TypeError, "decode_step takes 10 arguments"); return NULL; }
    if (as_int(a[0], &f) || struct_address(a[1], s_shape, &w[0]) || struct_address(a[2], s_ragged, &w[1]) ||
        address(a[3], &w[2]) || address(a[4], &w[3]) || address(a[5], &w[4]) || as_int(a[6], &w[5]) ||
        address(a[7], &w[6]) || tail(a[8], a[9], &w[7]))
        return NULL;
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = ((int (*)(const void *, void *, const void *, const void *, const void *, int32_t, float *, void *, int64_t,
                   void *))(intptr_t)f)((const void *)w[0], (void *)w[1], (const void *)w[2], (const void *)w[3],
                                        (const void *)w[4], (int32_t)w[5], (float *)w[6], (void *)w[7], w[8],
                                        (void *)w[9]);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

/* setup(Shape, Ragged, get_device, get_raw_stream), once */
static PyObject *setup(PyObject *self, PyObject *args) {
    (void)self;
    PyObject *shape, *ragged, *dev, *stream;
    if (!PyArg_ParseTuple(args, "O!O!OO", &PyType_Type, &shape, &PyType_Type, &ragged, &dev, &stream)) return NULL;
    Py_INCREF(shape); Py_INCREF(ragged); Py_INCREF(dev); Py_INCREF(stream);
    s_shape = shape; s_ragged = ragged; s_get_device = dev; s_get_stream = stream;
    Py_RETURN_NONE;
}

static PyMethodDef s_methods[] = {
    {"setup", setup, METH_VARARGS, NULL},
    {"decode_attn", (PyCFunction)(void (*)(void))decode_attn, METH_FASTCALL, NULL},
    {"decode_step", (PyCFunction)(void (*)(void))decode_step, METH_FASTCALL, NULL},
    {NULL, NULL, 0, NULL}};
static struct PyModuleDef s_module = {PyModuleDef_HEAD_INIT, "_binding", NULL, -1, s_methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__binding(void) {
    s_data_ptr = PyUnicode_InternFromString("data_ptr");
    s_numel = PyUnicode_InternFromString("numel");
    s_element_size = PyUnicode_InternFromString("element_size");
    if (!s_data_ptr || !s_numel || !s_element_size) return NULL;
    return PyModule_Create(&s_module);
}
