/* CPython entry points of the calls a program makes once per layer or batch (see binding.py).
 *
 * Marshalling a call through ctypes costs 8-12 us -- argument conversion against `argtypes`, a `c_void_p` object per
 * tensor, the Python-level current-stream lookup -- while the launch behind it takes 2-3 us, so short layers were bound
 * by it.  Here a tensor argument is one `data_ptr()` method call, a descriptor is read through the buffer protocol and
 * the current stream comes from torch's C function: 1-2 us a call.  The functions return the ebs_status; the library
 * itself is reached through function pointers handed over by `bind` (so that either build of it can be used), and the
 * GIL is released around it as ctypes does.
 */
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include "ebs.h"

static PyObject *s_data_ptr, *s_cuda_stream, *f_raw_stream, *f_get_device, *t_desc, *t_epilogue, *t_head;

#define EACH_ENTRY(X)                                                                                                 \
    X(ebs_pack_acts) X(ebs_pack_acts_s2d) X(ebs_conv2d_mixed) X(ebs_conv2d_mixed_variant) X(ebs_dequant)              \
    X(ebs_global_avgpool) X(ebs_maxpool_packed) X(ebs_resnet_cifar_forward) X(ebs_search_weight_forward)              \
    X(ebs_search_act_forward) X(ebs_graph_launch)
#define DECLARE_ENTRY(name) static __typeof__(&name) p_##name;
EACH_ENTRY(DECLARE_ENTRY)

/* Device or host address of a tensor argument; None is the null pointer. */
static int as_ptr(PyObject *o, void **out) {
    *out = NULL;
    if (o == Py_None) return 1;
    PyObject *v = PyObject_CallMethodNoArgs(o, s_data_ptr);
    if (!v) return 0;
    *out = PyLong_AsVoidPtr(v);
    Py_DECREF(v);
    return !(*out == NULL && PyErr_Occurred());
}
/* The raw stream of a torch stream object; None is the current stream of the current device. */
static int as_stream(PyObject *o, void **out) {
    PyObject *v;
    if (o == Py_None) {
        PyObject *d = PyObject_CallNoArgs(f_get_device);
        if (!d) return 0;
        v = PyObject_CallOneArg(f_raw_stream, d);
        Py_DECREF(d);
    } else {
        v = PyObject_GetAttr(o, s_cuda_stream);
    }
    if (!v) return 0;
    *out = PyLong_AsVoidPtr(v);
    Py_DECREF(v);
    return !(*out == NULL && PyErr_Occurred());
}
/* An integer: int or a type that is one by __index__ (no conversion: 2.7 or "5" is an error, as it is for a ctypes c_int). */
static int as_int(PyObject *o, int *out) {
    const long v = PyLong_AsLong(o);                        /* (takes __index__, not __int__) */
    if (v == -1 && PyErr_Occurred()) return 0;
    if (v < INT_MIN || v > INT_MAX) {
        PyErr_SetString(PyExc_OverflowError, "integer argument out of range");
        return 0;
    }
    *out = (int)v;
    return 1;
}
static int as_float(PyObject *o, float *out) {
    double v = PyFloat_AsDouble(o);
    if (v == -1.0 && PyErr_Occurred()) return 0;
    *out = (float)v;
    return 1;
}
static int as_size(PyObject *o, size_t *out) {
    PyObject *whole = PyNumber_Index(o);
    if (!whole) return 0;
    *out = PyLong_AsSize_t(whole);
    Py_DECREF(whole);
    return !(*out == (size_t)-1 && PyErr_Occurred());
}
/* A ctypes structure of the given type by value. */
static int as_struct(PyObject *o, PyObject *type, void *out, size_t size) {
    if (!PyObject_TypeCheck(o, (PyTypeObject *)type)) {
        PyErr_Format(PyExc_TypeError, "%s expected instead of %s", ((PyTypeObject *)type)->tp_name, Py_TYPE(o)->tp_name);
        return 0;
    }
    Py_buffer b;
    if (PyObject_GetBuffer(o, &b, PyBUF_SIMPLE)) return 0;
    const int fits = (size_t)b.len == size;
    if (fits) memcpy(out, b.buf, size);
    PyBuffer_Release(&b);
    if (!fits) PyErr_SetString(PyExc_TypeError, "structure argument has another size than the C type");
    return fits;
}
static int arg_count(Py_ssize_t got, Py_ssize_t want) {
    if (got == want) return 1;
    PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, got);
    return 0;
}

#define FAST(name) static PyObject *fast_##name(PyObject *self, PyObject *const *a, Py_ssize_t n)
#define CALL(...)                                                                                                     \
    do {                                                                                                              \
        int rc;                                                                                                       \
        Py_BEGIN_ALLOW_THREADS rc = __VA_ARGS__;                                                                      \
        Py_END_ALLOW_THREADS return PyLong_FromLong(rc);                                                              \
    } while (0)

FAST(pack_acts) {
    void *x, *out, *st;
    int i[7];
    float scale;
    if (!arg_count(n, 11) || !as_ptr(a[0], &x)) return NULL;
    for (int k = 0; k < 7; ++k)
        if (!as_int(a[1 + k], &i[k])) return NULL;
    if (!as_float(a[8], &scale) || !as_ptr(a[9], &out) || !as_stream(a[10], &st)) return NULL;
    CALL(p_ebs_pack_acts(x, i[0], i[1], i[2], i[3], i[4], i[5], i[6], scale, out, st));
}

FAST(pack_acts_s2d) {
    void *x, *out, *st;
    int i[6];
    if (!arg_count(n, 9) || !as_ptr(a[0], &x)) return NULL;
    for (int k = 0; k < 6; ++k)
        if (!as_int(a[1 + k], &i[k])) return NULL;
    if (!as_ptr(a[7], &out) || !as_stream(a[8], &st)) return NULL;
    CALL(p_ebs_pack_acts_s2d(x, i[0], i[1], i[2], i[3], i[4], i[5], out, st));
}

FAST(conv2d_mixed) {
    void *x, *w, *acc, *y, *pn, *st;
    int i[3], variant;
    ebs_conv_desc d;
    ebs_epilogue e;
    if (!arg_count(n, 12) || !as_ptr(a[0], &x)) return NULL;
    for (int k = 0; k < 3; ++k)
        if (!as_int(a[1 + k], &i[k])) return NULL;
    if (!as_ptr(a[4], &w) || !as_struct(a[5], t_desc, &d, sizeof(d)) ||
        (a[6] != Py_None && !as_struct(a[6], t_epilogue, &e, sizeof(e))) ||
        !as_ptr(a[7], &acc) || !as_ptr(a[8], &y) || !as_ptr(a[9], &pn) || !as_stream(a[10], &st) || !as_int(a[11], &variant))
        return NULL;
    const ebs_epilogue *ep = a[6] != Py_None ? &e : NULL;
    if (variant == -1) CALL(p_ebs_conv2d_mixed(x, i[0], i[1], i[2], w, &d, ep, acc, y, pn, st));
    CALL(p_ebs_conv2d_mixed_variant(x, i[0], i[1], i[2], w, &d, ep, acc, y, pn, st, variant));
}

FAST(dequant) {
    void *acc, *cs, *cb, *y, *st;
    size_t pixels;
    int co, relu;
    float scale;
    if (!arg_count(n, 9) || !as_ptr(a[0], &acc) || !as_size(a[1], &pixels) || !as_int(a[2], &co) || !as_float(a[3], &scale) ||
        !as_ptr(a[4], &cs) || !as_ptr(a[5], &cb) || (relu = PyObject_IsTrue(a[6])) < 0 || !as_ptr(a[7], &y) ||
        !as_stream(a[8], &st))
        return NULL;
    CALL(p_ebs_dequant(acc, pixels, co, scale, cs, cb, relu, y, st));
}

FAST(global_avgpool) {
    void *y, *out, *st;
    int i[3];
    if (!arg_count(n, 6) || !as_ptr(a[0], &y)) return NULL;
    for (int k = 0; k < 3; ++k)
        if (!as_int(a[1 + k], &i[k])) return NULL;
    if (!as_ptr(a[4], &out) || !as_stream(a[5], &st)) return NULL;
    CALL(p_ebs_global_avgpool(y, i[0], i[1], i[2], out, st));
}

FAST(maxpool_packed) {
    void *x, *out, *st;
    int i[8];
    if (!arg_count(n, 11) || !as_ptr(a[0], &x)) return NULL;
    for (int k = 0; k < 8; ++k)
        if (!as_int(a[1 + k], &i[k])) return NULL;
    if (!as_ptr(a[9], &out) || !as_stream(a[10], &st)) return NULL;
    CALL(p_ebs_maxpool_packed(x, i[0], i[1], i[2], i[3], i[4], i[5], i[6], i[7], out, st));
}

FAST(resnet_cifar_forward) {
    void *img, *layers, *logits, *trace, *st;
    int i[3], nl;
    ebs_fused_head head;
    if (!arg_count(n, 11) || !as_ptr(a[0], &img)) return NULL;
    for (int k = 0; k < 3; ++k)
        if (!as_int(a[1 + k], &i[k])) return NULL;
    if (!as_ptr(a[4], &layers) || !as_int(a[5], &nl) || !as_struct(a[6], t_head, &head, sizeof(head)) ||
        !as_ptr(a[7], &logits) || !as_ptr(a[8], &trace))
        return NULL;
    const long long stride = PyLong_AsLongLong(a[9]);
    if ((stride == -1 && PyErr_Occurred()) || !as_stream(a[10], &st)) return NULL;
    CALL(p_ebs_resnet_cifar_forward(img, i[0], i[1], i[2], layers, nl, &head, logits, trace, stride, st));
}

/* bits / coefficients: sequences of whatever int() and float() take.  More candidates than the library takes are its error
 * to report. */
static int candidates(PyObject *bits, PyObject *coeff, int *b, float *c, int *n_cand) {
    if (PyObject_Size(bits) < 0 || PyObject_Size(coeff) < 0) return 0;
    PyObject *fb = PySequence_Fast(bits, "bits is not a sequence");
    if (!fb) return 0;
    PyObject *fc = PySequence_Fast(coeff, "coeff is not a sequence");
    int ok = fc != NULL;
    const Py_ssize_t n = PySequence_Fast_GET_SIZE(fb);
    *n_cand = (int)n;
    if (ok && PySequence_Fast_GET_SIZE(fc) != n) {
        PyErr_SetString(PyExc_ValueError, "bits and coeff have different lengths");
        ok = 0;
    }
    for (Py_ssize_t k = 0; ok && k < n && k < EBS_MAX_CANDIDATES; ++k) {
        PyObject *whole = PyNumber_Long(PySequence_Fast_GET_ITEM(fb, k));
        PyObject *real = whole ? PyNumber_Float(PySequence_Fast_GET_ITEM(fc, k)) : NULL;
        ok = real && as_int(whole, &b[k]) && as_float(real, &c[k]);
        Py_XDECREF(whole);
        Py_XDECREF(real);
    }
    Py_DECREF(fb);
    Py_XDECREF(fc);
    return ok;
}

FAST(search_weight_forward) {
    void *w, *out, *scratch, *st;
    size_t count;
    int b[EBS_MAX_CANDIDATES], nc;
    float c[EBS_MAX_CANDIDATES];
    if (!arg_count(n, 7) || !as_ptr(a[0], &w) || !as_size(a[1], &count) || !candidates(a[2], a[3], b, c, &nc) ||
        !as_ptr(a[4], &out) || !as_ptr(a[5], &scratch) || !as_stream(a[6], &st))
        return NULL;
    CALL(p_ebs_search_weight_forward(w, count, b, c, nc, out, scratch, st));
}

FAST(search_act_forward) {
    void *x, *out, *st;
    size_t count;
    int b[EBS_MAX_CANDIDATES], nc;
    float c[EBS_MAX_CANDIDATES], alpha;
    if (!arg_count(n, 7) || !as_ptr(a[0], &x) || !as_size(a[1], &count) || !as_float(a[2], &alpha) ||
        !candidates(a[3], a[4], b, c, &nc) || !as_ptr(a[5], &out) || !as_stream(a[6], &st))
        return NULL;
    CALL(p_ebs_search_act_forward(x, count, alpha, b, c, nc, out, st));
}

FAST(graph_launch) {
    void *st;
    if (!arg_count(n, 2)) return NULL;
    void *exec = PyLong_AsVoidPtr(a[0]);
    if ((!exec && PyErr_Occurred()) || !as_stream(a[1], &st)) return NULL;
    CALL(p_ebs_graph_launch(exec, st));
}

/* same_bytes(structs, bytes): whether the concatenated contents of the structures are exactly `bytes`. */
FAST(same_bytes) {
    if (!arg_count(n, 2)) return NULL;
    PyObject *seq = PySequence_Fast(a[0], "structs is not a sequence");
    if (!seq) return NULL;
    char *want;
    Py_ssize_t left;
    int same = PyBytes_AsStringAndSize(a[1], &want, &left) == 0 ? 1 : -1;
    for (Py_ssize_t k = 0; same > 0 && k < PySequence_Fast_GET_SIZE(seq); ++k) {
        Py_buffer b;
        if (PyObject_GetBuffer(PySequence_Fast_GET_ITEM(seq, k), &b, PyBUF_SIMPLE)) {
            same = -1;
            break;
        }
        same = b.len <= left && memcmp(b.buf, want, b.len) == 0;
        want += b.len;
        left -= b.len;
        PyBuffer_Release(&b);
    }
    Py_DECREF(seq);
    return same < 0 ? NULL : PyBool_FromLong(same && left == 0);
}

/* same_addresses(tensors, bytes): whether the tensors' data pointers, in order, are exactly those in `bytes`. */
FAST(same_addresses) {
    if (!arg_count(n, 2)) return NULL;
    PyObject *seq = PySequence_Fast(a[0], "tensors is not a sequence");
    if (!seq) return NULL;
    char *want;
    Py_ssize_t left;
    int same = PyBytes_AsStringAndSize(a[1], &want, &left) == 0 ? 1 : -1;
    if (same > 0) same = left == PySequence_Fast_GET_SIZE(seq) * (Py_ssize_t)sizeof(void *);
    for (Py_ssize_t k = 0; same > 0 && k < PySequence_Fast_GET_SIZE(seq); ++k, want += sizeof(void *)) {
        void *ptr;
        if (!as_ptr(PySequence_Fast_GET_ITEM(seq, k), &ptr)) same = -1;
        else same = memcmp(&ptr, want, sizeof(ptr)) == 0;
    }
    Py_DECREF(seq);
    return same < 0 ? NULL : PyBool_FromLong(same);
}

/* bind(addresses, raw_stream, get_device, desc, epilogue, head): library entry points by name, torch's raw current stream of
 * a device, torch's current device and the ctypes structure types. */
static PyObject *bind(PyObject *self, PyObject *args) {
    PyObject *addr, *raw, *dev, *desc, *epi, *head;
    if (!PyArg_ParseTuple(args, "O!OOO!O!O!", &PyDict_Type, &addr, &raw, &dev, &PyType_Type, &desc, &PyType_Type, &epi,
                          &PyType_Type, &head))
        return NULL;
#define BIND_ENTRY(name)                                                                                              \
    {                                                                                                                 \
        PyObject *v = PyDict_GetItemString(addr, #name);                                                              \
        if (!v) return PyErr_Format(PyExc_KeyError, "%s", #name);                                                     \
        p_##name = (__typeof__(p_##name))PyLong_AsVoidPtr(v);                                                         \
        if (!p_##name) return PyErr_Occurred() ? NULL : PyErr_Format(PyExc_ValueError, "null address: %s", #name);    \
    }
    EACH_ENTRY(BIND_ENTRY)
    Py_INCREF(raw);
    Py_XSETREF(f_raw_stream, raw);
    Py_INCREF(dev);
    Py_XSETREF(f_get_device, dev);
    Py_INCREF(desc);
    Py_XSETREF(t_desc, desc);
    Py_INCREF(epi);
    Py_XSETREF(t_epilogue, epi);
    Py_INCREF(head);
    Py_XSETREF(t_head, head);
    Py_RETURN_NONE;
}

#define FAST_METHOD(name) {#name, (PyCFunction)(void (*)(void))fast_##name, METH_FASTCALL, NULL}
static PyMethodDef methods[] = {{"bind", bind, METH_VARARGS, NULL},
                                FAST_METHOD(pack_acts),
                                FAST_METHOD(pack_acts_s2d),
                                FAST_METHOD(conv2d_mixed),
                                FAST_METHOD(dequant),
                                FAST_METHOD(global_avgpool),
                                FAST_METHOD(maxpool_packed),
                                FAST_METHOD(resnet_cifar_forward),
                                FAST_METHOD(search_weight_forward),
                                FAST_METHOD(search_act_forward),
                                FAST_METHOD(graph_launch),
                                FAST_METHOD(same_bytes),
                                FAST_METHOD(same_addresses),
                                {NULL, NULL, 0, NULL}};

static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_fastcall", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__fastcall(void) {
    s_data_ptr = PyUnicode_InternFromString("data_ptr");
    s_cuda_stream = PyUnicode_InternFromString("cuda_stream");
    if (!s_data_ptr || !s_cuda_stream) return NULL;
    return PyModule_Create(&module);
}
