/* The entry points a program calls for every layer and step, bound natively: each takes the arguments of its C counterpart
 * (tensors as objects with data_ptr(), raw addresses as ints, None as NULL; sequences where the C function takes arrays) and
 * returns its status.  Through ctypes a call of a dozen arguments spent 5 to 8 us in argument conversion, which bounded
 * single layers: a 16-channel layer's forward, backward and update took 67 us for 45 us of kernels. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>
#include <string.h>

#include "eoq.h"

static PyObject *str_data_ptr, *str_numel, *str_element_size;

/* address of a tensor, an int that already is one, or None */
static int get_ptr(PyObject *o, void **out)
{
    if (o == Py_None) {
        *out = NULL;
        return 1;
    }
    PyObject *v = NULL;
    if (!PyLong_Check(o)) {
        v = PyObject_CallMethodNoArgs(o, str_data_ptr);
        if (!v) return 0;
        o = v;
    }
    *out = PyLong_AsVoidPtr(o);
    Py_XDECREF(v);
    return *out != NULL || !PyErr_Occurred();
}

static int get_int(PyObject *o, long long *out)
{
    if (PyLong_Check(o)) {
        *out = PyLong_AsLongLong(o);
    } else {
        PyObject *v = PyNumber_Long(o);
        if (!v) return 0;
        *out = PyLong_AsLongLong(v);
        Py_DECREF(v);
    }
    return *out != -1 || !PyErr_Occurred();
}

static int get_u64(PyObject *o, uint64_t *out)
{
    PyObject *v = PyNumber_Long(o);
    if (!v) return 0;
    *out = PyLong_AsUnsignedLongLongMask(v);
    Py_DECREF(v);
    return !PyErr_Occurred();
}

static int call_size(PyObject *o, PyObject *name, size_t *out)
{
    PyObject *v = PyObject_CallMethodNoArgs(o, name);
    if (!v) return 0;
    *out = PyLong_AsSize_t(v);
    Py_DECREF(v);
    return *out != (size_t)-1 || !PyErr_Occurred();
}

static int get_bytes(PyObject *o, size_t *out)
{
    size_t n = 0, e = 0;
    if (o != Py_None && (!call_size(o, str_numel, &n) || !call_size(o, str_element_size, &e))) return 0;
    *out = n * e;
    return 1;
}

static int get_desc(PyObject *o, eoq_conv_desc_t *out)
{
    Py_buffer view;
    if (PyObject_GetBuffer(o, &view, PyBUF_SIMPLE)) return 0;
    const int ok = view.len == (Py_ssize_t)sizeof(*out);
    if (ok) memcpy(out, view.buf, sizeof(*out));
    else PyErr_SetString(PyExc_TypeError, "not a convolution descriptor");
    PyBuffer_Release(&view);
    return ok;
}

static int want(Py_ssize_t n, Py_ssize_t expected)
{
    if (n != expected) PyErr_Format(PyExc_TypeError, "%zd arguments expected, %zd given", expected, n);
    return n == expected;
}

/* The host work of a call runs without the interpreter lock (hooks that call back into Python take it again). */
#define CALL(expr)                                  \
    int st;                                         \
    Py_BEGIN_ALLOW_THREADS st = (expr);             \
    Py_END_ALLOW_THREADS return PyLong_FromLong(st)

#define PTRS(first, count)                                    \
    for (int i = 0; i < (count); ++i)                         \
        if (!get_ptr(a[(first) + i], &p[i])) return NULL

static PyObject *conv_fwd_dev(PyObject *self, PyObject *const *a, Py_ssize_t n)
{
    /* handle desc | x x_exp scalars w w_prep shortcut | relu | x5 x2 relu_mask stream */
    void *h, *p[6], *q[4];
    eoq_conv_desc_t d;
    long long relu;
    if (!want(n, 13) || !get_ptr(a[0], &h) || !get_desc(a[1], &d) || !get_int(a[8], &relu)) return NULL;
    PTRS(2, 6);
    for (int i = 0; i < 4; ++i)
        if (!get_ptr(a[9 + i], &q[i])) return NULL;
    CALL(eoq_conv_fwd_dev((eoq_handle_t)h, &d, (const int8_t *)p[0], (const int32_t *)p[1], (const int32_t *)p[2], (const int8_t *)p[3],
                          p[4], (const int8_t *)p[5], (int)relu, (int8_t *)q[0], (int16_t *)q[1], (uint8_t *)q[2], q[3]));
}

static PyObject *conv_dgrad(PyObject *self, PyObject *const *a, Py_ssize_t n)
{
    /* handle desc | e3 e3_exp w e4 e4_exp sum_e4 acc_dump workspace stream */
    void *h, *p[9];
    eoq_conv_desc_t d;
    size_t bytes;
    if (!want(n, 11) || !get_ptr(a[0], &h) || !get_desc(a[1], &d) || !get_bytes(a[9], &bytes)) return NULL;
    PTRS(2, 9);
    CALL(eoq_conv_dgrad((eoq_handle_t)h, &d, (const int8_t *)p[0], (const int32_t *)p[1], (const int8_t *)p[2], (int8_t *)p[3],
                        (int32_t *)p[4], (int64_t *)p[5], (int32_t *)p[6], p[7], bytes, p[8]));
}

static PyObject *conv_wgrad_dev(PyObject *self, PyObject *const *a, Py_ssize_t n)
{
    /* handle desc | e3 e3_exp x b1_c g g_exp workspace stream */
    void *h, *p[8];
    eoq_conv_desc_t d;
    size_t bytes;
    if (!want(n, 10) || !get_ptr(a[0], &h) || !get_desc(a[1], &d) || !get_bytes(a[8], &bytes)) return NULL;
    PTRS(2, 8);
    CALL(eoq_conv_wgrad_dev((eoq_handle_t)h, &d, (const int8_t *)p[0], (const int32_t *)p[1], (const int8_t *)p[2],
                            (const int32_t *)p[3], (int8_t *)p[4], (int32_t *)p[5], p[6], bytes, p[7]));
}

static PyObject *err_prescale_dev(PyObject *self, PyObject *const *a, Py_ssize_t n)
{
    /* handle | e0 e0_exp relu_mask x2 | n_el | gamma_c e3 e3_exp sum_e1 sum_e1x2 stream */
    void *h, *p[4], *q[6];
    long long n_el;
    if (!want(n, 12) || !get_ptr(a[0], &h) || !get_int(a[5], &n_el)) return NULL;
    PTRS(1, 4);
    for (int i = 0; i < 6; ++i)
        if (!get_ptr(a[6 + i], &q[i])) return NULL;
    CALL(eoq_err_prescale_dev((eoq_handle_t)h, (const int8_t *)p[0], (const int32_t *)p[1], (const uint8_t *)p[2],
                              (const int16_t *)p[3], (size_t)n_el, (const int32_t *)q[0], (int8_t *)q[1], (int32_t *)q[2],
                              (int64_t *)q[3], (int64_t *)q[4], q[5]));
}

static PyObject *quantize(PyObject *self, PyObject *const *a, Py_ssize_t n)
{
    /* handle mode src is_float src_exp n | dst dst_exp workspace stream */
    void *h, *src, *src_exp, *p[4];
    long long mode, is_float, count;
    size_t bytes;
    if (!want(n, 10) || !get_ptr(a[0], &h) || !get_int(a[1], &mode) || !get_ptr(a[2], &src) || !get_int(a[3], &is_float) ||
        !get_ptr(a[4], &src_exp) || !get_int(a[5], &count) || !get_bytes(a[8], &bytes))
        return NULL;
    PTRS(6, 4);
    CALL(eoq_quantize((eoq_handle_t)h, (int)mode, src, (int)is_float, (const int32_t *)src_exp, (size_t)count, p[0], (int32_t *)p[1],
                      p[2], bytes, p[3]));
}

/* `k` arrays of `num` addresses each, one after the other in `out` */
static int get_ptr_arrays(PyObject *const *seqs, int k, Py_ssize_t num, void **out)
{
    for (int j = 0; j < k; ++j) {
        PyObject *f = PySequence_Fast(seqs[j], "a sequence of tensors is expected");
        if (!f) return 0;
        int ok = PySequence_Fast_GET_SIZE(f) == num;
        if (!ok) PyErr_SetString(PyExc_ValueError, "sequences of different lengths");
        for (Py_ssize_t i = 0; i < num && ok; ++i) ok = get_ptr(PySequence_Fast_GET_ITEM(f, i), &out[j * num + i]);
        Py_DECREF(f);
        if (!ok) return 0;
    }
    return 1;
}

static PyObject *update_dev(PyObject *self, PyObject *const *a, Py_ssize_t n)
{
    /* handle | w g g_exp | lr_mant lr_exp round_mode | seed step stream */
    void *h, *step, *stream;
    long long lr_mant, lr_exp, mode;
    uint64_t seed;
    if (!want(n, 10) || !get_ptr(a[0], &h) || !get_int(a[4], &lr_mant) || !get_int(a[5], &lr_exp) || !get_int(a[6], &mode) ||
        !get_u64(a[7], &seed) || !get_ptr(a[8], &step) || !get_ptr(a[9], &stream))
        return NULL;
    const Py_ssize_t num = PySequence_Size(a[1]);
    if (num < 0) return NULL;
    void **ptrs = PyMem_New(void *, 3 * num + 1);
    size_t *sizes = PyMem_New(size_t, num + 1);
    int st = EOQ_OK, ok = ptrs && sizes;
    if (!ok) PyErr_NoMemory();
    ok = ok && get_ptr_arrays(a + 1, 3, num, ptrs);
    if (ok) {
        PyObject *f = PySequence_Fast(a[1], "a sequence of tensors is expected");
        ok = f != NULL;
        for (Py_ssize_t i = 0; i < num && ok; ++i) ok = call_size(PySequence_Fast_GET_ITEM(f, i), str_numel, &sizes[i]);
        Py_XDECREF(f);
    }
    if (ok) {
        Py_BEGIN_ALLOW_THREADS
        st = eoq_update_dev((eoq_handle_t)h, (int)num, (int8_t *const *)ptrs, (const int8_t *const *)(ptrs + num),
                            (const int32_t *const *)(ptrs + 2 * num), sizes, (int32_t)lr_mant, (int32_t)lr_exp, (int)mode, seed,
                            (uint64_t *)step, stream);
        Py_END_ALLOW_THREADS
    }
    PyMem_Free(ptrs);
    PyMem_Free(sizes);
    return ok ? PyLong_FromLong(st) : NULL;
}

static PyObject *weight_prep(PyObject *self, PyObject *const *a, Py_ssize_t n)
{
    /* handle | descs w prep | stream */
    void *h, *stream;
    if (!want(n, 5) || !get_ptr(a[0], &h) || !get_ptr(a[4], &stream)) return NULL;
    const Py_ssize_t num = PySequence_Size(a[1]);
    if (num < 0) return NULL;
    void **ptrs = PyMem_New(void *, 2 * num + 1);
    eoq_conv_desc_t *descs = PyMem_New(eoq_conv_desc_t, num + 1);
    int st = EOQ_OK, ok = ptrs && descs;
    if (!ok) PyErr_NoMemory();
    ok = ok && get_ptr_arrays(a + 2, 2, num, ptrs);
    if (ok) {
        PyObject *f = PySequence_Fast(a[1], "a sequence of descriptors is expected");
        ok = f != NULL;
        for (Py_ssize_t i = 0; i < num && ok; ++i) ok = get_desc(PySequence_Fast_GET_ITEM(f, i), &descs[i]);
        Py_XDECREF(f);
    }
    if (ok) {
        Py_BEGIN_ALLOW_THREADS
        st = eoq_weight_prep((eoq_handle_t)h, (int)num, descs, (const int8_t *const *)ptrs, (void *const *)(ptrs + num), stream);
        Py_END_ALLOW_THREADS
    }
    PyMem_Free(ptrs);
    PyMem_Free(descs);
    return ok ? PyLong_FromLong(st) : NULL;
}

#define METHOD(f) {#f, (PyCFunction)(void (*)(void))f, METH_FASTCALL, NULL}
static PyMethodDef methods[] = {METHOD(conv_fwd_dev), METHOD(conv_dgrad), METHOD(conv_wgrad_dev), METHOD(err_prescale_dev),
                                METHOD(quantize), METHOD(update_dev), METHOD(weight_prep), {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_eoqbind", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__eoqbind(void)
{
    str_data_ptr = PyUnicode_InternFromString("data_ptr");
    str_numel = PyUnicode_InternFromString("numel");
    str_element_size = PyUnicode_InternFromString("element_size");
    if (!str_data_ptr || !str_numel || !str_element_size) return NULL;
    return PyModule_Create(&module);
}
