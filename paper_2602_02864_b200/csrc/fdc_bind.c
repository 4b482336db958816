/* The calls of a pass (fdc_frontier, fdc_build_masks, and per layer fdc_kv_append, fdc_decode_attn) for Python without
 * ctypes.  What bounds a pass that the host issues call by call is the host: ctypes takes 2.1 to 2.9 us to convert the 8 to 13
 * arguments of a call, about as long as the launch itself; here the same arguments (integers, tensors, None) take 0.5 to 0.7 us.
 *
 * A function returns the library's return code, or None when an argument is of a kind that it does not convert;
 * the caller then makes the call through ctypes, which accepts and refuses what it always did. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <stdint.h>

#include "fdc.h"

static PyTypeObject *tensor_type, *kv_type;
static PyObject *data_ptr_name;
static __typeof__(&fdc_frontier) p_frontier;
static __typeof__(&fdc_build_masks) p_build_masks;
static __typeof__(&fdc_kv_append) p_kv_append;
static __typeof__(&fdc_decode_attn) p_decode_attn;

/* An address: None, an int or a tensor. */
static int as_ptr(PyObject *o, void **out)
{
    if (o == Py_None) {
        *out = NULL;
        return 1;
    }
    if (PyLong_CheckExact(o)) {
        *out = PyLong_AsVoidPtr(o);
    } else if (PyObject_TypeCheck(o, tensor_type)) {
        PyObject *r = PyObject_CallMethodNoArgs(o, data_ptr_name);
        if (!r || !PyLong_CheckExact(r)) {
            Py_XDECREF(r);
            PyErr_Clear();
            return 0;
        }
        *out = PyLong_AsVoidPtr(r);
        Py_DECREF(r);
    } else {
        return 0;
    }
    if (!*out && PyErr_Occurred()) {
        PyErr_Clear();
        return 0;
    }
    return 1;
}
static int as_ptrs(PyObject *const *args, int n, void **out)
{
    for (int i = 0; i < n; ++i)
        if (!as_ptr(args[i], out + i)) return 0;
    return 1;
}
static int as_i32(PyObject *o, int32_t *out)
{
    int over = 0;
    long v;
    if (!PyLong_CheckExact(o)) return 0;
    v = PyLong_AsLongAndOverflow(o, &over);
    if (over || v < INT32_MIN || v > INT32_MAX) return 0;
    *out = (int32_t)v;
    return 1;
}
/* The cache descriptor (a ctypes structure): copied, so that nothing refers to it once the lock is given up. */
static int as_kv(PyObject *o, fdc_kv_desc *out)
{
    Py_buffer b;
    int ok;
    if (Py_TYPE(o) != kv_type) return 0;
    if (PyObject_GetBuffer(o, &b, PyBUF_SIMPLE)) {
        PyErr_Clear();
        return 0;
    }
    ok = b.len == (Py_ssize_t)sizeof(*out);
    if (ok) *out = *(const fdc_kv_desc *)b.buf;
    PyBuffer_Release(&b);
    return ok;
}
static PyObject *done(int rc) { return PyLong_FromLong(rc); }

/* frontier(plan, batch, state, finish, n_active, node, tok_idx, kv_row, pos_id, all_done, stream) */
static PyObject *frontier(PyObject *self, PyObject *const *a, Py_ssize_t n)
{
    void *plan, *x[9];
    int32_t batch;
    int rc;
    if (n != 11 || !p_frontier || !as_ptr(a[0], &plan) || !as_i32(a[1], &batch) || !as_ptrs(a + 2, 9, x)) Py_RETURN_NONE;
    Py_BEGIN_ALLOW_THREADS
    rc = p_frontier((fdc_plan *)plan, batch, x[0], (const uint8_t *)x[1], (int32_t *)x[2], (int32_t *)x[3], (int32_t *)x[4], (int32_t *)x[5],
                    (int32_t *)x[6], (int32_t *)x[7], x[8]);
    Py_END_ALLOW_THREADS
    return done(rc);
}
/* build_masks(plan, batch, state, mask, umask, tiles, ntiles, stream) */
static PyObject *build_masks(PyObject *self, PyObject *const *a, Py_ssize_t n)
{
    void *plan, *x[6];
    int32_t batch;
    int rc;
    if (n != 8 || !p_build_masks || !as_ptr(a[0], &plan) || !as_i32(a[1], &batch) || !as_ptrs(a + 2, 6, x)) Py_RETURN_NONE;
    Py_BEGIN_ALLOW_THREADS
    rc = p_build_masks((fdc_plan *)plan, batch, x[0], (uint64_t *)x[1], (uint64_t *)x[2], (int32_t *)x[3], (int32_t *)x[4], x[5]);
    Py_END_ALLOW_THREADS
    return done(rc);
}
/* kv_append(plan, kv, layer, n_active, kv_row, k_new, v_new, stream) */
static PyObject *kv_append(PyObject *self, PyObject *const *a, Py_ssize_t n)
{
    void *plan, *x[5];
    fdc_kv_desc kv;
    int32_t layer;
    int rc;
    if (n != 8 || !p_kv_append || !as_ptr(a[0], &plan) || !as_kv(a[1], &kv) || !as_i32(a[2], &layer) || !as_ptrs(a + 3, 5, x)) Py_RETURN_NONE;
    Py_BEGIN_ALLOW_THREADS
    rc = p_kv_append((fdc_plan *)plan, &kv, layer, (const int32_t *)x[0], (const int32_t *)x[1], x[2], x[3], x[4]);
    Py_END_ALLOW_THREADS
    return done(rc);
}
/* decode_attn(plan, kv, layer, n_active, mask, tiles, ntiles, q, out, scale, workspace, ws_bytes, stream) */
static PyObject *decode_attn(PyObject *self, PyObject *const *a, Py_ssize_t n)
{
    void *plan, *x[6], *ws, *st;
    fdc_kv_desc kv;
    int32_t layer;
    size_t bytes;
    int rc;
    if (n != 13 || !p_decode_attn || !as_ptr(a[0], &plan) || !as_kv(a[1], &kv) || !as_i32(a[2], &layer) || !as_ptrs(a + 3, 6, x) ||
        !PyFloat_CheckExact(a[9]) || !as_ptr(a[10], &ws) || !PyLong_CheckExact(a[11]) || !as_ptr(a[12], &st))
        Py_RETURN_NONE;
    bytes = PyLong_AsSize_t(a[11]);
    if (bytes == (size_t)-1 && PyErr_Occurred()) {
        PyErr_Clear();
        Py_RETURN_NONE;
    }
    const float scale = (float)PyFloat_AS_DOUBLE(a[9]);
    Py_BEGIN_ALLOW_THREADS
    rc = p_decode_attn((fdc_plan *)plan, &kv, layer, (const int32_t *)x[0], (const uint64_t *)x[1], (const int32_t *)x[2], (const int32_t *)x[3], x[4],
                       x[5], scale, ws, bytes, st);
    Py_END_ALLOW_THREADS
    return done(rc);
}
/* setup(torch.Tensor, fdc_kv_desc, addresses of fdc_frontier, fdc_build_masks, fdc_kv_append, fdc_decode_attn) */
static PyObject *setup(PyObject *self, PyObject *const *a, Py_ssize_t n)
{
    void *x[4];
    if (n != 6 || !PyType_Check(a[0]) || !PyType_Check(a[1])) {
        PyErr_SetString(PyExc_TypeError, "setup(tensor type, descriptor type, four addresses)");
        return NULL;
    }
    for (int i = 0; i < 4; ++i) {
        x[i] = PyLong_AsVoidPtr(a[2 + i]);
        if (!x[i]) {
            if (!PyErr_Occurred()) PyErr_SetString(PyExc_ValueError, "address 0");
            return NULL;
        }
    }
    Py_INCREF(a[0]);
    Py_XSETREF(tensor_type, (PyTypeObject *)a[0]);
    Py_INCREF(a[1]);
    Py_XSETREF(kv_type, (PyTypeObject *)a[1]);
    p_frontier = (__typeof__(p_frontier))x[0];
    p_build_masks = (__typeof__(p_build_masks))x[1];
    p_kv_append = (__typeof__(p_kv_append))x[2];
    p_decode_attn = (__typeof__(p_decode_attn))x[3];
    Py_RETURN_NONE;
}

static PyMethodDef methods[] = {
    {"setup", (PyCFunction)(void (*)(void))setup, METH_FASTCALL, NULL},
    {"frontier", (PyCFunction)(void (*)(void))frontier, METH_FASTCALL, NULL},
    {"build_masks", (PyCFunction)(void (*)(void))build_masks, METH_FASTCALL, NULL},
    {"kv_append", (PyCFunction)(void (*)(void))kv_append, METH_FASTCALL, NULL},
    {"decode_attn", (PyCFunction)(void (*)(void))decode_attn, METH_FASTCALL, NULL},
    {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_fdc_bind", NULL, -1, methods, NULL, NULL, NULL, NULL};
PyMODINIT_FUNC PyInit__fdc_bind(void)
{
    data_ptr_name = PyUnicode_InternFromString("data_ptr");
    return data_ptr_name ? PyModule_Create(&module) : NULL;
}
