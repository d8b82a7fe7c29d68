/* The calls that a planner makes per layer or per group, for Python: argument marshalling in C over the C ABI.
 *
 * A planning step calls enl_attend once per layer; through ctypes the marshalling of one call (structure fields, array
 * conversions, pointer casts) took about 8 us of host time, longer than the kernel of a short decode step runs.  Here it
 * is about 1 us.  Nothing is computed and nothing is kept between calls; enl.py holds the signatures and raises the errors.
 *
 * Tensors are asked for data_ptr(), and for their sizes only where the caller has not given them.  Index lists are read in
 * place when they are contiguous int32 arrays; anything else goes through the converter that enl.py hands over once. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <string.h>

#include "../../include/enl.h"

static PyObject *s_data_ptr, *s_shape, *to_int32;

/* 0 and NULL for None */
static int tensor_ptr(PyObject *t, void **out)
{
    *out = NULL;
    if (t == Py_None) return 0;
    PyObject *v = PyObject_CallMethodNoArgs(t, s_data_ptr);
    if (!v) return -1;
    *out = PyLong_AsVoidPtr(v);
    Py_DECREF(v);
    return (!*out && PyErr_Occurred()) ? -1 : 0;
}

/* one dimension of a tensor, counted from the end if negative (by `shape`: len() and size() of a tensor take three times as long) */
static int dim_of(PyObject *t, Py_ssize_t at, int32_t *out)
{
    PyObject *shape = PyObject_GetAttr(t, s_shape);
    if (!shape) return -1;
    PyObject *v = NULL;
    if (PyTuple_Check(shape)) {
        const Py_ssize_t n = PyTuple_GET_SIZE(shape), i = at < 0 ? n + at : at;
        if (i >= 0 && i < n) {
            v = PyTuple_GET_ITEM(shape, i);
            Py_INCREF(v);
        } else {
            PyErr_SetString(PyExc_IndexError, "tensor has too few dimensions");
        }
    } else {
        v = PySequence_GetItem(shape, at);
    }
    Py_DECREF(shape);
    if (!v) return -1;
    *out = (int32_t)PyLong_AsLong(v);
    Py_DECREF(v);
    return (*out == -1 && PyErr_Occurred()) ? -1 : 0;
}
static int last_dim(PyObject *t, int32_t *out) { return dim_of(t, -1, out); }
static int first_dim(PyObject *t, int32_t *out) { return dim_of(t, 0, out); }

static int int_arg(PyObject *o, int32_t *out)
{
    const long v = PyLong_AsLong(o);
    if (v == -1 && PyErr_Occurred()) {
        /* numpy integers and the like */
        PyErr_Clear();
        PyObject *i = PyNumber_Index(o);
        if (!i) return -1;
        const long w = PyLong_AsLong(i);
        Py_DECREF(i);
        if (w == -1 && PyErr_Occurred()) return -1;
        *out = (int32_t)w;
        return 0;
    }
    *out = (int32_t)v;
    return 0;
}

static int handle_arg(PyObject *o, void **out)
{
    *out = NULL;
    if (o == Py_None) return 0;
    *out = PyLong_AsVoidPtr(o);
    return (!*out && PyErr_Occurred()) ? -1 : 0;
}

/* an index list as contiguous int32 */
typedef struct {
    const int32_t *p;
    Py_ssize_t n;
    Py_buffer view;
    int held;
} ints_t;

static int ints_get(PyObject *o, ints_t *a)
{
    a->p = NULL;
    a->n = 0;
    a->held = 0;
    if (o == Py_None) return 0;
    PyObject *conv = NULL;
    int got = PyObject_CheckBuffer(o) && PyObject_GetBuffer(o, &a->view, PyBUF_C_CONTIGUOUS | PyBUF_FORMAT) == 0;
    if (got && !(a->view.itemsize == 4 && a->view.ndim == 1 && a->view.format && strcmp(a->view.format, "i") == 0)) {
        PyBuffer_Release(&a->view);
        got = 0;
    }
    if (!got) {
        PyErr_Clear();
        conv = PyObject_CallOneArg(to_int32, o);
        if (!conv) return -1;
        const int rc = PyObject_GetBuffer(conv, &a->view, PyBUF_C_CONTIGUOUS | PyBUF_FORMAT);
        Py_DECREF(conv);                                    /* the view keeps it alive */
        if (rc != 0) return -1;
    }
    a->held = 1;
    a->p = (const int32_t *)a->view.buf;
    a->n = a->view.len / 4;
    return 0;
}

static void ints_free(ints_t *a)
{
    if (a->held) PyBuffer_Release(&a->view);
    a->held = 0;
}

static int want_args(Py_ssize_t n, Py_ssize_t want)
{
    if (n == want) return 0;
    PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, n);
    return -1;
}

/* attend(cache, layer, sel_ids, q, k_new, v_new, out, group_mass, cu_sel, cu_q, cu_new, n_q, n_new, mass_stride, sel_off,
 *        split_hint, flags, stream, group_mass_sum, obj_off) -> return code.  sel_off: a callable that makes the int32 array
 * for n entries and keeps it, or None. */
static PyObject *py_attend(PyObject *self, PyObject *const *v, Py_ssize_t nargs)
{
    (void)self;
    if (want_args(nargs, 20)) return NULL;
    enl_attend_args_t a;
    memset(&a, 0, sizeof a);
    ints_t sel, cs, cq, cn, oo, so;
    sel.held = cs.held = cq.held = cn.held = oo.held = so.held = 0;
    PyObject *so_obj = NULL, *ret = NULL;
    void *cache, *stream, *p;
    int32_t flags;
    if (handle_arg(v[0], &cache) || int_arg(v[1], &a.layer) || ints_get(v[2], &sel)) goto done;
    if (tensor_ptr(v[3], &p)) goto done;
    a.q = p;
    if (tensor_ptr(v[4], &p)) goto done;
    a.k_new = p;
    if (tensor_ptr(v[5], &p)) goto done;
    a.v_new = p;
    if (tensor_ptr(v[6], &a.out)) goto done;
    if (tensor_ptr(v[7], &p)) goto done;
    a.group_mass = (float *)p;
    if (ints_get(v[8], &cs) || ints_get(v[9], &cq) || ints_get(v[10], &cn)) goto done;
    a.batch = v[9] == Py_None ? 1 : (int32_t)cq.n - 1;
    a.sel_ids = sel.p;
    a.n_sel = (int32_t)sel.n;
    a.cu_sel = cs.p;
    a.cu_q = cq.p;
    a.cu_new = cn.p;
    if (v[11] != Py_None ? int_arg(v[11], &a.n_q) : first_dim(v[3], &a.n_q)) goto done;
    if (v[12] != Py_None ? int_arg(v[12], &a.n_new) : first_dim(v[4], &a.n_new)) goto done;
    if (v[13] != Py_None) {
        if (int_arg(v[13], &a.mass_stride)) goto done;
    } else if (v[7] != Py_None && last_dim(v[7], &a.mass_stride)) {
        goto done;
    }
    if (v[14] != Py_None) {
        so_obj = PyObject_CallFunction(v[14], "n", sel.n + (Py_ssize_t)a.batch);
        if (!so_obj || ints_get(so_obj, &so)) goto done;
        a.sel_off_out = (int32_t *)so.p;
    }
    if (int_arg(v[15], &a.split_hint) || int_arg(v[16], &flags) || handle_arg(v[17], &stream)) goto done;
    a.flags = (uint32_t)flags;
    if (v[18] != Py_None) {
        if (tensor_ptr(v[18], &p) || last_dim(v[18], &a.sum_stride)) goto done;
        a.group_mass_sum = (float *)p;
    }
    if (ints_get(v[19], &oo)) goto done;
    a.n_obj = v[19] == Py_None ? 0 : (int32_t)oo.n - 1;
    a.obj_off = oo.p;
    {
        int rc;
        Py_BEGIN_ALLOW_THREADS
        rc = enl_attend((enl_cache_t *)cache, &a, stream);
        Py_END_ALLOW_THREADS
        ret = PyLong_FromLong(rc);
    }
done:
    ints_free(&sel);
    ints_free(&cs);
    ints_free(&cq);
    ints_free(&cn);
    ints_free(&oo);
    ints_free(&so);
    Py_XDECREF(so_obj);
    return ret;
}

/* attend_static(seg_len, n_new, q, k, v, out, group_mass, stream) -> return code */
static PyObject *py_attend_static(PyObject *self, PyObject *const *v, Py_ssize_t nargs)
{
    (void)self;
    if (want_args(nargs, 8)) return NULL;
    enl_static_args_t a;
    memset(&a, 0, sizeof a);
    ints_t seg;
    seg.held = 0;
    PyObject *ret = NULL;
    void *stream, *p;
    if (ints_get(v[0], &seg) || int_arg(v[1], &a.n_new)) goto done;
    if (last_dim(v[2], &a.head_dim)) goto done;
    if (dim_of(v[2], -2, &a.n_q_heads) || dim_of(v[3], -2, &a.n_kv_heads)) goto done;
    a.n_seg = (int32_t)seg.n;
    a.seg_len = seg.n ? seg.p : NULL;
    if (tensor_ptr(v[2], &p)) goto done;
    a.q = p;
    if (tensor_ptr(v[3], &p)) goto done;
    a.k = p;
    if (tensor_ptr(v[4], &p)) goto done;
    a.v = p;
    if (tensor_ptr(v[5], &a.out) || tensor_ptr(v[6], &p)) goto done;
    a.group_mass = (float *)p;
    if (handle_arg(v[7], &stream)) goto done;
    {
        int rc;
        Py_BEGIN_ALLOW_THREADS
        rc = enl_attend_static(&a, stream);
        Py_END_ALLOW_THREADS
        ret = PyLong_FromLong(rc);
    }
done:
    ints_free(&seg);
    return ret;
}

/* store(cache, group_id, layer, n_tokens or None, k, v, mode, stream) -> return code */
static PyObject *py_store(PyObject *self, PyObject *const *v, Py_ssize_t nargs)
{
    (void)self;
    if (want_args(nargs, 8)) return NULL;
    void *cache, *stream, *k, *vv;
    int32_t group, layer, n, mode;
    if (handle_arg(v[0], &cache) || int_arg(v[1], &group) || int_arg(v[2], &layer)) return NULL;
    if (v[4] != Py_None ? first_dim(v[4], &n) : int_arg(v[3], &n)) return NULL;
    if (tensor_ptr(v[4], &k) || tensor_ptr(v[5], &vv) || int_arg(v[6], &mode) || handle_arg(v[7], &stream)) return NULL;
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = enl_group_store((enl_cache_t *)cache, group, layer, n, k, vv, mode, stream);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

/* store_all_layers(cache, group_id, ks, vs, mode, stream) -> return code; ks and vs are lists or tuples of equal length
 * whose tensors have the same number of rows (ValueError otherwise) */
static PyObject *py_store_all(PyObject *self, PyObject *const *v, Py_ssize_t nargs)
{
    (void)self;
    if (want_args(nargs, 6)) return NULL;
    void *cache, *stream;
    int32_t group, mode, n = 0;
    if (handle_arg(v[0], &cache) || int_arg(v[1], &group) || int_arg(v[4], &mode) || handle_arg(v[5], &stream)) return NULL;
    PyObject *ks = PySequence_Fast(v[2], "one K tensor per layer");
    PyObject *vs = ks ? PySequence_Fast(v[3], "one V tensor per layer") : NULL;
    PyObject *ret = NULL;
    const void **ptrs = NULL;
    if (!vs) goto done;
    const Py_ssize_t L = PySequence_Fast_GET_SIZE(ks);
    if (L < 1 || PySequence_Fast_GET_SIZE(vs) != L) {
        PyErr_SetString(PyExc_ValueError, "one K and one V tensor per layer of the cache");
        goto done;
    }
    ptrs = PyMem_Malloc(2 * (size_t)L * sizeof *ptrs);
    if (!ptrs) { PyErr_NoMemory(); goto done; }
    for (int kv = 0; kv < 2; ++kv)
        for (Py_ssize_t l = 0; l < L; ++l) {
            PyObject *t = PySequence_Fast_GET_ITEM(kv ? vs : ks, l);
            int32_t rows;
            void *p;
            if (first_dim(t, &rows) || tensor_ptr(t, &p)) goto done;
            if (kv == 0 && l == 0) n = rows;
            if (rows != n) {
                PyErr_SetString(PyExc_ValueError, "every layer must bring the same number of rows");
                goto done;
            }
            ptrs[kv * L + l] = p;
        }
    {
        int rc;
        Py_BEGIN_ALLOW_THREADS
        rc = enl_group_store_all_layers((enl_cache_t *)cache, group, n, ptrs, ptrs + L, mode, stream);
        Py_END_ALLOW_THREADS
        ret = PyLong_FromLong(rc);
    }
done:
    PyMem_Free((void *)ptrs);
    Py_XDECREF(ks);
    Py_XDECREF(vs);
    return ret;
}

/* set_int32_converter(f): f(sequence) -> contiguous int32 array */
static PyObject *py_set_converter(PyObject *self, PyObject *f)
{
    (void)self;
    Py_INCREF(f);
    Py_XSETREF(to_int32, f);
    Py_RETURN_NONE;
}

static PyMethodDef methods[] = {
    {"attend", (PyCFunction)(void (*)(void))py_attend, METH_FASTCALL, NULL},
    {"attend_static", (PyCFunction)(void (*)(void))py_attend_static, METH_FASTCALL, NULL},
    {"store", (PyCFunction)(void (*)(void))py_store, METH_FASTCALL, NULL},
    {"store_all_layers", (PyCFunction)(void (*)(void))py_store_all, METH_FASTCALL, NULL},
    {"set_int32_converter", py_set_converter, METH_O, NULL},
    {NULL, NULL, 0, NULL},
};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_enl", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__enl(void)
{
    s_data_ptr = PyUnicode_InternFromString("data_ptr");
    s_shape = PyUnicode_InternFromString("shape");
    if (!s_data_ptr || !s_shape) return NULL;
    return PyModule_Create(&module);
}
