/* Argument marshalling for the calls a serving loop makes every step: the same work binding.py does through ctypes for
 * the others (check every tensor, take its address and the current stream, make the call without the GIL, return its
 * code), in C.  Twelve arguments through ctypes and Python cost 8 us a call, more than the step's kernel takes for
 * 64 sequences; here they cost under 2. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include "../../include/samdraft.h"

static PyObject *s_is_cuda, *s_dtype, *s_is_contiguous, *s_data_ptr, *s_shape;
static PyObject *s_out[6];
static PyObject *t_int32, *t_float32, *f_stream, *f_host_ptr;
static const char *out_names[6] = {"draft_tokens", "draft_len", "match_len", "source", "state", "status"};

/* address of a contiguous tensor of the given type, on the GPU (cuda = 1) or the host; None is a null pointer */
static int tensor_ptr(PyObject *t, PyObject *dtype, int cuda, const char *name, void **out) {
    *out = NULL;
    if (t == Py_None) return 0;
    PyObject *v = PyObject_GetAttr(t, s_is_cuda);
    int ok = v && (v == Py_True) == cuda;
    Py_XDECREF(v);
    if (ok) { v = PyObject_GetAttr(t, s_dtype); ok = v == dtype; Py_XDECREF(v); }
    if (ok) { v = PyObject_CallMethodNoArgs(t, s_is_contiguous); ok = v == Py_True; Py_XDECREF(v); }
    if (ok) {
        v = PyObject_CallMethodNoArgs(t, s_data_ptr);
        if (v) { *out = PyLong_AsVoidPtr(v); Py_DECREF(v); if (!PyErr_Occurred()) return 0; }
    }
    PyErr_Clear();
    PyErr_Format(PyExc_TypeError, "%s must be a contiguous %s %s tensor", name, dtype == t_float32 ? "float32" : "int32", cuda ? "CUDA" : "CPU");
    return -1;
}
static int dev(PyObject *t, const char *name, void **out) { return tensor_ptr(t, t_int32, 1, name, out); }

/* host buffer: a plain address, a CPU tensor, or anything binding._host_ptr takes */
static int host(PyObject *t, const char *name, void **out) {
    *out = NULL;
    if (t == Py_None) return 0;
    if (PyLong_Check(t)) { *out = PyLong_AsVoidPtr(t); return PyErr_Occurred() ? -1 : 0; }
    if (PyObject_HasAttr(t, s_is_cuda) && !tensor_ptr(t, t_int32, 0, name, out)) return 0;
    PyErr_Clear();
    PyObject *v = PyObject_CallFunction(f_host_ptr, "Os", t, name);
    if (!v) return -1;
    *out = PyLong_AsVoidPtr(v);
    Py_DECREF(v);
    return PyErr_Occurred() ? -1 : 0;
}

static int outputs(PyObject *o, void **p) {
    for (int i = 0; i < 6; i++) {
        PyObject *t = PyObject_GetAttr(o, s_out[i]);
        if (!t) return -1;
        int rc = dev(t, out_names[i], &p[i]);
        Py_DECREF(t);
        if (rc) return rc;
    }
    return 0;
}

/* a plain address, or the raw handle of the current stream of device -1 - x for x < 0 */
static int stream_ptr(PyObject *x, void **out) {
    if (PyLong_Check(x)) {
        long long n = PyLong_AsLongLong(x);
        if (n == -1 && PyErr_Occurred()) { PyErr_Clear(); *out = PyLong_AsVoidPtr(x); return PyErr_Occurred() ? -1 : 0; }
        if (n >= 0) { *out = (void *)(uintptr_t)n; return 0; }
        PyObject *d = PyLong_FromLongLong(-1 - n);
        PyObject *v = d ? PyObject_CallOneArg(f_stream, d) : NULL;
        Py_XDECREF(d);
        if (!v) return -1;
        *out = PyLong_AsVoidPtr(v);
        Py_DECREF(v);
        return PyErr_Occurred() ? -1 : 0;
    }
    PyErr_SetString(PyExc_TypeError, "stream");
    return -1;
}

#define NEED(k) if (n != (k)) { PyErr_Format(PyExc_TypeError, "%d arguments expected, got %zd", (int)(k), n); return NULL; }
#define PTR(T, i) ((T)PyLong_AsVoidPtr(a[i]))
#define INT(i) ((int32_t)PyLong_AsLong(a[i]))
#define CALL(expr) do { if (PyErr_Occurred()) return NULL; int rc; Py_BEGIN_ALLOW_THREADS rc = (expr); Py_END_ALLOW_THREADS return PyLong_FromLong(rc); } while (0)

/* (fn, handle, new_tokens, counts, L, outputs object, stream): sam_step with the row length of new_tokens */
static PyObject *py_step_out(PyObject *self, PyObject *const *a, Py_ssize_t n) {
    NEED(7)
    void *nt, *ct, *o[6], *st;
    if (dev(a[2], "new_tokens", &nt) || dev(a[3], "counts", &ct) || outputs(a[5], o) || stream_ptr(a[6], &st)) return NULL;
    PyObject *shape = PyObject_GetAttr(a[2], s_shape);
    if (!shape) return NULL;
    Py_ssize_t d = PyTuple_Check(shape) ? PyTuple_GET_SIZE(shape) : 0;
    int32_t stride = d > 0 ? (int32_t)PyLong_AsLong(PyTuple_GET_ITEM(shape, d - 1)) : 0;
    Py_DECREF(shape);
    int (*fn)(sam_batch_t *, const int32_t *, int32_t, const int32_t *, int32_t, int32_t *, int32_t *, int32_t *, int32_t *, int32_t *, int32_t *, void *) =
        PTR(void *, 0);
    sam_batch_t *h = PTR(sam_batch_t *, 1);
    int32_t L = INT(4);
    CALL(fn(h, nt, stride, ct, L, o[0], o[1], o[2], o[3], o[4], o[5], st));
}

/* (fn, handle, new_tokens, stride, counts, L, six outputs, stream): sam_step */
static PyObject *py_step(PyObject *self, PyObject *const *a, Py_ssize_t n) {
    NEED(13)
    void *nt, *ct, *o[6], *st;
    if (dev(a[2], "new_tokens", &nt) || dev(a[4], "counts", &ct) || stream_ptr(a[12], &st)) return NULL;
    for (int i = 0; i < 6; i++) if (dev(a[6 + i], out_names[i], &o[i])) return NULL;
    int (*fn)(sam_batch_t *, const int32_t *, int32_t, const int32_t *, int32_t, int32_t *, int32_t *, int32_t *, int32_t *, int32_t *, int32_t *, void *) =
        PTR(void *, 0);
    sam_batch_t *h = PTR(sam_batch_t *, 1);
    int32_t stride = INT(3), L = INT(5);
    CALL(fn(h, nt, stride, ct, L, o[0], o[1], o[2], o[3], o[4], o[5], st));
}

/* the same for sam_step_host (host buffers) */
static PyObject *py_step_host(PyObject *self, PyObject *const *a, Py_ssize_t n) {
    NEED(13)
    void *nt, *ct, *o[6], *st;
    if (host(a[2], "new_tokens", &nt) || host(a[4], "counts", &ct) || stream_ptr(a[12], &st)) return NULL;
    for (int i = 0; i < 6; i++) if (host(a[6 + i], out_names[i], &o[i])) return NULL;
    int (*fn)(sam_batch_t *, const int32_t *, int32_t, const int32_t *, int32_t, int32_t *, int32_t *, int32_t *, int32_t *, int32_t *, int32_t *, void *) =
        PTR(void *, 0);
    sam_batch_t *h = PTR(sam_batch_t *, 1);
    int32_t stride = INT(3), L = INT(5);
    CALL(fn(h, nt, stride, ct, L, o[0], o[1], o[2], o[3], o[4], o[5], st));
}

/* (fn, handle, target, prev_L, prev_draft, prev_len, max_new, L, six outputs, counts_out, accepted_out, stream): sam_step_verified */
static PyObject *py_step_verified(PyObject *self, PyObject *const *a, Py_ssize_t n) {
    NEED(17)
    void *tg, *pd, *pl, *mx, *o[6], *co, *ao, *st;
    if (dev(a[2], "target_tokens", &tg) || dev(a[4], "prev_draft_tokens", &pd) || dev(a[5], "prev_draft_len", &pl) || dev(a[6], "max_new", &mx) ||
        dev(a[14], "counts_out", &co) || dev(a[15], "accepted_out", &ao) || stream_ptr(a[16], &st)) return NULL;
    for (int i = 0; i < 6; i++) if (dev(a[8 + i], out_names[i], &o[i])) return NULL;
    int (*fn)(sam_batch_t *, const int32_t *, int32_t, const int32_t *, const int32_t *, const int32_t *, int32_t, int32_t *, int32_t *, int32_t *, int32_t *,
              int32_t *, int32_t *, int32_t *, int32_t *, void *) = PTR(void *, 0);
    sam_batch_t *h = PTR(sam_batch_t *, 1);
    int32_t pL = INT(3), L = INT(7);
    CALL(fn(h, tg, pL, pd, pl, mx, L, o[0], o[1], o[2], o[3], o[4], o[5], co, ao, st));
}

/* (fn, batch, L, draft, draft_len, source, aux, aux_len, stream): sam_select_auxiliary */
static PyObject *py_select_auxiliary(PyObject *self, PyObject *const *a, Py_ssize_t n) {
    NEED(9)
    void *d, *dl, *so, *x, *xl, *st;
    if (dev(a[3], "draft_tokens", &d) || dev(a[4], "draft_len", &dl) || dev(a[5], "source", &so) || dev(a[6], "aux_tokens", &x) ||
        dev(a[7], "aux_len", &xl) || stream_ptr(a[8], &st)) return NULL;
    int (*fn)(int32_t, int32_t, int32_t *, int32_t *, int32_t *, const int32_t *, const int32_t *, void *) = PTR(void *, 0);
    int32_t B = INT(1), L = INT(2);
    CALL(fn(B, L, d, dl, so, x, xl, st));
}

/* (fn, batch, draft, draft_len, L, target, max_new, new_tokens, stride, counts, accepted, stream): sam_accept_greedy */
static PyObject *py_accept_greedy(PyObject *self, PyObject *const *a, Py_ssize_t n) {
    NEED(12)
    void *d, *dl, *tg, *mx, *nt, *ct, *ac, *st;
    if (dev(a[2], "draft_tokens", &d) || dev(a[3], "draft_len", &dl) || dev(a[5], "target_tokens", &tg) || dev(a[6], "max_new", &mx) ||
        dev(a[7], "new_tokens", &nt) || dev(a[9], "counts", &ct) || dev(a[10], "accepted", &ac) || stream_ptr(a[11], &st)) return NULL;
    int (*fn)(int32_t, const int32_t *, const int32_t *, int32_t, const int32_t *, const int32_t *, int32_t *, int32_t, int32_t *, int32_t *, void *) = PTR(void *, 0);
    int32_t B = INT(1), L = INT(4), stride = INT(8);
    CALL(fn(B, d, dl, L, tg, mx, nt, stride, ct, ac, st));
}

/* (fn, static, batch, states, starts, max_size, k, tokens, parents, probs, sizes, stream): sam_tree_draft */
static PyObject *py_tree_draft(PyObject *self, PyObject *const *a, Py_ssize_t n) {
    NEED(12)
    void *s, *t0, *tk, *pa, *pr, *sz, *st;
    if (dev(a[3], "states", &s) || dev(a[4], "start_tokens", &t0) || dev(a[7], "tree_tokens", &tk) || dev(a[8], "tree_parents", &pa) ||
        tensor_ptr(a[9], t_float32, 1, "tree_probs", &pr) || dev(a[10], "tree_size", &sz) || stream_ptr(a[11], &st)) return NULL;
    int (*fn)(const sam_static_t *, int32_t, const int32_t *, const int32_t *, int32_t, int32_t, int32_t *, int32_t *, float *, int32_t *, void *) = PTR(void *, 0);
    const sam_static_t *h = PTR(const sam_static_t *, 1);
    int32_t B = INT(2), M = INT(5), k = INT(6);
    CALL(fn(h, B, s, t0, M, k, tk, pa, pr, sz, st));
}

/* (fn, static, vocab, batch, tokens, stride, counts, L, l_bias, min_match, six outputs, stream): sam_retrieve_noalloc */
static PyObject *py_retrieve_noalloc(PyObject *self, PyObject *const *a, Py_ssize_t n) {
    NEED(17)
    void *nt, *ct, *o[6], *st;
    if (dev(a[4], "tokens", &nt) || dev(a[6], "counts", &ct) || stream_ptr(a[16], &st)) return NULL;
    for (int i = 0; i < 6; i++) if (dev(a[10 + i], out_names[i], &o[i])) return NULL;
    int (*fn)(const sam_static_t *, int32_t, int32_t, const int32_t *, int32_t, const int32_t *, int32_t, int32_t, int32_t, int32_t *, int32_t *, int32_t *,
              int32_t *, int32_t *, int32_t *, void *) = PTR(void *, 0);
    const sam_static_t *h = PTR(const sam_static_t *, 1);
    int32_t vocab = INT(2), B = INT(3), stride = INT(5), L = INT(7), bias = INT(8), mm = INT(9);
    CALL(fn(h, vocab, B, nt, stride, ct, L, bias, mm, o[0], o[1], o[2], o[3], o[4], o[5], st));
}

/* (torch.int32, torch.float32, raw current stream of a device index, binding._host_ptr) */
static PyObject *py_setup(PyObject *self, PyObject *const *a, Py_ssize_t n) {
    NEED(4)
    Py_INCREF(a[0]); Py_INCREF(a[1]); Py_INCREF(a[2]); Py_INCREF(a[3]);
    t_int32 = a[0]; t_float32 = a[1]; f_stream = a[2]; f_host_ptr = a[3];
    Py_RETURN_NONE;
}

#define M(name) {#name, (PyCFunction)(void (*)(void))py_##name, METH_FASTCALL, NULL}
static PyMethodDef methods[] = {M(setup), M(step_out), M(step), M(step_host), M(step_verified), M(select_auxiliary), M(accept_greedy), M(tree_draft),
                                M(retrieve_noalloc), {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_calls", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__calls(void) {
    s_is_cuda = PyUnicode_InternFromString("is_cuda"); s_dtype = PyUnicode_InternFromString("dtype");
    s_is_contiguous = PyUnicode_InternFromString("is_contiguous"); s_data_ptr = PyUnicode_InternFromString("data_ptr");
    s_shape = PyUnicode_InternFromString("shape");
    for (int i = 0; i < 6; i++) s_out[i] = PyUnicode_InternFromString(out_names[i]);
    return PyModule_Create(&module);
}
