/* The kernel entry points that a decode step or a prefill calls op by op, from Python without ctypes: a call of tgp_k_attn() over five KV tiles
 * spent 5 of its 8 us in Python building argument arrays, one of tgp_k_rmsnorm() 1.6 of 4.
 *
 * Every function takes the arguments of its namesake in binding.py, all by position, and returns the library's code - or None, having done
 * nothing, for arguments of any other kind than those that a program passes as a rule (exact lists or tuples of equal length, integers,
 * objects whose type says how their address is read).  binding.py then takes its general path, which accepts or refuses them. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>
#include "tgp.h"

#define TILES_MAX 256

static struct {
    int (*embed)(const void *, const int32_t *, float *, uint32_t, uint32_t, uint32_t, void *);
    int (*rmsnorm)(const float *, uint32_t, const void *, void *, uint32_t, uint32_t, float, void *);
    int (*gemm)(const void *, const void *, float *, uint32_t, uint32_t, uint32_t, uint32_t, uint32_t, int, void *);
    int (*gemm_group)(const void *, uint32_t, const void *const *, float *const *, const uint32_t *, const uint32_t *, uint32_t, uint32_t, int, void *);
    int (*rope_kv)(const float *, const float *, const float *, void *, void *const *, void *const *, uint32_t, const float *, const float *, const tgp_model_cfg *,
                   uint32_t, uint32_t, uint32_t, void *);
    int (*attn)(const void *, void *const *, void *const *, uint32_t, void *, const tgp_model_cfg *, uint32_t, uint32_t, uint32_t, float *, void *);
    int (*swiglu)(const float *, const float *, void *, uint64_t, void *);
    int (*argmax)(const float *, int32_t *, uint32_t, uint32_t, void *);
} lib;
static PyObject *s_data_ptr, *s_cuda_stream, *cfg_type, *array_type;

/* What an argument raised on the way is the general path's to raise again, but for what is no Exception (an interrupt). */
static PyObject *not_mine(void) {
    if (PyErr_Occurred()) {
        if (!PyErr_ExceptionMatches(PyExc_Exception)) return NULL;
        PyErr_Clear();
    }
    Py_RETURN_NONE;
}

/* How the address of an object of a type is read, for the types that say it themselves: a method (a tensor's data_ptr) or an attribute (a stream's
 * cuda_stream) of C.  Written under the interpreter's lock; what is full takes the general path. */
static struct { PyTypeObject *type; PyObject *how; int method; } known[16];
static int n_known;

/* how a type says it (a new reference), or NULL */
static PyObject *how_of(PyTypeObject *t, PyObject *x, int *method) {
    if (PyObject_IsInstance(x, array_type)) return NULL;
    PyObject *d = PyObject_GetAttr((PyObject *)t, s_data_ptr);
    *method = d != NULL;
    if (!d) {
        if (!PyErr_ExceptionMatches(PyExc_AttributeError)) return NULL;
        PyErr_Clear();
        d = PyObject_GetAttr((PyObject *)t, s_cuda_stream);
    }
    if (d && (*method ? !Py_IS_TYPE(d, &PyMethodDescr_Type) : !Py_IS_TYPE(d, &PyGetSetDescr_Type) && !Py_IS_TYPE(d, &PyMemberDescr_Type))) Py_CLEAR(d);
    return d;
}

/* (asking a type may run Python, which may come back here: the table is looked at only when all is known) */
static int learn(PyObject *x) {
    PyTypeObject *t = Py_TYPE(x);
    int method;
    Py_INCREF(t);
    PyObject *d = how_of(t, x, &method);
    if (!d || n_known == (int)(sizeof(known) / sizeof(known[0]))) { Py_XDECREF(d); Py_DECREF(t); return -1; }
    known[n_known].type = t;
    known[n_known].how = d;
    known[n_known].method = method;
    return n_known++;
}

static int address(PyObject *x, void **out) {
    if (x == Py_None) { *out = NULL; return 1; }
    if (PyLong_Check(x)) { *out = (void *)(uintptr_t)PyLong_AsUnsignedLongLongMask(x); return 1; }
    PyTypeObject *t = Py_TYPE(x);
    int i = 0;
    while (i < n_known && known[i].type != t) ++i;
    if (i == n_known && (i = learn(x)) < 0) return 0;
    PyObject *v = known[i].method ? PyObject_CallOneArg(known[i].how, x) : Py_TYPE(known[i].how)->tp_descr_get(known[i].how, x, (PyObject *)t);
    const int ok = v && PyLong_Check(v);
    if (ok) *out = (void *)(uintptr_t)PyLong_AsUnsignedLongLongMask(v);
    Py_XDECREF(v);
    return ok;
}

static int u32(PyObject *x, uint32_t *out) {
    if (!PyLong_Check(x)) return 0;
    *out = (uint32_t)PyLong_AsUnsignedLongMask(x);
    return 1;
}

static int real(PyObject *x, float *out) {
    if (!PyFloat_Check(x)) return 0;
    *out = (float)PyFloat_AS_DOUBLE(x);
    return 1;
}

/* the length of an exact list or tuple, -1: anything else; and an item of it */
static Py_ssize_t length(PyObject *x) { return PyList_CheckExact(x) ? PyList_GET_SIZE(x) : PyTuple_CheckExact(x) ? PyTuple_GET_SIZE(x) : -1; }
static PyObject *item(PyObject *x, Py_ssize_t i) { return PyList_CheckExact(x) ? PyList_GET_ITEM(x, i) : PyTuple_GET_ITEM(x, i); }

/* A data_ptr() may run Python - a function mode is active, as under torch.device(), or a tensor subclass has one - and Python may change the list: its
 * length is looked at before each item, and the item is held while it is asked. */
static int addresses(PyObject *x, Py_ssize_t n, void **out) {
    for (Py_ssize_t i = 0; i < n; ++i) {
        if (length(x) != n) return 0;
        PyObject *v = item(x, i);
        Py_INCREF(v);
        const int ok = address(v, &out[i]);
        Py_DECREF(v);
        if (!ok) return 0;
    }
    return length(x) == n;
}

static int numbers(PyObject *x, Py_ssize_t n, uint32_t *out) {
    if (length(x) != n) return 0;
    for (Py_ssize_t i = 0; i < n; ++i) if (!u32(item(x, i), &out[i])) return 0;        /* (runs no Python) */
    return 1;
}

static int config(PyObject *x, tgp_model_cfg *out) {
    Py_buffer b;
    if ((PyObject *)Py_TYPE(x) != cfg_type) return 0;
    if (PyObject_GetBuffer(x, &b, PyBUF_SIMPLE)) { PyErr_Clear(); return 0; }
    const int ok = b.len == (Py_ssize_t)sizeof(*out);
    if (ok) memcpy(out, b.buf, sizeof(*out));
    PyBuffer_Release(&b);
    return ok;
}

#define CALL(rc, call) int rc; Py_BEGIN_ALLOW_THREADS rc = call; Py_END_ALLOW_THREADS return PyLong_FromLong(rc)
#define ARGS(n) if (nargs != (n)) return not_mine()

static PyObject *f_embed(PyObject *self, PyObject *const *a, Py_ssize_t nargs) {
    void *table, *tok, *x, *st;
    uint32_t M, d, V;
    ARGS(7);
    if (!address(a[0], &table) || !address(a[1], &tok) || !address(a[2], &x) || !u32(a[3], &M) || !u32(a[4], &d) || !u32(a[5], &V) || !address(a[6], &st)) return not_mine();
    CALL(rc, lib.embed(table, tok, x, M, d, V, st));
}

static PyObject *f_rmsnorm(PyObject *self, PyObject *const *a, Py_ssize_t nargs) {
    void *x, *g, *h, *st;
    uint32_t ldx, M, d;
    float eps;
    ARGS(8);
    if (!address(a[0], &x) || !u32(a[1], &ldx) || !address(a[2], &g) || !address(a[3], &h) || !u32(a[4], &M) || !u32(a[5], &d) || !real(a[6], &eps) || !address(a[7], &st)) return not_mine();
    CALL(rc, lib.rmsnorm(x, ldx, g, h, M, d, eps, st));
}

static PyObject *f_gemm(PyObject *self, PyObject *const *a, Py_ssize_t nargs) {
    void *A, *W, *C, *st;
    uint32_t M, n, K, ldc, col0, acc;
    ARGS(10);
    if (!address(a[0], &A) || !address(a[1], &W) || !address(a[2], &C) || !u32(a[3], &M) || !u32(a[4], &n) || !u32(a[5], &K) || !u32(a[6], &ldc) || !u32(a[7], &col0) ||
        !u32(a[8], &acc) || !address(a[9], &st)) return not_mine();
    CALL(rc, lib.gemm(A, W, C, M, n, K, ldc, col0, (int)acc, st));
}

static PyObject *f_gemm_group(PyObject *self, PyObject *const *a, Py_ssize_t nargs) {
    void *A, *st, *W[TGP_GEMM_GROUP_MAX], *C[TGP_GEMM_GROUP_MAX];
    uint32_t M, K, acc, n[TGP_GEMM_GROUP_MAX], ldc[TGP_GEMM_GROUP_MAX];
    ARGS(9);
    const Py_ssize_t c = length(a[1]);
    if (c < 1 || c > (Py_ssize_t)TGP_GEMM_GROUP_MAX || !address(a[0], &A) || !addresses(a[1], c, W) || !addresses(a[2], c, C) || !u32(a[3], &M) || !numbers(a[4], c, n) ||
        !u32(a[5], &K) || !numbers(a[6], c, ldc) || !u32(a[7], &acc) || !address(a[8], &st)) return not_mine();
    CALL(rc, lib.gemm_group(A, (uint32_t)c, (const void *const *)W, (float *const *)C, n, ldc, M, K, (int)acc, st));
}

static PyObject *f_rope_kv(PyObject *self, PyObject *const *a, Py_ssize_t nargs) {
    void *q, *k, *v, *qb, *cs, *sn, *st, *kt[TILES_MAX], *vt[TILES_MAX];
    uint32_t B, q_len, pos0;
    tgp_model_cfg cfg;
    ARGS(13);
    const Py_ssize_t n = length(a[4]);
    if (n < 1 || n > TILES_MAX || !address(a[0], &q) || !address(a[1], &k) || !address(a[2], &v) || !address(a[3], &qb) || !addresses(a[4], n, kt) || !addresses(a[5], n, vt) ||
        !address(a[6], &cs) || !address(a[7], &sn) || !config(a[8], &cfg) || !u32(a[9], &B) || !u32(a[10], &q_len) || !u32(a[11], &pos0) || !address(a[12], &st)) return not_mine();
    CALL(rc, lib.rope_kv(q, k, v, qb, kt, vt, (uint32_t)n, cs, sn, &cfg, B, q_len, pos0, st));
}

static PyObject *f_attn(PyObject *self, PyObject *const *a, Py_ssize_t nargs) {
    void *qb, *ob, *scratch, *st, *kt[TILES_MAX], *vt[TILES_MAX];
    uint32_t B, q_len, pos0;
    tgp_model_cfg cfg;
    ARGS(10);
    const Py_ssize_t n = length(a[1]);
    if (n < 1 || n > TILES_MAX || !address(a[0], &qb) || !addresses(a[1], n, kt) || !addresses(a[2], n, vt) || !address(a[3], &ob) || !config(a[4], &cfg) || !u32(a[5], &B) ||
        !u32(a[6], &q_len) || !u32(a[7], &pos0) || !address(a[8], &scratch) || !address(a[9], &st)) return not_mine();
    CALL(rc, lib.attn(qb, kt, vt, (uint32_t)n, ob, &cfg, B, q_len, pos0, scratch, st));
}

static PyObject *f_swiglu(PyObject *self, PyObject *const *a, Py_ssize_t nargs) {
    void *g, *u, *ab, *st;
    ARGS(5);
    if (!address(a[0], &g) || !address(a[1], &u) || !address(a[2], &ab) || !PyLong_Check(a[3]) || !address(a[4], &st)) return not_mine();
    const uint64_t n = PyLong_AsUnsignedLongLongMask(a[3]);
    CALL(rc, lib.swiglu(g, u, ab, n, st));
}

static PyObject *f_argmax(PyObject *self, PyObject *const *a, Py_ssize_t nargs) {
    void *logits, *out, *st;
    uint32_t B, V;
    ARGS(5);
    if (!address(a[0], &logits) || !address(a[1], &out) || !u32(a[2], &B) || !u32(a[3], &V) || !address(a[4], &st)) return not_mine();
    CALL(rc, lib.argmax(logits, out, B, V, st));
}

/* bind(addresses of the eight entry points in the order of `lib`, type of the model configuration, type of numpy's arrays) */
static PyObject *f_bind(PyObject *self, PyObject *args) {
    unsigned long long p[8];
    PyObject *cfg, *array;
    if (!PyArg_ParseTuple(args, "(KKKKKKKK)OO", &p[0], &p[1], &p[2], &p[3], &p[4], &p[5], &p[6], &p[7], &cfg, &array)) return NULL;
    void **f = (void **)&lib;
    for (int i = 0; i < 8; ++i) f[i] = (void *)(uintptr_t)p[i];
    Py_INCREF(cfg); Py_XSETREF(cfg_type, cfg);
    Py_INCREF(array); Py_XSETREF(array_type, array);
    Py_RETURN_NONE;
}

#define FAST(name) {#name, (PyCFunction)(void (*)(void))f_##name, METH_FASTCALL, NULL}
static PyMethodDef methods[] = {{"bind", f_bind, METH_VARARGS, NULL}, FAST(embed), FAST(rmsnorm), FAST(gemm), FAST(gemm_group), FAST(rope_kv), FAST(attn), FAST(swiglu), FAST(argmax), {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_fastcall", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__fastcall(void) {
    s_data_ptr = PyUnicode_InternFromString("data_ptr");
    s_cuda_stream = PyUnicode_InternFromString("cuda_stream");
    return s_data_ptr && s_cuda_stream ? PyModule_Create(&module) : NULL;
}
