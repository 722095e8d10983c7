/* Argument marshalling between Python and the C ABI of include/jq.h: one C function per entry point that is called in
 * a loop.  A layer call costs the GPU 10 to 30 us; marshalled by ctypes, with the current stream asked for through
 * torch.cuda, a call of two launches took 18 us on the host and a decoding step 10, more than the GPU needs for short
 * prompts and for a decoding step.  Here a tensor costs its data_ptr(), the shape its buffer, the stream one raw lookup:
 * evict_layer 6.3 us in two launches and 3.5 in one, decode_attention 3.2.
 * The library itself is reached through addresses that the package takes from the libjq it has loaded (bind), so the
 * bounds-checked build can stand in for it. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <stdlib.h>

#include "jq.h"

static struct {
    jq_status (*score)(const void *, const void *, const jq_shape *, float *, void *, size_t, jq_stream_t);
    jq_status (*score_fma)(const void *, const void *, const jq_shape *, float *, void *, size_t, jq_stream_t);
    jq_status (*select_topk)(const float *, const jq_shape *, int32_t *, float *, void *, size_t, jq_stream_t);
    jq_status (*compact_kv)(const void *, const void *, const int32_t *, const jq_shape *, void *, void *, jq_stream_t);
    jq_status (*evict_layer)(const void *, const void *, const void *, const jq_shape *, void *, void *, int32_t *, void *, size_t, jq_stream_t);
    jq_status (*evict_layer_windowed)(const void *, const void *, const void *, const void *, const jq_shape *, void *, void *, int32_t *, void *, size_t, jq_stream_t);
    jq_status (*evict_layer_window_kept)(const void *, const void *, const void *, const void *, const void *, const jq_shape *, void *, void *, int32_t *, void *, size_t, jq_stream_t);
    jq_status (*evict_layer_host)(const void *, const void *, const void *, const jq_shape *, void *, void *, int32_t *, void *, size_t, jq_stream_t);
    jq_status (*evict_ragged)(const void *const *, const void *const *, const void *const *, int, const jq_shape *, const int *, const int *, void *, void *, int32_t *, void *, size_t, jq_stream_t);
    jq_status (*evict_append)(void *, void *, int, int, const void *, const void *, int, const void *, const jq_shape *, int32_t *, void *, size_t, jq_stream_t);
    jq_status (*decode_attention)(const void *, const void *, const void *, int, int, int, float *, void *, size_t, jq_stream_t);
} jq;

static PyObject *s_data_ptr, *s_numel, *s_element_size, *s_shape, *s_cuda_stream;
static PyObject *raw_stream;   /* callable: the current CUDA stream of the current device, as an integer */
static PyObject *shape_type;   /* JqShape */

static const struct { const char *name; void **slot; } slots[] = {
    {"jq_score", (void **)&jq.score}, {"jq_score_fma", (void **)&jq.score_fma}, {"jq_select_topk", (void **)&jq.select_topk},
    {"jq_compact_kv", (void **)&jq.compact_kv}, {"jq_evict_layer", (void **)&jq.evict_layer},
    {"jq_evict_layer_windowed", (void **)&jq.evict_layer_windowed}, {"jq_evict_layer_window_kept", (void **)&jq.evict_layer_window_kept},
    {"jq_evict_layer_host", (void **)&jq.evict_layer_host}, {"jq_evict_ragged", (void **)&jq.evict_ragged},
    {"jq_evict_append", (void **)&jq.evict_append}, {"jq_decode_attention", (void **)&jq.decode_attention},
};

/* bind(addresses, raw_stream, shape_type): the entry points' addresses by name, the stream lookup, the class of a shape. */
static PyObject *bind(PyObject *self, PyObject *args)
{
    PyObject *d, *fn, *cls;
    if (!PyArg_ParseTuple(args, "O!OO!", &PyDict_Type, &d, &fn, &PyType_Type, &cls)) return NULL;
    for (size_t i = 0; i < sizeof slots / sizeof *slots; ++i) {
        PyObject *a = PyDict_GetItemString(d, slots[i].name);
        if (!a) { PyErr_Format(PyExc_KeyError, "%s", slots[i].name); return NULL; }
        void *p = PyLong_AsVoidPtr(a);
        if (!p) { if (!PyErr_Occurred()) PyErr_SetString(PyExc_ValueError, slots[i].name); return NULL; }
        *slots[i].slot = p;
    }
    Py_INCREF(fn);
    Py_XSETREF(raw_stream, fn);
    Py_INCREF(cls);
    Py_XSETREF(shape_type, cls);
    Py_RETURN_NONE;
}

/* What int(o) gives, as a C int (as ctypes takes it: the low bits). */
static int to_int(PyObject *o, int *out)
{
    PyObject *v = PyNumber_Long(o);
    if (!v) return -1;
    *out = (int)PyLong_AsUnsignedLongMask(v);
    Py_DECREF(v);
    return 0;
}
/* Integer result of a method without arguments; -1 with an exception set on failure. */
static long long ask(PyObject *o, PyObject *method)
{
    PyObject *r = PyObject_CallMethodNoArgs(o, method);
    if (!r) return -1;
    const long long v = PyLong_AsLongLong(r);
    Py_DECREF(r);
    return v;
}
/* A tensor's address. */
static int address(PyObject *o, void **p)
{
    PyObject *r = PyObject_CallMethodNoArgs(o, s_data_ptr);
    if (!r) return -1;
    *p = PyLong_AsVoidPtr(r);
    Py_DECREF(r);
    return !*p && PyErr_Occurred() ? -1 : 0;
}
/* The same; None is a null pointer. */
static int ptr(PyObject *o, void **p)
{
    *p = NULL;
    return o == Py_None ? 0 : address(o, p);
}
/* Bytes of a workspace: its elements (a workspace is made of bytes; of another type it has to hold as many elements). */
static int bytes_of(PyObject *ws, size_t *n)
{
    const long long e = ask(ws, s_numel);
    if (e == -1 && PyErr_Occurred()) return -1;
    *n = (size_t)e;
    return 0;
}
/* Bytes of a decoding workspace, of any type. */
static int size_of(PyObject *ws, size_t *n)
{
    const long long k = ask(ws, s_element_size);
    if ((k == -1 && PyErr_Occurred()) || bytes_of(ws, n)) return -1;
    *n *= (size_t)k;
    return 0;
}
static int dim(PyObject *t, Py_ssize_t i, int *out)
{
    PyObject *sh = PyObject_GetAttr(t, s_shape);
    if (!sh) return -1;
    PyObject *v = PySequence_GetItem(sh, i);
    Py_DECREF(sh);
    if (!v) return -1;
    const int bad = to_int(v, out);
    Py_DECREF(v);
    return bad;
}
static int shape_of(PyObject *s, jq_shape *out)
{
    Py_buffer b;
    if (!PyObject_TypeCheck(s, (PyTypeObject *)shape_type)) {
        PyErr_Format(PyExc_TypeError, "expected a JqShape, got %.100s", Py_TYPE(s)->tp_name);
        return -1;
    }
    if (PyObject_GetBuffer(s, &b, PyBUF_SIMPLE)) return -1;
    const int ok = b.len == (Py_ssize_t)sizeof *out;
    if (ok) *out = *(const jq_shape *)b.buf;
    PyBuffer_Release(&b);
    if (!ok) { PyErr_SetString(PyExc_TypeError, "expected a JqShape"); return -1; }
    return 0;
}
static int stream_of(PyObject *o, jq_stream_t *out)
{
    PyObject *r = o == Py_None ? PyObject_CallNoArgs(raw_stream) : PyObject_GetAttr(o, s_cuda_stream);
    if (!r) return -1;
    *out = (jq_stream_t)PyLong_AsVoidPtr(r);
    Py_DECREF(r);
    return PyErr_Occurred() ? -1 : 0;
}
/* Leading tensors of a call. */
static int ptrs(PyObject *const *a, int n, void **p)
{
    for (int i = 0; i < n; ++i) if (ptr(a[i], p + i)) return -1;
    return 0;
}
static int want(Py_ssize_t n, Py_ssize_t m)
{
    if (n == m) return 0;
    PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", m, n);
    return -1;
}

#define CALL(expr) do { jq_status rc_; Py_BEGIN_ALLOW_THREADS rc_ = (expr); Py_END_ALLOW_THREADS return PyLong_FromLong((long)rc_); } while (0)
#define FN(name) static PyObject *name(PyObject *self, PyObject *const *a, Py_ssize_t n)

/* K, Q, shape, scores, ws, stream, fma */
FN(score)
{
    void *p[2], *sc, *ws; size_t wb; jq_shape s; jq_stream_t st;
    if (want(n, 7) || ptrs(a, 2, p) || shape_of(a[2], &s) || ptr(a[3], &sc) || ptr(a[4], &ws) || bytes_of(a[4], &wb) || stream_of(a[5], &st)) return NULL;
    const int fma = PyObject_IsTrue(a[6]);
    if (fma < 0) return NULL;
    CALL((fma ? jq.score_fma : jq.score)(p[0], p[1], &s, sc, ws, wb, st));
}
/* scores, shape, idx, ws, pooled, stream */
FN(select_topk)
{
    void *sc, *idx, *ws, *pooled; size_t wb; jq_shape s; jq_stream_t st;
    if (want(n, 6) || ptr(a[0], &sc) || shape_of(a[1], &s) || ptr(a[2], &idx) || ptr(a[3], &ws) || bytes_of(a[3], &wb) || ptr(a[4], &pooled) || stream_of(a[5], &st)) return NULL;
    CALL(jq.select_topk(sc, &s, idx, pooled, ws, wb, st));
}
/* K, V, idx, shape, Kout, Vout, stream */
FN(compact_kv)
{
    void *p[3], *o[2]; jq_shape s; jq_stream_t st;
    if (want(n, 7) || ptrs(a, 3, p) || shape_of(a[3], &s) || ptrs(a + 4, 2, o) || stream_of(a[6], &st)) return NULL;
    CALL(jq.compact_kv(p[0], p[1], p[2], &s, o[0], o[1], st));
}
/* K, V, Q, shape, Kout, Vout, idx, ws, stream */
FN(evict_layer)
{
    void *p[3], *o[4]; size_t wb; jq_shape s; jq_stream_t st;
    if (want(n, 9) || ptrs(a, 3, p) || shape_of(a[3], &s) || ptrs(a + 4, 4, o) || bytes_of(a[7], &wb) || stream_of(a[8], &st)) return NULL;
    CALL(jq.evict_layer(p[0], p[1], p[2], &s, o[0], o[1], o[2], o[3], wb, st));
}
/* the same with host tensors and a device buffer */
FN(evict_layer_host)
{
    void *p[3], *o[4]; size_t wb; jq_shape s; jq_stream_t st;
    if (want(n, 9) || ptrs(a, 3, p) || shape_of(a[3], &s) || ptrs(a + 4, 4, o) || bytes_of(a[7], &wb) || stream_of(a[8], &st)) return NULL;
    CALL(jq.evict_layer_host(p[0], p[1], p[2], &s, o[0], o[1], o[2], o[3], wb, st));
}
/* K, V, Q, Kwin, shape, Kout, Vout, idx, ws, stream */
FN(evict_layer_windowed)
{
    void *p[4], *o[4]; size_t wb; jq_shape s; jq_stream_t st;
    if (want(n, 10) || ptrs(a, 4, p) || shape_of(a[4], &s) || ptrs(a + 5, 4, o) || bytes_of(a[8], &wb) || stream_of(a[9], &st)) return NULL;
    CALL(jq.evict_layer_windowed(p[0], p[1], p[2], p[3], &s, o[0], o[1], o[2], o[3], wb, st));
}
/* K, V, Q, Kwin, Vwin, shape, Kout, Vout, idx, ws, stream */
FN(evict_layer_window_kept)
{
    void *p[5], *o[4]; size_t wb; jq_shape s; jq_stream_t st;
    if (want(n, 11) || ptrs(a, 5, p) || shape_of(a[5], &s) || ptrs(a + 6, 4, o) || bytes_of(a[9], &wb) || stream_of(a[10], &st)) return NULL;
    CALL(jq.evict_layer_window_kept(p[0], p[1], p[2], p[3], p[4], &s, o[0], o[1], o[2], o[3], wb, st));
}
/* Kc, Vc, n_old, Knew, Vnew, Qrecent, shape, idx, ws, stream */
FN(evict_append)
{
    void *p[2], *q[3], *o[2]; size_t wb; jq_shape s; jq_stream_t st; int cap, n_old, n_new = 0;
    if (want(n, 10) || ptrs(a, 2, p) || dim(a[0], 1, &cap) || to_int(a[2], &n_old) || ptrs(a + 3, 3, q) || (a[3] != Py_None && dim(a[3], 1, &n_new)) ||
        shape_of(a[6], &s) || ptrs(a + 7, 2, o) || bytes_of(a[8], &wb) || stream_of(a[9], &st)) return NULL;
    CALL(jq.evict_append(p[0], p[1], cap, n_old, q[0], q[1], n_new, q[2], &s, o[0], o[1], wb, st));
}
/* Kc, Vc, q, out, ws, stream */
FN(decode_attention)
{
    void *p[5]; size_t wb; jq_stream_t st; int Hkv, Hq, rows;
    if (want(n, 6) || ptrs(a, 5, p) || dim(a[0], 0, &Hkv) || dim(a[2], 0, &Hq) || dim(a[0], 1, &rows) || size_of(a[4], &wb) || stream_of(a[5], &st)) return NULL;
    CALL(jq.decode_attention(p[0], p[1], p[2], Hkv, Hq, rows, p[3], p[4], wb, st));
}

/* The addresses of a sequence of tensors, one per unit; units beyond its end get null pointers, which the call rejects. */
static int list_ptrs(PyObject *l, Py_ssize_t n, void **p)
{
    PyObject *f = PySequence_Fast(l, "expected a sequence of tensors");
    if (!f) return -1;
    const Py_ssize_t have = PySequence_Fast_GET_SIZE(f);
    int bad = have > n;
    if (bad) PyErr_Format(PyExc_IndexError, "%zd tensors for %zd units", have, n);
    for (Py_ssize_t i = 0; i < n && !bad; ++i) {
        p[i] = NULL;
        if (i < have) bad = address(PySequence_Fast_GET_ITEM(f, i), p + i) != 0;
    }
    Py_DECREF(f);
    return bad ? -1 : 0;
}
/* The first n of a list of numbers. */
static int list_ints(PyObject *l, Py_ssize_t n, int *p)
{
    if (PyObject_Size(l) < 0) return -1;   /* (an iterator is no list) */
    PyObject *f = PySequence_Fast(l, "expected a sequence of integers");
    if (!f) return -1;
    int bad = PySequence_Fast_GET_SIZE(f) < n;
    if (bad) PyErr_Format(PyExc_ValueError, "%zd numbers for %zd units", PySequence_Fast_GET_SIZE(f), n);
    for (Py_ssize_t i = 0; i < n && !bad; ++i) bad = to_int(PySequence_Fast_GET_ITEM(f, i), p + i) != 0;
    Py_DECREF(f);
    return bad ? -1 : 0;
}
/* Ks, Vs, Qs, shape, L or None, budget or None, Kout, Vout, idx, ws, stream */
FN(evict_ragged)
{
    if (want(n, 11)) return NULL;
    const Py_ssize_t m = PyObject_Size(a[0]);
    if (m < 0) return NULL;
    void **buf = malloc((3 * (size_t)m + 1) * sizeof *buf);
    int *ib = malloc((2 * (size_t)m + 1) * sizeof *ib);
    PyObject *res = NULL;
    void *o[4]; size_t wb; jq_shape s; jq_stream_t st;
    if (!buf || !ib) { PyErr_NoMemory(); goto out; }
    if (list_ptrs(a[0], m, buf) || list_ptrs(a[1], m, buf + m) || list_ptrs(a[2], m, buf + 2 * m) || shape_of(a[3], &s) ||
        (a[4] != Py_None && list_ints(a[4], m, ib)) || (a[5] != Py_None && list_ints(a[5], m, ib + m)) ||
        ptrs(a + 6, 4, o) || bytes_of(a[9], &wb) || stream_of(a[10], &st)) goto out;
    {
        jq_status rc;
        Py_BEGIN_ALLOW_THREADS
        rc = jq.evict_ragged((const void *const *)buf, (const void *const *)(buf + m), (const void *const *)(buf + 2 * m), (int)m, &s,
                             a[4] == Py_None ? NULL : ib, a[5] == Py_None ? NULL : ib + m, o[0], o[1], o[2], o[3], wb, st);
        Py_END_ALLOW_THREADS
        res = PyLong_FromLong((long)rc);
    }
out:
    free(buf);
    free(ib);
    return res;
}

#define DEF(name) {#name, (PyCFunction)(void (*)(void))name, METH_FASTCALL, NULL}
static PyMethodDef methods[] = {
    {"bind", bind, METH_VARARGS, NULL},
    DEF(score), DEF(select_topk), DEF(compact_kv), DEF(evict_layer), DEF(evict_layer_host), DEF(evict_layer_windowed),
    DEF(evict_layer_window_kept), DEF(evict_append), DEF(decode_attention), DEF(evict_ragged),
    {NULL, NULL, 0, NULL},
};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_jqcall", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__jqcall(void)
{
    s_data_ptr = PyUnicode_InternFromString("data_ptr");
    s_numel = PyUnicode_InternFromString("numel");
    s_element_size = PyUnicode_InternFromString("element_size");
    s_shape = PyUnicode_InternFromString("shape");
    s_cuda_stream = PyUnicode_InternFromString("cuda_stream");
    return PyModule_Create(&module);
}
