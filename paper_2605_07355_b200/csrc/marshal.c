/* Argument marshalling of the Python binding in C: the entry points of include/ttf.h that a program calls per clip or
 * per batch.  A call through ctypes converts its 12 to 17 arguments one by one in about 4 us, which is more than the
 * driver takes to launch a kernel; here it is about 0.3 us.  No CUDA, no torch: pointers and streams arrive as integers
 * (0 = NULL), the addresses of the library's functions are handed in once by bind().  The GIL is released around every
 * call. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include "ttf.h"

#define NFN 11
static struct {
    int (*compress)(const void*, int, int, int, int, int, float, int, void*, int*, int*, ttf_stream_t);
    int (*compress_ws)(const void*, int, int, int, int, int, float, int, void*, int*, int*, void*, size_t, ttf_stream_t);
    int (*compress_ex)(const void*, int, int, int, int, int, float, int, const ttf_options*, void*, int*, int*, ttf_stream_t);
    int (*compress_segment)(const void*, int, int, int, int, int, float, int, int, void*, int*, int*, ttf_stream_t);
    int (*compress_batch)(const void* const*, int, int, int, int, int, int, float, int, void* const*, int* const*,
                          int* const*, ttf_stream_t);
    int (*compress_batch_ex)(const void* const*, int, int, int, int, int, int, float, int, const ttf_options*, void* const*,
                             int* const*, int* const*, ttf_stream_t);
    int (*query)(const void*, int, int, int, int, int, float, int, int*, unsigned char*, int*, float*, int*, ttf_stream_t);
    int (*query_ws)(const void*, int, int, int, int, int, float, int, int*, unsigned char*, int*, float*, int*, void*, size_t,
                    ttf_stream_t);
    int (*query_ex)(const void*, int, int, int, int, int, float, int, const ttf_options*, int*, unsigned char*, int*, float*,
                    int*, ttf_stream_t);
    int (*restore)(const void*, size_t, int, int, int, const int*, const unsigned char*, const int*, void*, int*,
                   ttf_stream_t);
    int (*stats)(const float*, const unsigned char*, const int*, int, int, int, float, float, long long*, ttf_stream_t);
} fn;

/* the arguments of one call, taken in order; the first conversion that fails leaves a Python error set */
typedef struct { PyObject* const* a; Py_ssize_t n, at; int bad; } Args;

static PyObject* next_arg(Args* s) {
    if (s->bad) return NULL;
    if (s->at >= s->n) { s->bad = 1; PyErr_SetString(PyExc_TypeError, "too few arguments"); return NULL; }
    return s->a[s->at++];
}
static void* ptr(Args* s) {
    PyObject* o = next_arg(s);
    if (!o) return NULL;
    void* p = PyLong_AsVoidPtr(o);
    if (!p && PyErr_Occurred()) s->bad = 1;
    return p;
}
static int num(Args* s) {
    PyObject* o = next_arg(s);
    if (!o) return 0;
    long v = PyLong_AsLong(o);
    if (v == -1 && PyErr_Occurred()) s->bad = 1;
    else if (v != (int)v) { s->bad = 1; PyErr_SetString(PyExc_OverflowError, "argument does not fit an int"); }
    return (int)v;
}
static size_t size(Args* s) {
    PyObject* o = next_arg(s);
    if (!o) return 0;
    size_t v = PyLong_AsSize_t(o);
    if (v == (size_t)-1 && PyErr_Occurred()) s->bad = 1;
    return v;
}
static float real(Args* s) {
    PyObject* o = next_arg(s);
    if (!o) return 0.f;
    double v = PyFloat_AsDouble(o);
    if (v == -1.0 && PyErr_Occurred()) s->bad = 1;
    return (float)v;
}
static int done(Args* s) {
    if (!s->bad && s->at != s->n) { s->bad = 1; PyErr_SetString(PyExc_TypeError, "too many arguments"); }
    return !s->bad;
}

/* the leading arguments that most entry points share */
typedef struct { const void* x; int F, H, W, C, r, dtype; float t; } Clip;
static Clip clip(Args* s) {
    Clip c;
    c.x = ptr(s); c.F = num(s); c.H = num(s); c.W = num(s); c.C = num(s); c.r = num(s); c.t = real(s); c.dtype = num(s);
    return c;
}
static ttf_options options(Args* s) {
    ttf_options o;
    o.anchor_mode = num(s); o.anchor_frame = num(s); o.order = num(s); o.pos_base = num(s);
    return o;
}
static int plain(const ttf_options* o) { return !(o->anchor_mode || o->anchor_frame || o->order || o->pos_base); }

#define CALL(expr)                      \
    if (!done(&s)) return NULL;         \
    int rc;                             \
    Py_BEGIN_ALLOW_THREADS rc = (expr); \
    Py_END_ALLOW_THREADS return PyLong_FromLong(rc)

static PyObject* m_bind(PyObject* self, PyObject* const* a, Py_ssize_t n) {
    if (n != NFN) { PyErr_SetString(PyExc_TypeError, "bind() takes the address of every function"); return NULL; }
    void* p[NFN];
    for (int i = 0; i < NFN; ++i) {
        p[i] = PyLong_AsVoidPtr(a[i]);
        if (!p[i]) { if (!PyErr_Occurred()) PyErr_SetString(PyExc_ValueError, "NULL function"); return NULL; }
    }
    *(void**)&fn.compress = p[0]; *(void**)&fn.compress_ws = p[1]; *(void**)&fn.compress_ex = p[2];
    *(void**)&fn.compress_segment = p[3]; *(void**)&fn.compress_batch = p[4]; *(void**)&fn.compress_batch_ex = p[5];
    *(void**)&fn.query = p[6]; *(void**)&fn.query_ws = p[7]; *(void**)&fn.query_ex = p[8];
    *(void**)&fn.restore = p[9]; *(void**)&fn.stats = p[10];
    Py_RETURN_NONE;
}

/* clip, 4 options, tokens, count, positions, stream */
static PyObject* m_compress(PyObject* self, PyObject* const* a, Py_ssize_t n) {
    Args s = {a, n, 0, 0};
    Clip c = clip(&s);
    ttf_options o = options(&s);
    void* tok = ptr(&s); int* cnt = ptr(&s); int* pos = ptr(&s); ttf_stream_t st = ptr(&s);
    CALL(plain(&o) ? fn.compress(c.x, c.F, c.H, c.W, c.C, c.r, c.t, c.dtype, tok, cnt, pos, st)
                   : fn.compress_ex(c.x, c.F, c.H, c.W, c.C, c.r, c.t, c.dtype, &o, tok, cnt, pos, st));
}
/* clip, tokens, count, positions, workspace, bytes, stream */
static PyObject* m_compress_ws(PyObject* self, PyObject* const* a, Py_ssize_t n) {
    Args s = {a, n, 0, 0};
    Clip c = clip(&s);
    void* tok = ptr(&s); int* cnt = ptr(&s); int* pos = ptr(&s); void* ws = ptr(&s); size_t b = size(&s);
    ttf_stream_t st = ptr(&s);
    CALL(fn.compress_ws(c.x, c.F, c.H, c.W, c.C, c.r, c.t, c.dtype, tok, cnt, pos, ws, b, st));
}
/* clip, frame base, tokens, count, positions, stream */
static PyObject* m_compress_segment(PyObject* self, PyObject* const* a, Py_ssize_t n) {
    Args s = {a, n, 0, 0};
    Clip c = clip(&s);
    int base = num(&s); void* tok = ptr(&s); int* cnt = ptr(&s); int* pos = ptr(&s); ttf_stream_t st = ptr(&s);
    CALL(fn.compress_segment(c.x, c.F, c.H, c.W, c.C, c.r, c.t, c.dtype, base, tok, cnt, pos, st));
}
/* clip, 4 options, anchor, keep, dst, best_sim, fuse_cnt, stream */
static PyObject* m_query(PyObject* self, PyObject* const* a, Py_ssize_t n) {
    Args s = {a, n, 0, 0};
    Clip c = clip(&s);
    ttf_options o = options(&s);
    int* an = ptr(&s); unsigned char* keep = ptr(&s); int* dst = ptr(&s); float* sim = ptr(&s); int* fuse = ptr(&s);
    ttf_stream_t st = ptr(&s);
    CALL(plain(&o) ? fn.query(c.x, c.F, c.H, c.W, c.C, c.r, c.t, c.dtype, an, keep, dst, sim, fuse, st)
                   : fn.query_ex(c.x, c.F, c.H, c.W, c.C, c.r, c.t, c.dtype, &o, an, keep, dst, sim, fuse, st));
}
/* clip, anchor, keep, dst, best_sim, fuse_cnt, workspace, bytes, stream */
static PyObject* m_query_ws(PyObject* self, PyObject* const* a, Py_ssize_t n) {
    Args s = {a, n, 0, 0};
    Clip c = clip(&s);
    int* an = ptr(&s); unsigned char* keep = ptr(&s); int* dst = ptr(&s); float* sim = ptr(&s); int* fuse = ptr(&s);
    void* ws = ptr(&s); size_t b = size(&s); ttf_stream_t st = ptr(&s);
    CALL(fn.query_ws(c.x, c.F, c.H, c.W, c.C, c.r, c.t, c.dtype, an, keep, dst, sim, fuse, ws, b, st));
}
/* compressed, row bytes, F, H, W, anchor, keep, dst, out, row index, stream */
static PyObject* m_restore(PyObject* self, PyObject* const* a, Py_ssize_t n) {
    Args s = {a, n, 0, 0};
    const void* x = ptr(&s); size_t b = size(&s); int F = num(&s), H = num(&s), W = num(&s);
    const int* an = ptr(&s); const unsigned char* keep = ptr(&s); const int* dst = ptr(&s);
    void* out = ptr(&s); int* idx = ptr(&s); ttf_stream_t st = ptr(&s);
    CALL(fn.restore(x, b, F, H, W, an, keep, dst, out, idx, st));
}
/* best_sim, keep, anchor, F, H, W, t, band, out, stream */
static PyObject* m_stats(PyObject* self, PyObject* const* a, Py_ssize_t n) {
    Args s = {a, n, 0, 0};
    const float* sim = ptr(&s); const unsigned char* keep = ptr(&s); const int* an = ptr(&s);
    int F = num(&s), H = num(&s), W = num(&s); float t = real(&s), band = real(&s);
    long long* out = ptr(&s); ttf_stream_t st = ptr(&s);
    CALL(fn.stats(sim, keep, an, F, H, W, t, band, out, st));
}
/* list of clip addresses, F, H, W, C, r, t, dtype, 4 options, lists of token, count and position addresses, stream */
static PyObject* m_compress_batch(PyObject* self, PyObject* const* a, Py_ssize_t n) {
    Args s = {a, n, 0, 0};
    PyObject* lists[4];
    lists[0] = next_arg(&s);
    int F = num(&s), H = num(&s), W = num(&s), C = num(&s), r = num(&s); float t = real(&s); int dtype = num(&s);
    ttf_options o = options(&s);
    for (int q = 1; q < 4; ++q) lists[q] = next_arg(&s);
    ttf_stream_t st = ptr(&s);
    if (!done(&s)) return NULL;
    Py_ssize_t B = PyList_Check(lists[0]) ? PyList_GET_SIZE(lists[0]) : -1;
    for (int q = 0; q < 4; ++q)
        if (!PyList_Check(lists[q]) || PyList_GET_SIZE(lists[q]) != B || B < 1 || B > 0x7fffffff) {
            PyErr_SetString(PyExc_ValueError, "four lists of one length");
            return NULL;
        }
    void** p = PyMem_Malloc(sizeof(void*) * 4 * (size_t)B);
    if (!p) return PyErr_NoMemory();
    for (int q = 0; q < 4; ++q)
        for (Py_ssize_t i = 0; i < B; ++i) {
            p[q * B + i] = PyLong_AsVoidPtr(PyList_GET_ITEM(lists[q], i));
            if (!p[q * B + i] && PyErr_Occurred()) { PyMem_Free(p); return NULL; }
        }
    int rc;
    Py_BEGIN_ALLOW_THREADS
    const void* const* x = (const void* const*)p;
    int* const* cnt = (int* const*)(p + 2 * B);
    int* const* pos = (int* const*)(p + 3 * B);
    rc = plain(&o) ? fn.compress_batch(x, (int)B, F, H, W, C, r, t, dtype, p + B, cnt, pos, st)
                   : fn.compress_batch_ex(x, (int)B, F, H, W, C, r, t, dtype, &o, p + B, cnt, pos, st);
    Py_END_ALLOW_THREADS
    PyMem_Free(p);
    return PyLong_FromLong(rc);
}

#define METHOD(name) {#name, (PyCFunction)(void (*)(void))m_##name, METH_FASTCALL, NULL}
static PyMethodDef methods[] = {METHOD(bind), METHOD(compress), METHOD(compress_ws), METHOD(compress_segment),
                                METHOD(compress_batch), METHOD(query), METHOD(query_ws), METHOD(restore), METHOD(stats),
                                {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_marshal", NULL, -1, methods, NULL, NULL, NULL, NULL};
PyMODINIT_FUNC PyInit__marshal(void) { return PyModule_Create(&module); }
