/*
 * Argument marshalling of the Python binding's hot calls, as a CPython extension
 * (paper_2506_07416_gb300/_fastcall.so). Each function takes the arguments of the
 * C function of the same name (include/litevlm_select.h) as Python objects:
 * pointers as integers, numpy arrays or objects with data_ptr() (torch tensors),
 * host offset arrays as int32 numpy arrays (anything else goes through the binding's
 * own conversion), handles and numbers as ctypes takes them, and returns the status
 * code. No other object is a pointer, whatever memory it may show: the address of a
 * numpy scalar or of a bytes object is not the value it holds. The GIL is
 * released around the call. The C functions' addresses come from the library that
 * the binding loaded (bind).
 *
 * Why: with ctypes, a call's 12 to 18 argument conversions and numpy's ctypes
 * attribute took 15 to 20 us of a single-request step that needs 13 us of GPU time.
 */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>

enum { F_SCORE, F_FULL, F_SCORE_TOPK, F_TOPK, F_COMPACT, F_SPLICE, F_PROJECT, F_KEEP, F_COUNT };
static const char *const kNames[F_COUNT] = {"score", "score_full_keys", "score_topk", "topk",
                                            "compact", "splice", "project", "keep_offsets"};
/* h handle / stream, i int32, l int64, f float, p pointer, n host int32 array */
static const char *const kSigs[F_COUNT] = {"hippnppnffph", "hippnppnppnpffph", "hippnppnffppnfppph", "hippnpnfppph",
                                           "", "hippnppnppnppnlpppph", "hliipppfippifph", ""};
static void *g_fn[F_COUNT];
static PyObject *g_host_i32;      /* the binding's conversion of a host offset array */
static PyObject *g_ndarray;       /* numpy.ndarray */
static PyObject *g_ctypes_value;  /* the value of a ctypes object of a signature's kind */
static PyObject *g_data_ptr;      /* "data_ptr" */

#define MAX_ARGS 24
typedef struct {
    Py_buffer buf[MAX_ARGS];
    PyObject *obj[MAX_ARGS];
    int nbuf, nobj;
} Held;

static void release(Held *h)
{
    while (h->nbuf > 0) PyBuffer_Release(&h->buf[--h->nbuf]);
    while (h->nobj > 0) Py_DECREF(h->obj[--h->nobj]);
}

static int as_ptr(PyObject *o, Held *h, void **out)
{
    if (o == Py_None) {
        *out = NULL;
        return 0;
    }
    if (PyLong_Check(o)) {
        *out = (void *)(uintptr_t)PyLong_AsUnsignedLongLongMask(o);
        return PyErr_Occurred() ? -1 : 0;
    }
    if (PyObject_TypeCheck(o, (PyTypeObject *)g_ndarray)) {
        Py_buffer *b = &h->buf[h->nbuf];
        if (PyObject_GetBuffer(o, b, PyBUF_STRIDED_RO) == 0) {
            ++h->nbuf;
            *out = b->buf;
            return 0;
        }
        PyErr_Clear(); /* a type without a buffer format */
        PyObject *c = PyObject_GetAttrString(o, "ctypes");
        PyObject *d = c ? PyObject_GetAttrString(c, "data") : NULL;
        Py_XDECREF(c);
        if (!d) return -1;
        *out = (void *)(uintptr_t)PyLong_AsUnsignedLongLongMask(d);
        Py_DECREF(d);
        return PyErr_Occurred() ? -1 : 0;
    }
    PyObject *r = PyObject_CallMethodNoArgs(o, g_data_ptr);
    if (!r) return -1;
    *out = (void *)(uintptr_t)PyLong_AsUnsignedLongLongMask(r);
    Py_DECREF(r);
    return PyErr_Occurred() ? -1 : 0;
}

/* a handle, a stream or a whole number: an int, an object with __index__ (not for
 * handles), or the ctypes object of its kind; longer ones are cut to 64 bits */
static int as_bits(PyObject *o, char kind, uint64_t *out)
{
    PyObject *v;
    if (kind == 'h' && o == Py_None) {
        *out = 0;
        return 0;
    }
    if (PyLong_Check(o)) v = Py_NewRef(o);
    else if (kind != 'h' && PyIndex_Check(o)) v = PyNumber_Index(o);
    else v = PyObject_CallFunction(g_ctypes_value, "OC", o, kind);
    if (!v) return -1;
    *out = (uint64_t)PyLong_AsUnsignedLongLongMask(v);
    Py_DECREF(v);
    return PyErr_Occurred() ? -1 : 0;
}

static int as_double(PyObject *o, double *out)
{
    *out = PyFloat_AsDouble(o);
    if (*out != -1.0 || !PyErr_Occurred()) return 0;
    PyErr_Clear();
    PyObject *v = PyObject_CallFunction(g_ctypes_value, "OC", o, 'f');
    if (!v) return -1;
    *out = PyFloat_AsDouble(v);
    Py_DECREF(v);
    return PyErr_Occurred() ? -1 : 0;
}

static int as_host_i32(PyObject *o, Held *h, const int32_t **out, Py_ssize_t *len)
{
    *out = NULL;
    if (len) *len = 0;
    if (o == Py_None) return 0;
    for (int tries = 0; tries < 2; ++tries) {
        if (PyObject_CheckBuffer(o)) {
            Py_buffer *b = &h->buf[h->nbuf];
            if (PyObject_GetBuffer(o, b, PyBUF_C_CONTIGUOUS | PyBUF_FORMAT) == 0) {
                if (b->itemsize == 4 && b->format && b->format[0] == 'i' && !b->format[1]) {
                    ++h->nbuf;
                    *out = (const int32_t *)b->buf;
                    if (len) *len = b->len / 4;
                    return 0;
                }
                PyBuffer_Release(b);
            } else {
                PyErr_Clear();
            }
        }
        if (tries == 1) break;
        o = PyObject_CallOneArg(g_host_i32, o);
        if (!o) return -1;
        h->obj[h->nobj++] = o;
    }
    PyErr_SetString(PyExc_TypeError, "a host offset array is not an int32 array");
    return -1;
}

typedef union {
    void *p;
    int32_t i;
    int64_t l;
    float f;
} Arg;

static int convert(const char *sig, PyObject *const *args, Py_ssize_t n, Held *h, Arg *a)
{
    Py_ssize_t k = 0;
    for (; sig[k]; ++k) {
        if (k >= n) break;
        PyObject *o = args[k];
        switch (sig[k]) {
        case 'p':
            if (as_ptr(o, h, &a[k].p) != 0) return -1;
            break;
        case 'n': {
            const int32_t *q;
            if (as_host_i32(o, h, &q, NULL) != 0) return -1;
            a[k].p = (void *)q;
            break;
        }
        case 'h':
        case 'i':
        case 'l': {
            uint64_t v;
            if (as_bits(o, sig[k], &v) != 0) return -1;
            if (sig[k] == 'i') a[k].i = (int32_t)(uint32_t)v;
            else if (sig[k] == 'l') a[k].l = (int64_t)v;
            else a[k].p = (void *)(uintptr_t)v;
            break;
        }
        default: {
            double v;
            if (as_double(o, &v) != 0) return -1;
            a[k].f = (float)v;
        }
        }
    }
    if (sig[k] || k != n) {
        PyErr_SetString(PyExc_TypeError, "wrong number of arguments");
        return -1;
    }
    return 0;
}

typedef void *P;
typedef int32_t I;

#define BEGIN(which)                                                                    \
    (void)self;                                                                         \
    Held h;                                                                             \
    h.nbuf = h.nobj = 0;                                                                \
    Arg a[MAX_ARGS];                                                                    \
    int rc = 0;                                                                         \
    if (convert(kSigs[which], args, n, &h, a) != 0) {                                   \
        release(&h);                                                                    \
        return NULL;                                                                    \
    }                                                                                   \
    Py_BEGIN_ALLOW_THREADS
#define END                                                                             \
    Py_END_ALLOW_THREADS                                                                \
    release(&h);                                                                        \
    return PyLong_FromLong(rc);

static PyObject *f_score(PyObject *self, PyObject *const *args, Py_ssize_t n)
{
    BEGIN(F_SCORE)
    rc = ((int (*)(P, I, P, P, P, P, P, P, float, float, P, P))g_fn[F_SCORE])(
        a[0].p, a[1].i, a[2].p, a[3].p, a[4].p, a[5].p, a[6].p, a[7].p, a[8].f, a[9].f, a[10].p, a[11].p);
    END
}

static PyObject *f_full(PyObject *self, PyObject *const *args, Py_ssize_t n)
{
    BEGIN(F_FULL)
    rc = ((int (*)(P, I, P, P, P, P, P, P, P, P, P, P, float, float, P, P))g_fn[F_FULL])(
        a[0].p, a[1].i, a[2].p, a[3].p, a[4].p, a[5].p, a[6].p, a[7].p, a[8].p, a[9].p, a[10].p, a[11].p, a[12].f,
        a[13].f, a[14].p, a[15].p);
    END
}

static PyObject *f_score_topk(PyObject *self, PyObject *const *args, Py_ssize_t n)
{
    BEGIN(F_SCORE_TOPK)
    rc = ((int (*)(P, I, P, P, P, P, P, P, float, float, P, P, P, float, P, P, P, P))g_fn[F_SCORE_TOPK])(
        a[0].p, a[1].i, a[2].p, a[3].p, a[4].p, a[5].p, a[6].p, a[7].p, a[8].f, a[9].f, a[10].p, a[11].p, a[12].p,
        a[13].f, a[14].p, a[15].p, a[16].p, a[17].p);
    END
}

static PyObject *f_topk(PyObject *self, PyObject *const *args, Py_ssize_t n)
{
    BEGIN(F_TOPK)
    rc = ((int (*)(P, I, P, P, P, P, P, float, P, P, P, P))g_fn[F_TOPK])(
        a[0].p, a[1].i, a[2].p, a[3].p, a[4].p, a[5].p, a[6].p, a[7].f, a[8].p, a[9].p, a[10].p, a[11].p);
    END
}

static PyObject *f_splice(PyObject *self, PyObject *const *args, Py_ssize_t n)
{
    BEGIN(F_SPLICE)
    rc = ((int (*)(P, I, P, P, P, P, P, P, P, P, P, P, P, P, int64_t, P, P, P, P, P))g_fn[F_SPLICE])(
        a[0].p, a[1].i, a[2].p, a[3].p, a[4].p, a[5].p, a[6].p, a[7].p, a[8].p, a[9].p, a[10].p, a[11].p, a[12].p,
        a[13].p, a[14].l, a[15].p, a[16].p, a[17].p, a[18].p, a[19].p);
    END
}

static PyObject *f_project(PyObject *self, PyObject *const *args, Py_ssize_t n)
{
    BEGIN(F_PROJECT)
    rc = ((int (*)(P, int64_t, I, I, P, P, P, float, I, P, P, I, float, P, P))g_fn[F_PROJECT])(
        a[0].p, a[1].l, a[2].i, a[3].i, a[4].p, a[5].p, a[6].p, a[7].f, a[8].i, a[9].p, a[10].p, a[11].i, a[12].f,
        a[13].p, a[14].p);
    END
}

/* compact(handle, total_kept, kept_idx, src_rows, srcs, dsts, row_bytes, stream): the three are lists */
static PyObject *f_compact(PyObject *self, PyObject *const *args, Py_ssize_t n)
{
    (void)self;
    if (n != 8 || !PyList_Check(args[4]) || !PyList_Check(args[5]) || !PyList_Check(args[6])) {
        PyErr_SetString(PyExc_TypeError, "compact takes eight arguments, three of them lists");
        return NULL;
    }
    const Py_ssize_t t = PyList_GET_SIZE(args[4]);
    if (t > 8 || PyList_GET_SIZE(args[5]) < t || PyList_GET_SIZE(args[6]) < t) {
        PyErr_SetString(PyExc_ValueError, "one destination and row size per source, at most 8");
        return NULL;
    }
    Held h;
    h.nbuf = h.nobj = 0;
    void *kept, *src[8], *dst[8];
    uint64_t hd, stream, total, rows, size;
    int64_t rb[8];
    int bad = as_bits(args[0], 'h', &hd) || as_bits(args[1], 'l', &total) || as_ptr(args[2], &h, &kept) ||
              as_bits(args[3], 'l', &rows) || as_bits(args[7], 'h', &stream);
    for (Py_ssize_t k = 0; k < t && !bad; ++k) {
        bad = as_ptr(PyList_GET_ITEM(args[4], k), &h, &src[k]) || as_ptr(PyList_GET_ITEM(args[5], k), &h, &dst[k]) ||
              as_bits(PyList_GET_ITEM(args[6], k), 'l', &size);
        if (!bad) rb[k] = (int64_t)size;
    }
    if (bad) {
        release(&h);
        return NULL;
    }
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = ((int (*)(P, int64_t, P, int64_t, I, P, P, P, P))g_fn[F_COMPACT])(
        (P)(uintptr_t)hd, (int64_t)total, kept, (int64_t)rows, (I)t, src, dst, rb, (P)(uintptr_t)stream);
    Py_END_ALLOW_THREADS
    release(&h);
    return PyLong_FromLong(rc);
}

/* keep_total(seq_offsets_h, keep_k_h or None, keep_ratio): the batch's kept tokens, or -status */
static PyObject *f_keep_total(PyObject *self, PyObject *const *args, Py_ssize_t n)
{
    (void)self;
    if (n != 3) {
        PyErr_SetString(PyExc_TypeError, "keep_total takes three arguments");
        return NULL;
    }
    Held h;
    h.nbuf = h.nobj = 0;
    const int32_t *so, *kk;
    Py_ssize_t len = 0;
    double ratio;
    if (as_double(args[2], &ratio) != 0 || as_host_i32(args[0], &h, &so, &len) != 0 ||
        as_host_i32(args[1], &h, &kk, NULL) != 0) {
        release(&h);
        return NULL;
    }
    int32_t small[65];
    int32_t *off = len <= 65 ? small : (int32_t *)PyMem_Malloc(sizeof(int32_t) * (size_t)len);
    if (!off) {
        release(&h);
        return PyErr_NoMemory();
    }
    const int rc = ((int (*)(I, const int32_t *, const int32_t *, float, int32_t *))g_fn[F_KEEP])((I)(len - 1), so, kk,
                                                                                             (float)ratio, off);
    const long total = rc ? -(long)rc : (long)off[len - 1];
    if (off != small) PyMem_Free(off);
    release(&h);
    return PyLong_FromLong(total);
}

/* bind({name: address}, host_i32, numpy.ndarray, ctypes_value) */
static PyObject *f_bind(PyObject *self, PyObject *const *args, Py_ssize_t n)
{
    (void)self;
    if (n != 4 || !PyDict_Check(args[0]) || !PyCallable_Check(args[1]) || !PyType_Check(args[2]) ||
        !PyCallable_Check(args[3])) {
        PyErr_SetString(PyExc_TypeError, "bind takes a dict of addresses, a callable, a type and a callable");
        return NULL;
    }
    for (int k = 0; k < F_COUNT; ++k) {
        PyObject *v = PyDict_GetItemString(args[0], kNames[k]);
        if (!v) {
            PyErr_Format(PyExc_KeyError, "%s", kNames[k]);
            return NULL;
        }
        g_fn[k] = PyLong_AsVoidPtr(v);
        if (PyErr_Occurred()) return NULL;
    }
    Py_INCREF(args[1]);
    Py_XSETREF(g_host_i32, args[1]);
    Py_INCREF(args[2]);
    Py_XSETREF(g_ndarray, args[2]);
    Py_INCREF(args[3]);
    Py_XSETREF(g_ctypes_value, args[3]);
    Py_RETURN_NONE;
}

#define DEF(name, fn) {name, (PyCFunction)(void (*)(void))fn, METH_FASTCALL, NULL}
static PyMethodDef kMethods[] = {DEF("bind", f_bind), DEF("score", f_score), DEF("score_full_keys", f_full),
                                 DEF("score_topk", f_score_topk), DEF("topk", f_topk), DEF("compact", f_compact),
                                 DEF("splice", f_splice), DEF("project", f_project),
                                 DEF("keep_total", f_keep_total), {NULL, NULL, 0, NULL}};
static struct PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "_fastcall", NULL, -1, kMethods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__fastcall(void)
{
    g_data_ptr = PyUnicode_InternFromString("data_ptr");
    return g_data_ptr ? PyModule_Create(&kModule) : NULL;
}
