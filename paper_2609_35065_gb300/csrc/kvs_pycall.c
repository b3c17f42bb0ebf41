/* kvs_pycall.c -- argument marshalling of the Python binding, as a CPython extension.
 *
 * Turns the binding's arguments (a geometry, plane addresses, RequestArg / ChunkArg
 * objects) into the C ABI's structs and calls one of its functions by address, with
 * the interpreter lock released.  It takes the ordinary forms only -- exact ints in
 * range, lists and tuples, objects with data_ptr(), contiguous int32 block tables --
 * and returns None, without calling, for anything else: the binding then builds the
 * arguments with numpy, which accepts or refuses them as it always has.
 *
 * What it replaces cost 10 to 16 us for one chunk and 80 us for 128, most of a small
 * call; this takes about 1 us and 25 us.
 */
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <stdint.h>
#include <stdlib.h>
#include <string.h>

#include "kvs.h"

static PyObject *s_data_ptr, *s_block_table, *s_chunks, *s_first_token, *s_num_tokens, *s_base, *s_residency;

/* 1: *out is the exact int `o`, in [lo, hi]; 0: something else. */
static int small_int(PyObject* o, int64_t lo, int64_t hi, int64_t* out) {
    if (!o || !PyLong_CheckExact(o)) return 0;
    int overflow = 0;
    const long long v = PyLong_AsLongLongAndOverflow(o, &overflow);
    if (overflow || v < lo || v > hi) return 0;
    *out = v;
    return 1;
}

/* An address: an exact int, or an object whose data_ptr() returns one.  1 / 0, or -1 with an exception
 * that data_ptr() raised. */
static int address(PyObject* o, uint64_t* out) {
    if (PyLong_CheckExact(o)) {
        const unsigned long long v = PyLong_AsUnsignedLongLong(o);
        if (v == (unsigned long long)-1 && PyErr_Occurred()) {
            PyErr_Clear();
            return 0;
        }
        *out = v;
        return 1;
    }
    PyObject* f = PyObject_GetAttr(o, s_data_ptr);
    if (!f) {
        PyErr_Clear();
        return 0;
    }
    PyObject* r = PyObject_CallNoArgs(f);
    Py_DECREF(f);
    if (!r) return -1;
    int ok = PyLong_CheckExact(r);
    if (ok) {
        *out = PyLong_AsUnsignedLongLong(r);
        if (PyErr_Occurred()) {
            PyErr_Clear();
            ok = 0;
        }
    }
    Py_DECREF(r);
    return ok;
}

static int is_seq(PyObject* o) { return PyList_CheckExact(o) || PyTuple_CheckExact(o); }

typedef struct {
    kvs_geometry    geom;
    kvs_paged_cache cache;
    void**          planes;
    kvs_chunk*      chunks;
    kvs_request*    reqs;
    Py_buffer*      tables;
    Py_ssize_t      nreq, nchunk, chunk_cap, nviews;
    void **         ready, **events;
} Args;

static void drop(Args* a) {
    for (Py_ssize_t r = 0; r < a->nviews; ++r) PyBuffer_Release(&a->tables[r]);
    free(a->planes);
    free(a->chunks);
    free(a->reqs);
    free(a->tables);
    free(a->ready);
    free(a->events);
}

static int read_geometry(PyObject* o, kvs_geometry* g) {
    if (PyTuple_CheckExact(o)) {
        int32_t* f[6] = {&g->num_layers, &g->num_kv_heads, &g->head_dim, &g->elem_bytes, &g->block_size, &g->chunk_tokens};
        if (PyTuple_GET_SIZE(o) != 6) return 0;
        for (int k = 0; k < 6; ++k) {
            int64_t v;
            if (!small_int(PyTuple_GET_ITEM(o, k), INT32_MIN, INT32_MAX, &v)) return 0;
            *f[k] = (int32_t)v;
        }
        return 1;
    }
    Py_buffer b;                                             /* a kvs_geometry of the binding */
    if (PyObject_GetBuffer(o, &b, PyBUF_SIMPLE) != 0) {
        PyErr_Clear();
        return 0;
    }
    const int ok = b.len == (Py_ssize_t)sizeof *g;
    if (ok) memcpy(g, b.buf, sizeof *g);
    PyBuffer_Release(&b);
    return ok;
}

/* Attribute `name` of `o`, held in *held until the next call. */
static PyObject* attr(PyObject* o, PyObject* name, PyObject** held) {
    Py_XDECREF(*held);
    *held = PyObject_GetAttr(o, name);
    if (!*held) PyErr_Clear();
    return *held;
}

/* 1, 0 (not an ordinary request), -1 (exception). */
static int read_request(PyObject* o, Args* a, kvs_request* q) {
    PyObject *held = NULL, *list = NULL, *x;
    int rc = 0;
    int64_t v;
    if (!small_int(attr(o, s_first_token, &held), INT64_MIN, INT64_MAX, &v)) goto out;
    q->first_token = v;
    list = PyObject_GetAttr(o, s_chunks);
    if (!list) PyErr_Clear();
    if (!list || !is_seq(list)) goto out;
    const Py_ssize_t n = PySequence_Fast_GET_SIZE(list);
    if (a->nchunk + n > a->chunk_cap) {
        const Py_ssize_t cap = (a->nchunk + n) * 2;
        kvs_chunk* grown = realloc(a->chunks, (size_t)cap * sizeof *grown);
        if (!grown) goto out;
        a->chunks = grown;
        a->chunk_cap = cap;
    }
    int64_t sum = 0;
    for (Py_ssize_t k = 0; k < n; ++k) {
        if (k >= PySequence_Fast_GET_SIZE(list)) goto out;   /* data_ptr() may run code that shortens it */
        PyObject* c = PySequence_Fast_GET_ITEM(list, k);
        kvs_chunk* d = &a->chunks[a->nchunk + k];
        uint64_t base;
        Py_INCREF(c);
        x = attr(c, s_base, &held);
        int got = x ? address(x, &base) : 0;
        if (got == 1 && !small_int(attr(c, s_num_tokens, &held), INT32_MIN, INT32_MAX, &v)) got = 0;
        if (got == 1) {
            d->base = (void*)(uintptr_t)base;
            d->num_tokens = (int32_t)v;
            sum += v;
            if (!small_int(attr(c, s_residency, &held), INT32_MIN, INT32_MAX, &v)) got = 0;
            else d->residency = (int32_t)v;
        }
        Py_DECREF(c);
        if (got != 1) {
            rc = got;
            goto out;
        }
    }
    a->nchunk += n;
    q->num_chunks = (int32_t)n;
    x = attr(o, s_num_tokens, &held);
    if (x == Py_None) q->num_tokens = sum;
    else if (small_int(x, INT64_MIN, INT64_MAX, &v)) q->num_tokens = v;
    else goto out;
    x = attr(o, s_block_table, &held);
    Py_buffer* b = &a->tables[a->nviews];
    if (!x) goto out;
    if (PyObject_GetBuffer(x, b, PyBUF_C_CONTIGUOUS | PyBUF_FORMAT) != 0) {
        PyErr_Clear();
        goto out;
    }
    a->nviews++;
    if (b->itemsize != 4 || !b->format || strcmp(b->format, "i") != 0 || b->len / 4 > INT32_MAX) goto out;
    q->block_table = (const int32_t*)b->buf;
    q->block_table_len = (int32_t)(b->len / 4);
    rc = 1;
out:
    Py_XDECREF(held);
    Py_XDECREF(list);
    return rc;
}

/* A list of event handles, or None; 1 / 0. */
static int read_handles(PyObject* o, void*** out) {
    *out = NULL;
    if (o == Py_None) return 1;
    if (!PyList_CheckExact(o)) return 0;
    const Py_ssize_t n = PyList_GET_SIZE(o);
    *out = calloc(n ? (size_t)n : 1, sizeof **out);
    if (!*out) return 0;
    for (Py_ssize_t k = 0; k < n; ++k) {
        uint64_t h;
        if (!PyLong_CheckExact(PyList_GET_ITEM(o, k)) || address(PyList_GET_ITEM(o, k), &h) != 1) return 0;
        (*out)[k] = (void*)(uintptr_t)h;
    }
    return 1;
}

typedef int (*whole_fn)(const kvs_geometry*, const kvs_paged_cache*, const kvs_request*, int32_t, void*, uint32_t);
typedef int (*layers_fn)(const kvs_geometry*, const kvs_paged_cache*, const kvs_request*, int32_t, int32_t, void* const*,
                         void*, uint32_t);
typedef int (*store_layers_fn)(const kvs_geometry*, const kvs_paged_cache*, const kvs_request*, int32_t, int32_t,
                               void* const*, void* const*, void*, uint32_t);

/* call(function, geometry, planes, num_blocks, requests, stream, flags[, kind, layers_per_step, ready, events])
 * -> the status, or None.  kind 1: a layer-wise retrieval, 2: a layer-wise store-back. */
static PyObject* call(PyObject* self, PyObject* const* v, Py_ssize_t nv) {
    (void)self;
    Args a;
    memset(&a, 0, sizeof a);
    PyObject* result = NULL;
    int64_t fn, nb, stream, flags, kind = 0, lps = 0;
    int got = 0, rc = 0;
    if (nv != 7 && nv != 11) {
        PyErr_SetString(PyExc_TypeError, "call takes 7 or 11 arguments");
        return NULL;
    }
    if (!small_int(v[0], 1, INT64_MAX, &fn) || !read_geometry(v[1], &a.geom) || !is_seq(v[2]) ||
        !small_int(v[3], INT64_MIN, INT64_MAX, &nb) || !is_seq(v[4]) || !small_int(v[5], 0, INT64_MAX, &stream) ||
        !small_int(v[6], 0, UINT32_MAX, &flags))
        goto out;
    if (nv == 11 && (!small_int(v[7], 1, 2, &kind) || !small_int(v[8], INT32_MIN, INT32_MAX, &lps) ||
                     !read_handles(v[9], &a.ready) || !read_handles(v[10], &a.events)))
        goto out;
    const Py_ssize_t np = PySequence_Fast_GET_SIZE(v[2]);
    a.nreq = PySequence_Fast_GET_SIZE(v[4]);
    /* a plane for every layer: the C call reads 2 * num_layers of them */
    if (np == 0 || np < 2 * (Py_ssize_t)a.geom.num_layers || a.nreq > INT32_MAX) goto out;
    a.planes = malloc((size_t)np * sizeof *a.planes);
    a.reqs = calloc((size_t)a.nreq + 1, sizeof *a.reqs);
    a.tables = calloc((size_t)a.nreq + 1, sizeof *a.tables);
    a.chunk_cap = 64;
    a.chunks = malloc((size_t)a.chunk_cap * sizeof *a.chunks);
    if (!a.planes || !a.reqs || !a.tables || !a.chunks) goto out;
    for (Py_ssize_t p = 0; p < np; ++p) {
        uint64_t x;
        if (p >= PySequence_Fast_GET_SIZE(v[2])) goto out;
        PyObject* o = PySequence_Fast_GET_ITEM(v[2], p);
        Py_INCREF(o);
        got = address(o, &x);
        Py_DECREF(o);
        if (got != 1) goto out;
        a.planes[p] = (void*)(uintptr_t)x;
    }
    for (Py_ssize_t r = 0; r < a.nreq; ++r) {
        if (r >= PySequence_Fast_GET_SIZE(v[4])) {
            got = 0;
            goto out;
        }
        PyObject* o = PySequence_Fast_GET_ITEM(v[4], r);
        Py_INCREF(o);
        got = read_request(o, &a, &a.reqs[r]);
        Py_DECREF(o);
        if (got != 1) goto out;
    }
    Py_ssize_t at = 0;                                       /* the chunk array has stopped moving */
    for (Py_ssize_t r = 0; r < a.nreq; ++r) {
        a.reqs[r].chunks = a.chunks + at;
        at += a.reqs[r].num_chunks;
    }
    a.cache.kv_planes = a.planes;
    a.cache.num_blocks = nb;
    got = 1;
    const int32_t n = (int32_t)a.nreq;
    void* s = (void*)(uintptr_t)stream;
    Py_BEGIN_ALLOW_THREADS
    if (kind == 0) rc = ((whole_fn)(uintptr_t)fn)(&a.geom, &a.cache, a.reqs, n, s, (uint32_t)flags);
    else if (kind == 1) rc = ((layers_fn)(uintptr_t)fn)(&a.geom, &a.cache, a.reqs, n, (int32_t)lps, a.events, s, (uint32_t)flags);
    else rc = ((store_layers_fn)(uintptr_t)fn)(&a.geom, &a.cache, a.reqs, n, (int32_t)lps, a.ready, a.events, s, (uint32_t)flags);
    Py_END_ALLOW_THREADS
    result = PyLong_FromLong(rc);
out:
    drop(&a);
    if (result) return result;
    if (got < 0 || PyErr_Occurred()) return NULL;
    Py_RETURN_NONE;
}

static PyMethodDef methods[] = {{"call", (PyCFunction)(void (*)(void))call, METH_FASTCALL, NULL}, {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "kvs_pycall", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit_kvs_pycall(void) {
    s_data_ptr = PyUnicode_InternFromString("data_ptr");
    s_block_table = PyUnicode_InternFromString("block_table");
    s_chunks = PyUnicode_InternFromString("chunks");
    s_first_token = PyUnicode_InternFromString("first_token");
    s_num_tokens = PyUnicode_InternFromString("num_tokens");
    s_base = PyUnicode_InternFromString("base");
    s_residency = PyUnicode_InternFromString("residency");
    return PyModule_Create(&module);
}
