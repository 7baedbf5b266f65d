/* Argument marshalling of the calls an engine makes per request, natively: a Python record costs ctypes about a microsecond
 * to turn into its C struct, which is a quarter of a small call (one 128-token chunk of one head: 5.2 us of host time, 3.3 this way).
 * The functions take the address of the library's entry point first, then the arguments of the kdn.py function.  They know the plain forms
 * (ints, None and c_void_p, lists and tuples, kdn.py's own Chunk) and raise for any other before the library is called: kdn.py then leaves
 * the call to ctypes, which takes more (an object with _as_parameter_, such as a torch stream) and says what is wrong with the rest. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdlib.h>
#include "kdn.h"

static PyObject *s_value, *s_block_table, *s_n_table_blocks, *s_token_offset, *s_chunk, *s_data, *s_bytes, *s_n_tokens, *s_codec, *s_mem,
    *s_base_pos, *s_parts, *s_part_dst_pos, *s_rope_theta, *s_rope_style, *s_c;

static PyObject *chunk_type, *pointer_type;               /* kdn.Chunk, ctypes.c_void_p */

/* o, if it is a list or a tuple (a new reference).  Items are taken with PySequence_GetItem, which looks at the length each time: reading a
 * record's attributes may run code that changes the list. */
static PyObject *plain_sequence(PyObject *o, const char *message)
{
    if (PyList_Check(o) || PyTuple_Check(o)) return Py_NewRef(o);
    PyErr_SetString(PyExc_TypeError, message);
    return NULL;
}

/* An address: an int, None (null) or a ctypes.c_void_p. */
static int as_address(PyObject *o, void **out)
{
    if (o == Py_None) { *out = NULL; return 0; }
    if (PyLong_Check(o)) {
        *out = (void *)(uintptr_t)PyLong_AsUnsignedLongLongMask(o);
        return PyErr_Occurred() ? -1 : 0;
    }
    if (PyIndex_Check(o)) {
        PyObject *i = PyNumber_Index(o);
        if (!i) return -1;
        *out = (void *)(uintptr_t)PyLong_AsUnsignedLongLongMask(i);
        Py_DECREF(i);
        return PyErr_Occurred() ? -1 : 0;
    }
    PyObject *v = (PyObject *)Py_TYPE(o) == pointer_type ? PyObject_GetAttr(o, s_value) : NULL;      /* an int or None */
    if (!v) {
        if (!PyErr_Occurred()) PyErr_SetString(PyExc_TypeError, "an address is an int or a c_void_p");
        return -1;
    }
    const int r = as_address(v, out);
    Py_DECREF(v);
    return r;
}
static int item_address(PyObject *seq, Py_ssize_t i, void **out)
{
    PyObject *o = PySequence_GetItem(seq, i);
    if (!o) return -1;
    const int r = as_address(o, out);
    Py_DECREF(o);
    return r;
}
static int get_address(PyObject *o, PyObject *name, void **out)
{
    PyObject *v = PyObject_GetAttr(o, name);
    if (!v) return -1;
    const int r = as_address(v, out);
    Py_DECREF(v);
    return r;
}
static int get_i64(PyObject *o, PyObject *name, int64_t *out)
{
    PyObject *v = PyObject_GetAttr(o, name);
    if (!v) return -1;
    /* (an int of any size, modulo 2^64, as ctypes has it; anything else with an index as that index) */
    PyObject *i = PyLong_Check(v) ? Py_NewRef(v) : PyNumber_Index(v);
    Py_DECREF(v);
    if (!i) return -1;
    *out = (int64_t)PyLong_AsUnsignedLongLongMask(i);
    Py_DECREF(i);
    return 0;
}
static int get_i32(PyObject *o, PyObject *name, int32_t *out)
{
    int64_t v;
    if (get_i64(o, name, &v)) return -1;
    *out = (int32_t)v;
    return 0;
}
static int get_chunk(PyObject *c, kdn_chunk *out)
{
    int64_t bytes;
    out->reserved = 0;
    /* (a chunk of a class of its own says itself, in c(), what its record is) */
    if ((PyObject *)Py_TYPE(c) != chunk_type && PyObject_HasAttr(c, s_c)) {
        PyErr_SetString(PyExc_TypeError, "not a kdn.Chunk");
        return -1;
    }
    if (get_address(c, s_data, &out->data) || get_i64(c, s_bytes, &bytes) || get_i32(c, s_n_tokens, &out->n_tokens) ||
        get_i32(c, s_codec, &out->codec) || get_i32(c, s_mem, &out->mem) || get_i64(c, s_base_pos, &out->base_pos)) return -1;
    out->bytes = (size_t)bytes;
    return 0;
}
static int get_op(PyObject *o, kdn_xfer_op *out)
{
    void *table;
    out->reserved = 0;
    if (get_address(o, s_block_table, &table) || get_i32(o, s_n_table_blocks, &out->n_table_blocks) ||
        get_i64(o, s_token_offset, &out->token_offset)) return -1;
    out->block_table = (const int32_t *)table;
    PyObject *c = PyObject_GetAttr(o, s_chunk);
    if (!c) return -1;
    const int r = get_chunk(c, &out->chunk);
    Py_DECREF(c);
    return r;
}
static int get_op_at(PyObject *seq, Py_ssize_t i, kdn_xfer_op *out)
{
    PyObject *o = PySequence_GetItem(seq, i);
    if (!o) return -1;
    const int r = get_op(o, out);
    Py_DECREF(o);
    return r;
}

enum { FEW = 16 };                        /* records on the stack */

/* call_xfer(entry, ctx, pool_id, ops, stream, side_stream) -> status */
typedef kdn_status (*xfer_fn)(kdn_ctx *, int, const kdn_xfer_op *, int, void *, void *);
static PyObject *call_xfer(PyObject *self, PyObject *const *a, Py_ssize_t n_args)
{
    (void)self;
    void *fn, *ctx, *stream, *side;
    if (n_args != 6) { PyErr_SetString(PyExc_TypeError, "six arguments"); return NULL; }
    const long pool = PyLong_AsLong(a[2]);
    if ((pool == -1 && PyErr_Occurred()) || as_address(a[0], &fn) || as_address(a[1], &ctx) || as_address(a[4], &stream) || as_address(a[5], &side)) return NULL;
    PyObject *seq = plain_sequence(a[3], "ops is a list or a tuple");
    if (!seq) return NULL;
    const Py_ssize_t n = PySequence_Size(seq);
    kdn_xfer_op few[FEW], *ops = n <= FEW ? few : malloc(sizeof *ops * (size_t)n);
    int bad = 0;
    if (!ops) { PyErr_NoMemory(); bad = 1; }
    for (Py_ssize_t i = 0; !bad && i < n; ++i) bad = get_op_at(seq, i, &ops[i]) != 0;
    kdn_status st = KDN_OK;
    if (!bad) {
        Py_BEGIN_ALLOW_THREADS
        st = ((xfer_fn)fn)((kdn_ctx *)ctx, (int)pool, ops, (int)n, stream, side);
        Py_END_ALLOW_THREADS
    }
    if (ops != few) free(ops);
    Py_DECREF(seq);
    return bad ? NULL : PyLong_FromLong((long)st);
}

/* call_sparse(entry, ctx, pool_id, ops, keeps, stream, side_stream) -> status */
typedef kdn_status (*sparse_fn)(kdn_ctx *, int, const kdn_sparse_op *, int, void *, void *);
static PyObject *call_sparse(PyObject *self, PyObject *const *a, Py_ssize_t n_args)
{
    (void)self;
    void *fn, *ctx, *stream, *side;
    if (n_args != 7) { PyErr_SetString(PyExc_TypeError, "seven arguments"); return NULL; }
    const long pool = PyLong_AsLong(a[2]);
    if ((pool == -1 && PyErr_Occurred()) || as_address(a[0], &fn) || as_address(a[1], &ctx) || as_address(a[5], &stream) || as_address(a[6], &side)) return NULL;
    PyObject *seq = plain_sequence(a[3], "ops is a list or a tuple"), *keeps = seq ? plain_sequence(a[4], "keeps is a list or a tuple") : NULL;
    if (!keeps) { Py_XDECREF(seq); return NULL; }
    const Py_ssize_t n = PySequence_Size(seq);
    kdn_sparse_op few[FEW], *ops = n <= FEW ? few : malloc(sizeof *ops * (size_t)n);
    int bad = 0;
    if (!ops) { PyErr_NoMemory(); bad = 1; }
    if (PySequence_Size(keeps) != n) { PyErr_SetString(PyExc_ValueError, "keeps have to have an entry per op"); bad = 1; }
    for (Py_ssize_t i = 0; !bad && i < n; ++i) {
        void *keep = NULL;
        bad = get_op_at(seq, i, &ops[i].op) != 0 || item_address(keeps, i, &keep) != 0;
        ops[i].keep = (const int32_t *)keep;
    }
    kdn_status st = KDN_OK;
    if (!bad) {
        Py_BEGIN_ALLOW_THREADS
        st = ((sparse_fn)fn)((kdn_ctx *)ctx, (int)pool, ops, (int)n, stream, side);
        Py_END_ALLOW_THREADS
    }
    if (ops != few) free(ops);
    Py_DECREF(keeps);
    Py_DECREF(seq);
    return bad ? NULL : PyLong_FromLong((long)st);
}

/* call_compose(entry, ctx, pool_id, reqs, stream, side_stream) -> status */
typedef kdn_status (*compose_fn)(kdn_ctx *, int, const kdn_compose_req *, int, void *, void *);
static int get_req(PyObject *q, kdn_compose_req *out, kdn_chunk *parts, int64_t *pos, Py_ssize_t room)
{
    void *table;
    out->reserved = 0;
    if (get_address(q, s_block_table, &table) || get_i32(q, s_n_table_blocks, &out->n_table_blocks) || get_i32(q, s_rope_style, &out->rope_style)) return -1;
    out->block_table = (const int32_t *)table;
    PyObject *theta = PyObject_GetAttr(q, s_rope_theta);
    if (!theta) return -1;
    out->rope_theta = PyFloat_AsDouble(theta);
    Py_DECREF(theta);
    if (out->rope_theta == -1.0 && PyErr_Occurred()) return -1;
    PyObject *po = PyObject_GetAttr(q, s_parts), *do_ = po ? PyObject_GetAttr(q, s_part_dst_pos) : NULL;
    PyObject *ps = do_ ? plain_sequence(po, "parts is a list or a tuple") : NULL, *ds = ps ? plain_sequence(do_, "part_dst_pos is a list or a tuple") : NULL;
    int bad = ds == NULL;
    if (!bad) {
        const Py_ssize_t n = PySequence_Size(ps);
        if (n > room || PySequence_Size(ds) != n) {
            PyErr_SetString(PyExc_ValueError, "parts and part_dst_pos have to be of one length");
            bad = 1;
        }
        for (Py_ssize_t j = 0; !bad && j < n; ++j) {
            PyObject *c = PySequence_GetItem(ps, j), *p = c ? PySequence_GetItem(ds, j) : NULL;
            bad = !p || get_chunk(c, &parts[j]) != 0;
            PyObject *i = bad ? NULL : PyNumber_Long(p);
            if (i) pos[j] = (int64_t)PyLong_AsUnsignedLongLongMask(i); else bad = 1;
            Py_XDECREF(i); Py_XDECREF(p); Py_XDECREF(c);
        }
        out->n_parts = (int32_t)n;
        out->parts = parts;
        out->part_dst_pos = pos;
    }
    Py_XDECREF(ds); Py_XDECREF(ps); Py_XDECREF(do_); Py_XDECREF(po);
    return bad ? -1 : 0;
}
/* selects[r]: a sequence with an entry per part of reqs[r], false (every token) or (address, count). */
static int get_select(PyObject *sel, kdn_select *out, const int32_t **ptrs, int32_t *counts, Py_ssize_t parts)
{
    PyObject *seq = plain_sequence(sel, "a request's selects are a list or a tuple");
    if (!seq) return -1;
    int bad = PySequence_Size(seq) != parts;
    if (bad) PyErr_SetString(PyExc_ValueError, "selects have to have an entry per part");
    for (Py_ssize_t j = 0; !bad && j < parts; ++j) {
        PyObject *e = PySequence_GetItem(seq, j);
        const int given = e ? PyObject_IsTrue(e) : -1;
        ptrs[j] = NULL;
        counts[j] = 0;
        if (given <= 0) { bad = given < 0; Py_XDECREF(e); continue; }
        PyObject *address = PySequence_GetItem(e, 0), *count = address ? PySequence_GetItem(e, 1) : NULL;
        void *p = NULL;
        bad = !count || as_address(address, &p) != 0;
        if (!bad) {
            const long long c = PyLong_AsLongLong(count);
            bad = c == -1 && PyErr_Occurred() != NULL;
            ptrs[j] = (const int32_t *)p;
            counts[j] = (int32_t)c;
        }
        Py_XDECREF(count);
        Py_XDECREF(address);
        Py_DECREF(e);
    }
    Py_DECREF(seq);
    out->part_select = ptrs;
    out->part_n_select = counts;
    return bad ? -1 : 0;
}

typedef kdn_status (*select_fn)(kdn_ctx *, int, const kdn_compose_req *, const kdn_select *, int, void *, void *);
static PyObject *compose(PyObject *entry, PyObject *ctx_, PyObject *pool_, PyObject *reqs_, PyObject *selects_, PyObject *stream_, PyObject *side_)
{
    void *fn, *ctx, *stream, *side;
    const long pool = PyLong_AsLong(pool_);
    if ((pool == -1 && PyErr_Occurred()) || as_address(entry, &fn) || as_address(ctx_, &ctx) || as_address(stream_, &stream) || as_address(side_, &side)) return NULL;
    PyObject *seq = plain_sequence(reqs_, "reqs is a list or a tuple");
    if (!seq) return NULL;
    PyObject *sels = selects_ ? plain_sequence(selects_, "selects is a list or a tuple") : NULL;
    if (selects_ && !sels) { Py_DECREF(seq); return NULL; }
    const Py_ssize_t n = PySequence_Size(seq);
    Py_ssize_t total = 0;
    int bad = 0;
    if (sels && PySequence_Size(sels) != n) {
        PyErr_SetString(PyExc_ValueError, "selects have to have an entry per request");
        bad = 1;
    }
    for (Py_ssize_t i = 0; !bad && i < n; ++i) {
        PyObject *q = PySequence_GetItem(seq, i), *p = q ? PyObject_GetAttr(q, s_parts) : NULL;
        const Py_ssize_t k = p ? PySequence_Size(p) : -1;
        Py_XDECREF(p);
        Py_XDECREF(q);
        if (k < 0) bad = 1; else total += k;
    }
    kdn_compose_req few[FEW], *reqs = n <= FEW ? few : malloc(sizeof *reqs * (size_t)n);
    kdn_chunk few_parts[FEW], *parts = total <= FEW ? few_parts : malloc(sizeof *parts * (size_t)total);
    int64_t few_pos[FEW], *pos = total <= FEW ? few_pos : malloc(sizeof *pos * (size_t)total);
    kdn_select few_sel[FEW], *sel = n <= FEW ? few_sel : malloc(sizeof *sel * (size_t)n);
    const int32_t *few_ptr[FEW], **ptr = total <= FEW ? few_ptr : malloc(sizeof *ptr * (size_t)total);
    int32_t few_cnt[FEW], *cnt = total <= FEW ? few_cnt : malloc(sizeof *cnt * (size_t)total);
    if (!bad && (!reqs || !parts || !pos || !sel || !ptr || !cnt)) { PyErr_NoMemory(); bad = 1; }
    Py_ssize_t used = 0;
    for (Py_ssize_t i = 0; !bad && i < n; ++i) {
        PyObject *q = PySequence_GetItem(seq, i), *e = q && sels ? PySequence_GetItem(sels, i) : NULL;
        bad = !q || (sels && !e) || get_req(q, &reqs[i], parts + used, pos + used, total - used) != 0;
        if (!bad && sels) bad = get_select(e, &sel[i], ptr + used, cnt + used, reqs[i].n_parts) != 0;
        if (!bad) used += reqs[i].n_parts;
        Py_XDECREF(e);
        Py_XDECREF(q);
    }
    kdn_status st = KDN_OK;
    if (!bad) {
        Py_BEGIN_ALLOW_THREADS
        st = sels ? ((select_fn)fn)((kdn_ctx *)ctx, (int)pool, reqs, sel, (int)n, stream, side) : ((compose_fn)fn)((kdn_ctx *)ctx, (int)pool, reqs, (int)n, stream, side);
        Py_END_ALLOW_THREADS
    }
    if (cnt != few_cnt) free(cnt);
    if (ptr != few_ptr) free(ptr);
    if (sel != few_sel) free(sel);
    if (pos != few_pos) free(pos);
    if (parts != few_parts) free(parts);
    if (reqs != few) free(reqs);
    Py_XDECREF(sels);
    Py_DECREF(seq);
    return bad ? NULL : PyLong_FromLong((long)st);
}
/* call_compose(entry, ctx, pool_id, reqs, stream, side_stream) -> status */
static PyObject *call_compose(PyObject *self, PyObject *const *a, Py_ssize_t n_args)
{
    (void)self;
    if (n_args != 6) { PyErr_SetString(PyExc_TypeError, "six arguments"); return NULL; }
    return compose(a[0], a[1], a[2], a[3], NULL, a[4], a[5]);
}
/* call_compose_select(entry, ctx, pool_id, reqs, selects, stream, side_stream) -> status */
static PyObject *call_compose_select(PyObject *self, PyObject *const *a, Py_ssize_t n_args)
{
    (void)self;
    if (n_args != 7) { PyErr_SetString(PyExc_TypeError, "seven arguments"); return NULL; }
    return compose(a[0], a[1], a[2], a[3], a[4], a[5], a[6]);
}

/* set_types(Chunk, c_void_p): the classes whose instances need no look at what they are. */
static PyObject *set_types(PyObject *self, PyObject *const *a, Py_ssize_t n_args)
{
    (void)self;
    if (n_args != 2) { PyErr_SetString(PyExc_TypeError, "two arguments"); return NULL; }
    Py_XSETREF(chunk_type, Py_NewRef(a[0]));
    Py_XSETREF(pointer_type, Py_NewRef(a[1]));
    Py_RETURN_NONE;
}

static PyMethodDef methods[] = {
    { "set_types", (PyCFunction)(void (*)(void))set_types, METH_FASTCALL, "set_types(Chunk, c_void_p)" },
    { "call_xfer", (PyCFunction)(void (*)(void))call_xfer, METH_FASTCALL, "call_xfer(entry, ctx, pool_id, ops, stream, side_stream) -> status" },
    { "call_sparse", (PyCFunction)(void (*)(void))call_sparse, METH_FASTCALL, "call_sparse(entry, ctx, pool_id, ops, keeps, stream, side_stream) -> status" },
    { "call_compose", (PyCFunction)(void (*)(void))call_compose, METH_FASTCALL, "call_compose(entry, ctx, pool_id, reqs, stream, side_stream) -> status" },
    { "call_compose_select", (PyCFunction)(void (*)(void))call_compose_select, METH_FASTCALL,
      "call_compose_select(entry, ctx, pool_id, reqs, selects, stream, side_stream) -> status" },
    { NULL, NULL, 0, NULL }
};
static struct PyModuleDef module = { PyModuleDef_HEAD_INIT, "_kdn_native", "Native argument marshalling for kdn.py.", -1, methods, NULL, NULL, NULL, NULL };

PyMODINIT_FUNC PyInit__kdn_native(void)
{
    struct { PyObject **to; const char *text; } names[] = {
        { &s_value, "value" }, { &s_block_table, "block_table" }, { &s_n_table_blocks, "n_table_blocks" }, { &s_token_offset, "token_offset" },
        { &s_chunk, "chunk" }, { &s_data, "data" }, { &s_bytes, "bytes" }, { &s_n_tokens, "n_tokens" }, { &s_codec, "codec" }, { &s_mem, "mem" },
        { &s_base_pos, "base_pos" }, { &s_parts, "parts" }, { &s_part_dst_pos, "part_dst_pos" }, { &s_rope_theta, "rope_theta" }, { &s_rope_style, "rope_style" }, { &s_c, "c" } };
    for (size_t i = 0; i < sizeof names / sizeof *names; ++i)
        if (!(*names[i].to = PyUnicode_InternFromString(names[i].text))) return NULL;
    PyObject *m = PyModule_Create(&module);
    if (m && PyModule_AddStringConstant(m, "stamp", KDN_STAMP)) { Py_DECREF(m); return NULL; }      /* (build.py looks for it in the file) */
    return m;
}
