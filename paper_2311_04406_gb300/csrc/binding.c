/* binding.c -- argument marshalling of abi.py in native code.
 *
 * abi.py keeps the general path (ctypes) and every error message.  Each
 * function here takes the same arguments, checks every tensor as abi._sized
 * does (contiguous, at least elements x words x 8 bytes; None and integer
 * addresses pass), calls libmpclinear and returns its status, or returns None
 * without calling it when a check fails or an argument is of a form it does not
 * handle; abi.py then takes the general path, which raises.  Tensors are read
 * through their Python attributes (nbytes, is_contiguous, data_ptr), so nothing
 * here depends on torch, and nothing is kept from one call for the next.  Reading
 * them may run Python code (subclasses, __index__), which may change the caller's
 * lists and dicts: every item is held while it is read, and taken with a look at
 * the list's present length.
 *
 * Why native: a grouped call checks some hundred tensors, and in Python their
 * marshalling took longer than the kernels (a call of 48 uneven layers: 1.4 ms
 * of host time for 1.1 ms of device time).
 */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <dlfcn.h>
#include <stdint.h>
#include <string.h>

#include "mpclinear.h"

typedef __int128 wide;

static PyObject *s_nbytes, *s_contig, *s_dataptr, *s_numel;
static PyObject *share_keys[6], *tag_keys[12], *check_keys[5];

/* entry points, resolved from the library that ctypes has loaded */
static __typeof__(&mpc_linear_share) f_share, f_share_trunc;
static __typeof__(&mpc_linear_tag) f_tag;
static __typeof__(&mpc_tag_check) f_check;
static __typeof__(&mpc_public_product) f_public;
static __typeof__(&mpc_optmac_trunc) f_optmac;
static __typeof__(&mpc_batchrec_mask) f_mask;
static __typeof__(&mpc_lincomb) f_lincomb;
static __typeof__(&mpc_im2col) f_im2col;
static __typeof__(&mpc_transpose) f_transpose;
static __typeof__(&mpc_linear_share_grouped) f_share_grouped;
static __typeof__(&mpc_linear_tag_grouped) f_tag_grouped;
static __typeof__(&mpc_tag_check_grouped) f_check_grouped;
static __typeof__(&mpc_lincomb_grouped) f_lincomb_grouped;

/* 1: *out is the address of `t`; 0: the check failed; -1: a Python error.
 * `need` bytes; unchecked when it does not apply to the call (sized = 0). */
static int addr(PyObject *t, int sized, wide need, uint64_t *out) {
    if (t == NULL || t == Py_None) {
        *out = 0;
        return 1;
    }
    if (PyLong_Check(t)) {
        *out = PyLong_AsUnsignedLongLongMask(t);
        return PyErr_Occurred() ? -1 : 1;
    }
    if (sized) {
        PyObject *n = PyObject_GetAttr(t, s_nbytes);
        if (!n) return -1;
        const long long nb = PyLong_AsLongLong(n);
        Py_DECREF(n);
        if (nb == -1 && PyErr_Occurred()) return -1;
        if ((wide)nb < need) return 0;
        PyObject *c = PyObject_CallMethodNoArgs(t, s_contig);
        if (!c) return -1;
        const int ok = c == Py_True;
        Py_DECREF(c);
        if (!ok) return 0;
    }
    PyObject *p = PyObject_CallMethodNoArgs(t, s_dataptr);   /* 0 for an empty tensor */
    if (!p) return -1;
    *out = PyLong_AsUnsignedLongLongMask(p);
    Py_DECREF(p);
    return PyErr_Occurred() ? -1 : 1;
}

/* a new reference to item i, or NULL without an error when the list has become shorter */
static PyObject *item(PyObject *list, Py_ssize_t i) {
    if (i >= PyList_GET_SIZE(list)) return NULL;
    PyObject *o = PyList_GET_ITEM(list, i);
    Py_INCREF(o);
    return o;
}
/* addr() of item i of a list */
static int item_addr(PyObject *list, Py_ssize_t i, wide need, uint64_t *out) {
    PyObject *o = item(list, i);
    if (!o) return 0;
    const int r = addr(o, 1, need, out);
    Py_DECREF(o);
    return r;
}

static uint64_t *as_words(uint64_t a) { return (uint64_t *)(uintptr_t)a; }
static void *as_ptr(uint64_t a) { return (void *)(uintptr_t)a; }

static int get_layer(PyObject *o, mpc_layer *L) {
    Py_buffer v;
    if (PyObject_GetBuffer(o, &v, PyBUF_SIMPLE) != 0) {
        PyErr_Clear();
        return 0;
    }
    const int ok = v.len == (Py_ssize_t)sizeof(mpc_layer);
    if (ok) memcpy(L, v.buf, sizeof(mpc_layer));
    PyBuffer_Release(&v);
    return ok;
}

/* workspace: an address and its bytes, or a tensor (bytes -1) */
static int get_ws(PyObject *o, PyObject *bytes, uint64_t *p, size_t *n) {
    const long long b = PyLong_AsLongLong(bytes);
    if (b == -1 && PyErr_Occurred()) return -1;
    const int r = addr(o, 0, 0, p);
    if (r != 1) return r;
    if (b >= 0) {
        *n = (size_t)b;
        return 1;
    }
    PyObject *nb = PyObject_GetAttr(o, s_nbytes);
    if (!nb) return -1;
    *n = (size_t)PyLong_AsUnsignedLongLongMask(nb);
    Py_DECREF(nb);
    return 1;
}

#define GIVE_UP(r) do { if ((r) < 0) return NULL; Py_RETURN_NONE; } while (0)
#define ARGS(n) do { if (nargs != (n)) { PyErr_SetString(PyExc_TypeError, "wrong argument count"); return NULL; } } while (0)
#define STREAM(i) as_ptr(PyLong_AsUnsignedLongLongMask(args[i]))
#define CALL(expr) do { int st_; Py_BEGIN_ALLOW_THREADS st_ = (expr); Py_END_ALLOW_THREADS return PyLong_FromLong(st_); } while (0)
#define FASTCALL(name) static PyObject *name(PyObject *self, PyObject *const *args, Py_ssize_t nargs)

/* addresses of args[first ..), element counts in `elems` (-1: not read) */
static int addrs(PyObject *const *args, int n, const int64_t *elems, int words, uint64_t *a) {
    for (int i = 0; i < n; ++i) {
        const int r = addr(args[i], elems[i] >= 0, (wide)elems[i] * words * 8, &a[i]);
        if (r != 1) return r;
    }
    return 1;
}

/* 1: *out is the C int; 0: not an integer of that range (the general path converts or raises) */
static int get_int(PyObject *o, int *out) {
    int over;
    const long v = PyLong_Check(o) ? PyLong_AsLongAndOverflow(o, &over) : 0;
    if (!PyLong_Check(o) || over || v < INT32_MIN || v > INT32_MAX) return 0;
    *out = (int)v;
    return 1;
}

static int sane(const mpc_layer *L) {   /* products below fit 64 bits; other layers take the general path */
    const int64_t lim = (int64_t)1 << 31;
    return L->M >= 0 && L->K >= 0 && L->N >= 0 && L->M <= lim && L->K <= lim && L->N <= lim;
}

static void share_elems(const mpc_layer *L, int64_t *e) {
    e[0] = e[2] = L->M * L->K;
    e[1] = e[3] = L->K * L->N;
    e[4] = e[5] = L->M * L->N;
}

static void tag_elems(const mpc_layer *L, int mode, int64_t *e) {
    const int64_t M = L->M, K = L->K, N = L->N, c = mode != MPC_TAG_FULL;
    const int64_t v[12] = {1, M * K, K * N, M * K, K * N, M * N, c ? M * N : -1, c ? M * N : -1, c ? N : -1,
                           M * N, c ? M : -1, c ? M : -1};
    memcpy(e, v, sizeof(v));
}

/* (layer, E, F, A, B, C, Z, ws, ws_bytes, stream) */
static PyObject *share(__typeof__(f_share) f, PyObject *const *args, Py_ssize_t nargs) {
    ARGS(10);
    mpc_layer L;
    if (!get_layer(args[0], &L) || !sane(&L)) Py_RETURN_NONE;
    int64_t e[6];
    uint64_t a[6], w;
    size_t wb;
    share_elems(&L, e);
    int r = addrs(args + 1, 6, e, L.ring.words, a);
    if (r != 1) GIVE_UP(r);
    if ((r = get_ws(args[7], args[8], &w, &wb)) != 1) GIVE_UP(r);
    void *st = STREAM(9);
    CALL(f(&L, as_words(a[0]), as_words(a[1]), as_words(a[2]), as_words(a[3]), as_words(a[4]), as_words(a[5]), as_ptr(w),
           wb, st));
}

FASTCALL(py_share) { return share(f_share, args, nargs); }
FASTCALL(py_share_trunc) { return share(f_share_trunc, args, nargs); }

/* (layer, mode, the 12 operands in the order of mpc_tag_ptrs, ws, ws_bytes, stream) */
FASTCALL(py_tag) {
    ARGS(17);
    mpc_layer L;
    if (!get_layer(args[0], &L) || !sane(&L)) Py_RETURN_NONE;
    int mode;
    if (!get_int(args[1], &mode)) Py_RETURN_NONE;
    int64_t e[12];
    uint64_t a[12], w;
    size_t wb;
    tag_elems(&L, mode, e);
    int r = addrs(args + 2, 12, e, L.ring.words, a);
    if (r != 1) GIVE_UP(r);
    if ((r = get_ws(args[14], args[15], &w, &wb)) != 1) GIVE_UP(r);
    void *st = STREAM(16);
    CALL(f_tag(&L, mode, as_words(a[0]), as_words(a[1]), as_words(a[2]), as_words(a[3]), as_words(a[4]), as_words(a[5]),
               as_words(a[6]), as_words(a[7]), as_words(a[8]), as_words(a[9]), as_words(a[10]), as_words(a[11]), as_ptr(w),
               wb, st));
}

/* (layer, mode, alpha, chi_hat, opened, tag, cs, ws, ws_bytes, stream) */
FASTCALL(py_check) {
    ARGS(10);
    mpc_layer L;
    if (!get_layer(args[0], &L) || !sane(&L)) Py_RETURN_NONE;
    int mode;
    if (!get_int(args[1], &mode)) Py_RETURN_NONE;
    const int64_t n = mode == MPC_CHECK_COMPACT ? L.M : L.M * L.N;
    uint64_t a[5], w;
    size_t wb;
    const int64_t e[5] = {1, n, n, n, 1};
    for (int i = 0; i < 5; ++i) {
        /* the seeded check's chi_hat is one 64-bit seed word */
        const int seed = i == 1 && mode == MPC_CHECK_BATCHREC_SEEDED;
        const int r = addr(args[2 + i], 1, seed ? 8 : (wide)e[i] * L.ring.words * 8, &a[i]);
        if (r != 1) GIVE_UP(r);
    }
    const int r = get_ws(args[7], args[8], &w, &wb);
    if (r != 1) GIVE_UP(r);
    void *st = STREAM(9);
    CALL(f_check(&L, mode, as_words(a[0]), as_words(a[1]), as_words(a[2]), as_words(a[3]), as_words(a[4]), as_ptr(w), wb,
                 st));
}

/* (layer, E, F, P, ws, ws_bytes, stream) */
FASTCALL(py_public) {
    ARGS(7);
    mpc_layer L;
    if (!get_layer(args[0], &L) || !sane(&L)) Py_RETURN_NONE;
    const int64_t e[3] = {L.M * L.K, L.K * L.N, L.M * L.N};
    uint64_t a[3], w;
    size_t wb;
    int r = addrs(args + 1, 3, e, L.ring.words, a);
    if (r != 1) GIVE_UP(r);
    if ((r = get_ws(args[4], args[5], &w, &wb)) != 1) GIVE_UP(r);
    void *st = STREAM(6);
    CALL(f_public(&L, as_words(a[0]), as_words(a[1]), as_words(a[2]), as_ptr(w), wb, st));
}

/* (layer, f, alpha, Rf, mRf, Dtilde, P, Zf, mZf, stream) */
FASTCALL(py_optmac) {
    ARGS(10);
    mpc_layer L;
    if (!get_layer(args[0], &L) || !sane(&L)) Py_RETURN_NONE;
    int f;
    if (!get_int(args[1], &f)) Py_RETURN_NONE;
    const int64_t n = L.M * L.N, e[7] = {1, n, n, n, n, n, n};
    uint64_t a[7];
    const int r = addrs(args + 2, 7, e, L.ring.words, a);
    if (r != 1) GIVE_UP(r);
    void *st = STREAM(9);
    CALL(f_optmac(&L, f, as_words(a[0]), as_words(a[1]), as_words(a[2]), as_words(a[3]), as_words(a[4]), as_words(a[5]),
                  as_words(a[6]), st));
}

static int get_ints(PyObject *const *args, int n, int64_t *v) {
    for (int i = 0; i < n; ++i) {
        v[i] = PyLong_AsLongLong(args[i]);
        if (v[i] == -1 && PyErr_Occurred()) {
            PyErr_Clear();
            return 0;
        }
    }
    return 1;
}
static int item_int(PyObject *list, Py_ssize_t i, int64_t *v) {
    PyObject *o = item(list, i);
    const int ok = o && get_ints(&o, 1, v);
    Py_XDECREF(o);
    return ok;
}
static mpc_ring ring_of(const int64_t *ks) {
    mpc_ring r = {(int32_t)ks[0], (int32_t)ks[1], (int32_t)((ks[0] + ks[1] + 63) / 64)};
    return r;
}
static int small(const int64_t *v, int n, int64_t lim) {
    for (int i = 0; i < n; ++i)
        if (v[i] < 0 || v[i] > lim) return 0;
    return 1;
}

/* (k, s, rows, cols, 8 operands, stream) */
FASTCALL(py_mask) {
    ARGS(13);
    int64_t v[4];
    if (!get_ints(args, 4, v) || !small(v, 2, 4096) || !small(v + 2, 2, (int64_t)1 << 31)) Py_RETURN_NONE;
    const mpc_ring ring = ring_of(v);
    const int64_t n = v[2] * v[3], e[8] = {n, n, n, n, n, n, n, n};
    uint64_t a[8];
    const int r = addrs(args + 4, 8, e, ring.words, a);
    if (r != 1) GIVE_UP(r);
    void *st = STREAM(12);
    CALL(f_mask(&ring, v[2], v[3], as_words(a[0]), as_words(a[1]), as_words(a[2]), as_words(a[3]), as_words(a[4]),
                as_words(a[5]), as_words(a[6]), as_words(a[7]), st));
}

/* (k, s, rows, cols, src, dst, stream) */
FASTCALL(py_transpose) {
    ARGS(7);
    int64_t v[4];
    if (!get_ints(args, 4, v) || !small(v, 2, 4096) || !small(v + 2, 2, (int64_t)1 << 31)) Py_RETURN_NONE;
    const mpc_ring ring = ring_of(v);
    const int64_t e[2] = {v[2] * v[3], v[2] * v[3]};
    uint64_t a[2];
    const int r = addrs(args + 4, 2, e, ring.words, a);
    if (r != 1) GIVE_UP(r);
    void *st = STREAM(6);
    CALL(f_transpose(&ring, v[2], v[3], as_words(a[0]), as_words(a[1]), st));
}

/* (k, s, batch, channels, height, width, f, pad, stride, src, dst, stream) */
FASTCALL(py_im2col) {
    ARGS(12);
    int64_t v[9];
    if (!get_ints(args, 9, v) || !small(v, 2, 4096) || !small(v + 2, 4, 1 << 24) || !small(v + 6, 3, 64)) Py_RETURN_NONE;
    const int64_t b = v[2], c = v[3], h = v[4], w = v[5], f = v[6], pad = v[7], s = v[8];
    if (f < 1 || pad >= f || s < 1 || h + 2 * pad < f || w + 2 * pad < f) Py_RETURN_NONE;
    const int64_t ho = (h - f + 2 * pad) / s + 1, wo = (w - f + 2 * pad) / s + 1;
    const mpc_ring ring = ring_of(v);
    uint64_t src, dst;
    int r = addr(args[9], 1, (wide)b * c * h * w * ring.words * 8, &src);
    if (r != 1) GIVE_UP(r);
    if ((r = addr(args[10], 1, (wide)b * ho * wo * c * f * f * ring.words * 8, &dst)) != 1) GIVE_UP(r);
    void *st = STREAM(11);
    CALL(f_im2col(&ring, b, c, h, w, (int)f, (int)pad, (int)s, as_words(src), as_words(dst), st));
}

static int64_t numel(PyObject *t) {
    PyObject *n = PyObject_CallMethodNoArgs(t, s_numel);
    if (!n) return -1;
    const int64_t v = PyLong_AsLongLong(n);
    Py_DECREF(n);
    return v;
}

/* (k, s, coefs, ins, out, stream) */
FASTCALL(py_lincomb) {
    ARGS(6);
    int64_t v[2], coef[16];
    if (!get_ints(args, 2, v) || !small(v, 2, 4096) || !PyList_Check(args[2]) || !PyList_Check(args[3])) Py_RETURN_NONE;
    const Py_ssize_t cnt = PyList_GET_SIZE(args[2]);
    if (cnt < 1 || cnt > 16 || PyList_GET_SIZE(args[3]) != cnt || args[4] == Py_None || PyLong_Check(args[4]))
        Py_RETURN_NONE;
    const mpc_ring ring = ring_of(v);
    if (ring.words < 1) Py_RETURN_NONE;
    const int64_t tot = numel(args[4]);
    if (tot < 0) GIVE_UP(PyErr_Occurred() ? -1 : 0);
    const int64_t n = tot / ring.words;
    const uint64_t *in[16];
    uint64_t o;
    for (Py_ssize_t j = 0; j < cnt; ++j) {
        if (!item_int(args[2], j, &coef[j])) Py_RETURN_NONE;
        const int r = item_addr(args[3], j, (wide)n * ring.words * 8, &o);
        if (r != 1) GIVE_UP(r);
        in[j] = as_words(o);
    }
    const int r = addr(args[4], 1, (wide)n * ring.words * 8, &o);
    if (r != 1) GIVE_UP(r);
    void *st = STREAM(5);
    CALL(f_lincomb(&ring, n, (int)cnt, coef, in, as_words(o), st));
}

/* ---- grouped calls ---- */

/* the layers of a list, or NULL */
static mpc_layer *get_layers(PyObject *list, Py_ssize_t n) {
    mpc_layer *L = PyMem_Malloc((size_t)n * sizeof(mpc_layer));
    for (Py_ssize_t i = 0; L && i < n; ++i) {
        PyObject *o = item(list, i);
        const int ok = o && get_layer(o, &L[i]) && sane(&L[i]);
        Py_XDECREF(o);
        if (!ok) {
            PyMem_Free(L);
            return NULL;
        }
    }
    return L;
}

/* addresses of the operands `keys` of one layer's dict */
static int dict_addrs(PyObject *d, PyObject *const *keys, int n, int required, const int64_t *elems, int words, uint64_t *a) {
    if (!PyDict_Check(d)) return 0;
    for (int j = 0; j < n; ++j) {
        PyObject *t = PyDict_GetItemWithError(d, keys[j]);
        if (!t) {
            if (PyErr_Occurred()) return -1;
            if (required) return 0;
        }
        Py_XINCREF(t);
        const int r = addr(t, elems[j] >= 0, (wide)elems[j] * words * 8, &a[j]);
        Py_XDECREF(t);
        if (r != 1) return r;
    }
    return 1;
}

/* kind 0: shares, 1: tags of `mode`, 2: checks; (layers, ptrs, ...) */
static PyObject *grouped(int kind, int mode, PyObject *layers, PyObject *ptrs, PyObject *ws, PyObject *wbytes, void *st) {
    if (!PyList_Check(layers) || !PyList_Check(ptrs)) Py_RETURN_NONE;
    const Py_ssize_t n = PyList_GET_SIZE(layers);
    if (n < 1 || PyList_GET_SIZE(ptrs) != n) Py_RETURN_NONE;
    PyObject *const *keys = kind == 0 ? share_keys : kind == 1 ? tag_keys : check_keys;
    const int nk = kind == 0 ? 6 : kind == 1 ? 12 : 5;
    mpc_layer *L = get_layers(layers, n);
    if (!L) Py_RETURN_NONE;
    uint64_t *a = PyMem_Malloc((size_t)n * nk * 8);
    int r = a ? 1 : 0;
    for (Py_ssize_t i = 0; r == 1 && i < n; ++i) {
        int64_t e[12];
        if (kind == 0) {
            share_elems(&L[i], e);
        } else if (kind == 1) {
            tag_elems(&L[i], mode, e);
        } else {
            e[0] = e[4] = 1;
            e[1] = e[2] = e[3] = L[i].M;
        }
        PyObject *d = item(ptrs, i);
        r = d ? dict_addrs(d, keys, nk, kind == 2, e, L[i].ring.words, a + i * nk) : 0;
        Py_XDECREF(d);
    }
    uint64_t w = 0;
    size_t wb = 0;
    if (r == 1 && kind != 2) r = get_ws(ws, wbytes, &w, &wb);
    int status = 0;
    if (r == 1) {
        Py_BEGIN_ALLOW_THREADS
        /* the pointer structs are arrays of addresses in this order */
        if (kind == 0) status = f_share_grouped(L, (int)n, (const mpc_share_ptrs *)a, as_ptr(w), wb, st);
        else if (kind == 1) status = f_tag_grouped(L, (int)n, mode, (const mpc_tag_ptrs *)a, as_ptr(w), wb, st);
        else status = f_check_grouped(L, (int)n, (const mpc_check_ptrs *)a, st);
        Py_END_ALLOW_THREADS
    }
    PyMem_Free(a);
    PyMem_Free(L);
    if (r != 1) GIVE_UP(r);
    return PyLong_FromLong(status);
}
_Static_assert(sizeof(mpc_share_ptrs) == 6 * 8 && sizeof(mpc_tag_ptrs) == 12 * 8 && sizeof(mpc_check_ptrs) == 5 * 8,
               "pointer structs are arrays of 64-bit addresses");

FASTCALL(py_share_grouped) {
    ARGS(5);
    return grouped(0, 0, args[0], args[1], args[2], args[3], STREAM(4));
}
FASTCALL(py_tag_grouped) {
    ARGS(6);
    int mode;
    if (!get_int(args[1], &mode)) Py_RETURN_NONE;
    return grouped(1, mode, args[0], args[2], args[3], args[4], STREAM(5));
}
FASTCALL(py_check_grouped) {
    ARGS(3);
    return grouped(2, 0, args[0], args[1], NULL, NULL, STREAM(2));
}

/* (k, s, coefs, ins, outs, n or None, stream) */
FASTCALL(py_lincomb_grouped) {
    ARGS(7);
    int64_t v[2], coef[4];
    if (!get_ints(args, 2, v) || !small(v, 2, 4096)) Py_RETURN_NONE;
    if (!PyList_Check(args[2]) || !PyList_Check(args[3]) || !PyList_Check(args[4])) Py_RETURN_NONE;
    const Py_ssize_t cnt = PyList_GET_SIZE(args[2]), G = PyList_GET_SIZE(args[4]);
    if (cnt < 1 || cnt > 4 || G < 1 || PyList_GET_SIZE(args[3]) < G) Py_RETURN_NONE;
    if (args[5] != Py_None && (!PyList_Check(args[5]) || PyList_GET_SIZE(args[5]) != G)) Py_RETURN_NONE;
    const mpc_ring ring = ring_of(v);
    if (ring.words < 1) Py_RETURN_NONE;
    for (Py_ssize_t j = 0; j < cnt; ++j)
        if (!item_int(args[2], j, &coef[j])) Py_RETURN_NONE;
    uint64_t *buf = PyMem_Malloc((size_t)G * (cnt + 2) * 8);   /* ins, outs, sizes */
    if (!buf) Py_RETURN_NONE;
    uint64_t *in = buf, *out = buf + G * cnt;
    int64_t *n = (int64_t *)(out + G);
    int r = 1;
    for (Py_ssize_t g = 0; r == 1 && g < G; ++g) {
        PyObject *o = item(args[4], g), *row = item(args[3], g);
        if (!o || !row) {
            r = 0;
        } else if (args[5] != Py_None) {
            r = item_int(args[5], g, &n[g]);
        } else if (o == Py_None || PyLong_Check(o)) {
            r = 0;
        } else {
            n[g] = numel(o);
            if (n[g] < 0) r = PyErr_Occurred() ? -1 : 0;
            else n[g] /= ring.words;
        }
        if (r == 1 && (!PyList_Check(row) || PyList_GET_SIZE(row) != cnt)) r = 0;
        for (Py_ssize_t j = 0; r == 1 && j < cnt; ++j)
            r = item_addr(row, j, (wide)n[g] * ring.words * 8, &in[g * cnt + j]);
        if (r == 1) r = addr(o, 1, (wide)n[g] * ring.words * 8, &out[g]);
        Py_XDECREF(o);
        Py_XDECREF(row);
    }
    int status = 0;
    void *st = STREAM(6);
    if (r == 1) {
        Py_BEGIN_ALLOW_THREADS
        status = f_lincomb_grouped(&ring, (int)G, n, (int)cnt, coef, (const uint64_t *const *)in, (uint64_t *const *)out, st);
        Py_END_ALLOW_THREADS
    }
    PyMem_Free(buf);
    if (r != 1) GIVE_UP(r);
    return PyLong_FromLong(status);
}

/* open(path): resolve the entry points of the loaded library */
static PyObject *py_open(PyObject *self, PyObject *path) {
    const char *p = PyUnicode_AsUTF8(path);
    if (!p) return NULL;
    void *h = dlopen(p, RTLD_NOW | RTLD_LOCAL);
    if (!h) return PyErr_Format(PyExc_RuntimeError, "cannot open %s: %s", p, dlerror());
#define RESOLVE(var, name) \
    if (!(*(void **)&var = dlsym(h, #name))) return PyErr_Format(PyExc_RuntimeError, "%s lacks %s", p, #name)
    RESOLVE(f_share, mpc_linear_share);
    RESOLVE(f_share_trunc, mpc_linear_share_trunc);
    RESOLVE(f_tag, mpc_linear_tag);
    RESOLVE(f_check, mpc_tag_check);
    RESOLVE(f_public, mpc_public_product);
    RESOLVE(f_optmac, mpc_optmac_trunc);
    RESOLVE(f_mask, mpc_batchrec_mask);
    RESOLVE(f_lincomb, mpc_lincomb);
    RESOLVE(f_im2col, mpc_im2col);
    RESOLVE(f_transpose, mpc_transpose);
    RESOLVE(f_share_grouped, mpc_linear_share_grouped);
    RESOLVE(f_tag_grouped, mpc_linear_tag_grouped);
    RESOLVE(f_check_grouped, mpc_tag_check_grouped);
    RESOLVE(f_lincomb_grouped, mpc_lincomb_grouped);
    Py_RETURN_NONE;
}

#define FC(name, fn) {name, (PyCFunction)(void (*)(void))fn, METH_FASTCALL, NULL}
static PyMethodDef methods[] = {
    {"open", py_open, METH_O, NULL},
    FC("share", py_share), FC("share_trunc", py_share_trunc),
    FC("tag", py_tag), FC("check", py_check),
    FC("public_product", py_public), FC("optmac_trunc", py_optmac), FC("batchrec_mask", py_mask),
    FC("transpose", py_transpose), FC("im2col", py_im2col), FC("lincomb", py_lincomb),
    FC("share_grouped", py_share_grouped), FC("tag_grouped", py_tag_grouped), FC("check_grouped", py_check_grouped),
    FC("lincomb_grouped", py_lincomb_grouped), {NULL, NULL, 0, NULL}};

static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_binding", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__binding(void) {
    static const char *sk[6] = {"E", "F", "A_i", "B_i", "C_i", "Z_i"};
    static const char *tk[12] = {"alpha_i", "E", "F", "mA_i", "mB_i", "mC_i", "mR_i", "Dtilde", "chi", "mZ_i", "mDc_i", "Dc"};
    static const char *ck[5] = {"alpha_i", "chi_hat", "Dc", "mDc_i", "cs_i"};
    for (int i = 0; i < 6; ++i) share_keys[i] = PyUnicode_InternFromString(sk[i]);
    for (int i = 0; i < 12; ++i) tag_keys[i] = PyUnicode_InternFromString(tk[i]);
    for (int i = 0; i < 5; ++i) check_keys[i] = PyUnicode_InternFromString(ck[i]);
    s_nbytes = PyUnicode_InternFromString("nbytes");
    s_contig = PyUnicode_InternFromString("is_contiguous");
    s_dataptr = PyUnicode_InternFromString("data_ptr");
    s_numel = PyUnicode_InternFromString("numel");
    return PyModule_Create(&module);
}
