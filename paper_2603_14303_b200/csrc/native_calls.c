/* CPython entry to the C ABI for the calls a serving loop makes per layer or per token: one METH_FASTCALL function per
 * call, arguments in the order of the header, pointers as integers (None = NULL), the status code returned.  ctypes takes
 * about 4 us to marshal such a call (eighteen arguments), this 0.5 us; the GIL is released meanwhile, as ctypes does. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include "semanticache.h"

static void* ptr(PyObject* o) { return o == Py_None ? NULL : (void*)PyLong_AsUnsignedLongLong(o); }
/* integers modulo 2^32: what ctypes' c_int32 and c_uint32 take */
static uint32_t u32(PyObject* o) { return (uint32_t)PyLong_AsUnsignedLongMask(o); }
static int32_t i32(PyObject* o) { return (int32_t)u32(o); }
static size_t sz(PyObject* o) { return (size_t)PyLong_AsUnsignedLongLong(o); }
static float f32(PyObject* o) { return (float)PyFloat_AsDouble(o); }

static int arity(Py_ssize_t n, Py_ssize_t want, const char* name) {
    if (n == want) return 1;
    PyErr_Format(PyExc_TypeError, "%s takes %zd arguments, got %zd", name, want, n);
    return 0;
}
/* anything that has a length and can be iterated, its items made ints; the length, or -1 with an exception set.  One too many
 * is kept: the library refuses the count. */
static int32_t ids_of(PyObject* seq, int32_t* out) {
    if (PyObject_Size(seq) < 0) return -1;
    PyObject* fast = PySequence_Fast(seq, "delim_ids must be a sequence");
    if (!fast) return -1;
    const Py_ssize_t n = PySequence_Fast_GET_SIZE(fast);
    for (Py_ssize_t i = 0; i < n && i < SC_MAX_DELIMS; ++i) {
        PyObject* v = PyNumber_Long(PySequence_Fast_GET_ITEM(fast, i));
        if (v) { out[i] = i32(v); Py_DECREF(v); }
        if (PyErr_Occurred()) { Py_DECREF(fast); return -1; }
    }
    Py_DECREF(fast);
    return n > SC_MAX_DELIMS ? SC_MAX_DELIMS + 1 : (int32_t)n;
}
#define CALL(expr)                          \
    do {                                    \
        if (PyErr_Occurred()) return NULL;  \
        sc_status code_;                    \
        Py_BEGIN_ALLOW_THREADS              \
        code_ = (expr);                     \
        Py_END_ALLOW_THREADS                \
        return PyLong_FromLong((long)code_);\
    } while (0)

static PyObject* chunk_sizes(PyObject* self, PyObject* const* a, Py_ssize_t n) {   /* B, n -> code, segments, tiles, bytes */
    int32_t segs = 0, tiles = 0;
    (void)self;
    if (!arity(n, 2, "chunk_sizes")) return NULL;
    const int32_t B = i32(a[0]), len = i32(a[1]);
    if (PyErr_Occurred()) return NULL;
    const sc_status code = sc_chunk_bounds(B, len, &segs, &tiles);
    return Py_BuildValue("iiin", (int)code, (int)segs, (int)tiles, (Py_ssize_t)sc_chunk_workspace_bytes(B, len));
}
static PyObject* chunk(PyObject* self, PyObject* const* a, Py_ssize_t n) {   /* delim_ids, n_delim -> one sequence */
    int32_t delims[SC_MAX_DELIMS + 1];
    (void)self;
    if (!arity(n, 16, "chunk")) return NULL;
    const int32_t nd = ids_of(a[3], delims);
    if (nd < 0) return NULL;
    const void* ids = ptr(a[0]);
    const int32_t B = i32(a[1]), len = i32(a[2]), max_len = i32(a[4]), seg_cap = i32(a[6]), tile_cap = i32(a[10]);
    void *seg_off = ptr(a[5]), *seq_off = ptr(a[7]), *n_seg = ptr(a[8]), *tile_seg = ptr(a[9]), *tile_cnt = ptr(a[11]), *ws = ptr(a[12]),
         *status = ptr(a[14]), *stream = ptr(a[15]);
    const size_t bytes = sz(a[13]);
    CALL(sc_chunk(ids, B, len, delims, nd, max_len, seg_off, seg_cap, seq_off, n_seg, tile_seg, tile_cap, tile_cnt, ws, bytes, status, stream));
}
static PyObject* compress(PyObject* self, PyObject* const* a, Py_ssize_t n) {   /* strides and params flattened */
    (void)self;
    if (!arity(n, 28, "compress")) return NULL;
    const void *K = ptr(a[0]), *V = ptr(a[1]);
    const sc_strides st = {PyLong_AsLongLong(a[2]), PyLong_AsLongLong(a[3]), PyLong_AsLongLong(a[4])};
    const sc_dtype dt = (sc_dtype)i32(a[5]);
    const int32_t B = i32(a[6]), H = i32(a[7]), len = i32(a[8]), d = i32(a[9]), tile_cap = i32(a[15]), cap = i32(a[22]);
    const void *seg_off = ptr(a[10]), *seq_off = ptr(a[11]), *n_seg = ptr(a[12]), *tile_seg = ptr(a[13]), *tile_cnt = ptr(a[14]);
    const sc_gsc_params prm = {f32(a[16]), i32(a[17]), u32(a[18])};
    void *core_k = ptr(a[19]), *core_v = ptr(a[20]), *count = ptr(a[21]), *core_len = ptr(a[23]), *assign = ptr(a[24]), *ws = ptr(a[25]);
    const size_t bytes = sz(a[26]);
    PyObject* tail = a[27];   /* (status, stream) */
    if (!PyTuple_Check(tail) || PyTuple_GET_SIZE(tail) != 2) { PyErr_SetString(PyExc_TypeError, "(status, stream) expected"); return NULL; }
    void *status = ptr(PyTuple_GET_ITEM(tail, 0)), *stream = ptr(PyTuple_GET_ITEM(tail, 1));
    CALL(sc_compress(K, V, st, dt, B, H, len, d, seg_off, seq_off, n_seg, tile_seg, tile_cnt, tile_cap, &prm, core_k, core_v, count, cap,
                     core_len, assign, ws, bytes, status, stream));
}
static PyObject* decode_attn(PyObject* self, PyObject* const* a, Py_ssize_t n) {
    (void)self;
    if (!arity(n, 18, "decode_attn")) return NULL;
    const void *q = ptr(a[0]), *core_k = ptr(a[6]), *core_v = ptr(a[7]), *count = ptr(a[8]), *core_len = ptr(a[10]);
    const sc_dtype dt = (sc_dtype)i32(a[1]);
    const int32_t B = i32(a[2]), Hq = i32(a[3]), Hkv = i32(a[4]), d = i32(a[5]), cap = i32(a[9]);
    const float scale = f32(a[11]);
    const uint32_t flags = u32(a[12]);
    void *out = ptr(a[13]), *ws = ptr(a[14]), *status = ptr(a[16]), *stream = ptr(a[17]);
    const size_t bytes = sz(a[15]);
    CALL(sc_decode_attn(q, dt, B, Hq, Hkv, d, core_k, core_v, count, cap, core_len, scale, flags, out, ws, bytes, status, stream));
}
static PyObject* prefill_attn(PyObject* self, PyObject* const* a, Py_ssize_t n) {
    (void)self;
    if (!arity(n, 17, "prefill_attn")) return NULL;
    const void *q = ptr(a[0]), *core_k = ptr(a[7]), *core_v = ptr(a[8]), *count = ptr(a[9]), *core_len = ptr(a[11]);
    const sc_dtype dt = (sc_dtype)i32(a[1]);
    const int32_t B = i32(a[2]), Hq = i32(a[3]), Hkv = i32(a[4]), m = i32(a[5]), d = i32(a[6]), cap = i32(a[10]);
    const float scale = f32(a[12]);
    const uint32_t flags = u32(a[13]);
    void *out = ptr(a[14]), *status = ptr(a[15]), *stream = ptr(a[16]);
    CALL(sc_prefill_attn(q, dt, B, Hq, Hkv, m, d, core_k, core_v, count, cap, core_len, scale, flags, out, status, stream));
}
static PyObject* append(PyObject* self, PyObject* const* a, Py_ssize_t n) {   /* delim_ids, n_delim -> one sequence */
    int32_t delims[SC_MAX_DELIMS + 1];
    (void)self;
    if (!arity(n, 19, "append")) return NULL;
    const int32_t nd = ids_of(a[7], delims);
    if (nd < 0) return NULL;
    const void *k = ptr(a[0]), *v = ptr(a[1]), *ids = ptr(a[6]);
    const sc_dtype dt = (sc_dtype)i32(a[2]);
    const int32_t B = i32(a[3]), H = i32(a[4]), d = i32(a[5]), max_len = i32(a[8]), cap = i32(a[13]);
    const float tau = f32(a[9]);
    void *core_k = ptr(a[10]), *core_v = ptr(a[11]), *count = ptr(a[12]), *core_len = ptr(a[14]), *tail_len = ptr(a[15]),
         *attn_len = ptr(a[16]), *status = ptr(a[17]), *stream = ptr(a[18]);
    CALL(sc_append(k, v, dt, B, H, d, ids, delims, nd, max_len, tau, core_k, core_v, count, cap, core_len, tail_len, attn_len, status, stream));
}
static PyObject* append_layers(PyObject* self, PyObject* const* a, Py_ssize_t n) {   /* delim_ids, n_delim -> one sequence */
    int32_t delims[SC_MAX_DELIMS + 1];
    (void)self;
    if (!arity(n, 13, "append_layers")) return NULL;
    const int32_t nd = ids_of(a[7], delims);
    if (nd < 0) return NULL;
    const void *table = ptr(a[0]), *ids = ptr(a[6]);
    const sc_dtype dt = (sc_dtype)i32(a[2]);
    const int32_t L = i32(a[1]), B = i32(a[3]), H = i32(a[4]), d = i32(a[5]), max_len = i32(a[8]), cap = i32(a[10]);
    const float tau = f32(a[9]);
    void *status = ptr(a[11]), *stream = ptr(a[12]);
    CALL(sc_append_layers(table, L, dt, B, H, d, ids, delims, nd, max_len, tau, cap, status, stream));
}

#define FN(name) {#name, (PyCFunction)(void (*)(void))name, METH_FASTCALL, NULL}
static PyMethodDef methods[] = {FN(chunk_sizes), FN(chunk), FN(compress), FN(decode_attn), FN(prefill_attn), FN(append), FN(append_layers),
                                {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native_calls", NULL, -1, methods, NULL, NULL, NULL, NULL};
PyMODINIT_FUNC PyInit__native_calls(void) { return PyModule_Create(&module); }
