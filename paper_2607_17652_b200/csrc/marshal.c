/* CPython side of the binding: tensors -> raw device pointers -> one C call.
 *
 * Each function takes the context handle (an int), the Python objects of the
 * call in the order of the C entry point and the stream (an int), reads
 * `data_ptr()` of every tensor anew (nothing is kept from one call for the
 * next), fills fb_state / fb_pack on the stack, releases the GIL around the C
 * call and returns its error code.  What it is for: a decode step of a single
 * request is bound by the host, and marshalling through ctypes structures took
 * about 10 us a call (step of one small request: 55.6 us, now 32.2 us; the
 * marshalling part of a call is now about 2 us).
 *
 * The entry points come from libflowblock.so by address (bind), so this module
 * links against nothing. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include "../../include/flowblock.h"

static PyObject *s_data_ptr;
static PyObject *s_state[7], *s_pack[9];
static const char* const k_state[7] = {"active", "prefix_len", "L", "R", "tokens", "pe_done", "page_table"};
static const char* const k_pack[9] = {"n_live", "slot_req", "slot_s", "slot_pos0", "slot_kv_len", "slot_flags",
                                      "req_slot_begin", "qtok", "pos"};

/* entry points, in the order of `names` in bind() */
enum { F_PACK, F_ATTN, F_T2T, F_GATE, F_SCATTER, F_SCATTER8, F_ATTN8, F_EMBED, F_HEAD, F_STATIC, F_COUNT };
static void* fn[F_COUNT];

static PyObject* bind(PyObject* self, PyObject* const* args, Py_ssize_t n) {
  (void)self;
  if (n != F_COUNT) { PyErr_SetString(PyExc_TypeError, "bind: one address per entry point"); return NULL; }
  void* got[F_COUNT];
  for (int i = 0; i < F_COUNT; ++i) {
    got[i] = PyLong_AsVoidPtr(args[i]);
    if (!got[i]) {
      if (!PyErr_Occurred()) PyErr_SetString(PyExc_ValueError, "bind: null address");
      return NULL;
    }
  }
  for (int i = 0; i < F_COUNT; ++i) fn[i] = got[i];
  Py_RETURN_NONE;
}

/* None -> NULL, an int -> itself, anything else -> its data_ptr() */
static int as_ptr(PyObject* o, void** out) {
  if (o == Py_None) { *out = NULL; return 0; }
  if (PyLong_Check(o)) {
    *out = PyLong_AsVoidPtr(o);
    return *out == NULL && PyErr_Occurred() ? -1 : 0;
  }
  PyObject* v = PyObject_CallMethodNoArgs(o, s_data_ptr);
  if (!v) return -1;
  *out = PyLong_AsVoidPtr(v);
  Py_DECREF(v);
  return *out == NULL && PyErr_Occurred() ? -1 : 0;
}

static int fill(PyObject* o, PyObject* const* names, int n, void** out) {
  for (int i = 0; i < n; ++i) {
    PyObject* t = PyObject_GetAttr(o, names[i]);
    if (!t) return -1;
    const int e = as_ptr(t, &out[i]);
    Py_DECREF(t);
    if (e) return -1;
  }
  return 0;
}
_Static_assert(sizeof(fb_state) == 7 * sizeof(void*) && sizeof(fb_pack) == 9 * sizeof(void*), "plain pointer structures");

static int as_int(PyObject* o, int32_t* out) {
  const long v = PyLong_AsLong(o);
  if (v == -1 && PyErr_Occurred()) return -1;
  if (v < INT32_MIN || v > INT32_MAX) { PyErr_SetString(PyExc_OverflowError, "value does not fit in 32 bits"); return -1; }
  *out = (int32_t)v;
  return 0;
}

#define ARGS(count, name)                                                                        \
  (void)self;                                                                                    \
  if (n != (count)) { PyErr_SetString(PyExc_TypeError, name ": wrong number of arguments"); return NULL; } \
  if (!fn[F_PACK]) { PyErr_SetString(PyExc_RuntimeError, "the library is not bound"); return NULL; } \
  void* ctx;                                                                                     \
  if (as_ptr(a[0], &ctx)) return NULL;
#define STATE(i, st) fb_state st; if (fill(a[i], s_state, 7, (void**)&st)) return NULL;
#define PACK(i, pk) fb_pack pk; if (fill(a[i], s_pack, 9, (void**)&pk)) return NULL;
#define PTRS(first, count) void* q[count]; for (int i = 0; i < (count); ++i) if (as_ptr(a[(first) + i], &q[i])) return NULL;
#define CALL(expr) int rc; Py_BEGIN_ALLOW_THREADS rc = (expr); Py_END_ALLOW_THREADS return PyLong_FromLong(rc);
#define FN(index, f) ((__typeof__(&f))fn[index])

/* handle, st, pk, ws, status, stream */
static PyObject* m_pack(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  ARGS(6, "pack") STATE(1, st) PACK(2, pk) PTRS(3, 3)
  CALL(FN(F_PACK, fb_pack_wavefronts)(ctx, &st, &pk, q[0], q[1], q[2]))
}
/* handle, pk, q, k_win, v_win, k_pool, v_pool, page_table, out, ws, status, stream */
static PyObject* m_attn(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  ARGS(12, "attn") PACK(1, pk) PTRS(2, 10)
  CALL(FN(F_ATTN, fb_wavefront_attn)(ctx, &pk, q[0], q[1], q[2], q[3], q[4], q[5], q[6], q[7], q[8], q[9]))
}
/* handle, pk, q, k_pool8, v_pool8, k_scale, v_scale, page_table, out, ws, status, stream */
static PyObject* m_attn8(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  ARGS(12, "attn_fp8") PACK(1, pk) PTRS(2, 10)
  CALL(FN(F_ATTN8, fb_wavefront_attn_fp8)(ctx, &pk, q[0], q[1], q[2], q[3], q[4], q[5], q[6], q[7], q[8], q[9]))
}
/* handle, pk, logits, st, argmax, conf, action, slot_stats, status, stream */
static PyObject* m_t2t(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  ARGS(10, "t2t") PACK(1, pk) STATE(3, st) PTRS(4, 6)
  void* logits;
  if (as_ptr(a[2], &logits)) return NULL;
  CALL(FN(F_T2T, fb_t2t_step)(ctx, &pk, logits, &st, q[0], q[1], q[2], q[3], q[4], q[5]))
}
/* handle, pk, slot_stats, st, k_win, v_win, k_pool, v_pool, n_committed, spawned, step_counters, status, stream */
static PyObject* m_gate(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  ARGS(13, "gate") PACK(1, pk) STATE(3, st) PTRS(4, 9)
  void* stats;
  if (as_ptr(a[2], &stats)) return NULL;
  CALL(FN(F_GATE, fb_gate_commit)(ctx, &pk, stats, &st, q[0], q[1], q[2], q[3], q[4], q[5], q[6], q[7], q[8]))
}
/* handle, pk, page_table, k_new, v_new, k_pool, v_pool, rope_base, status, stream */
static PyObject* m_scatter(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  ARGS(10, "scatter") PACK(1, pk) PTRS(2, 5)
  void *status, *stream;
  const double base = PyFloat_AsDouble(a[7]);
  if (base == -1.0 && PyErr_Occurred()) return NULL;
  if (as_ptr(a[8], &status) || as_ptr(a[9], &stream)) return NULL;
  CALL(FN(F_SCATTER, fb_scatter_window_kv)(ctx, &pk, q[0], q[1], q[2], q[3], q[4], (float)base, status, stream))
}
/* handle, pk, page_table, k_new, v_new, k_pool8, v_pool8, k_scale, v_scale, rope_base, status, stream */
static PyObject* m_scatter8(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  ARGS(12, "scatter_fp8") PACK(1, pk) PTRS(2, 7)
  void *status, *stream;
  const double base = PyFloat_AsDouble(a[9]);
  if (base == -1.0 && PyErr_Occurred()) return NULL;
  if (as_ptr(a[10], &status) || as_ptr(a[11], &stream)) return NULL;
  CALL(FN(F_SCATTER8, fb_scatter_window_kv_fp8)(ctx, &pk, q[0], q[1], q[2], q[3], q[4], q[5], q[6], (float)base, status,
                                                stream))
}
/* handle, pk, table, table_rows, hidden, x, status, stream */
static PyObject* m_embed(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  ARGS(8, "embed") PACK(1, pk) PTRS(5, 3)
  void* table;
  int32_t rows, hidden;
  if (as_ptr(a[2], &table) || as_int(a[3], &rows) || as_int(a[4], &hidden)) return NULL;
  CALL(FN(F_EMBED, fb_embed_gather)(ctx, &pk, table, rows, hidden, q[0], q[1], q[2]))
}
/* handle, pk, x, w, hidden, st, argmax, conf, action, slot_stats, ws, status, stream */
static PyObject* m_head(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  ARGS(13, "lm_head") PACK(1, pk) STATE(5, st) PTRS(6, 7)
  void *x, *w;
  int32_t hidden;
  if (as_ptr(a[2], &x) || as_ptr(a[3], &w) || as_int(a[4], &hidden)) return NULL;
  CALL(FN(F_HEAD, fb_lm_head_t2t)(ctx, &pk, x, w, hidden, &st, q[0], q[1], q[2], q[3], q[4], q[5], q[6]))
}
/* handle, st, pk, q, k_win, v_win, k_pool, v_pool, out, status, stream */
static PyObject* m_static(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  ARGS(11, "attn_static") STATE(1, st) PACK(2, pk) PTRS(3, 8)
  CALL(FN(F_STATIC, fb_wavefront_attn_static)(ctx, &st, &pk, q[0], q[1], q[2], q[3], q[4], q[5], q[6], q[7]))
}

#define M(name, f) {name, (PyCFunction)(void (*)(void))f, METH_FASTCALL, NULL}
static PyMethodDef methods[] = {
    M("bind", bind), M("pack", m_pack), M("attn", m_attn), M("attn_fp8", m_attn8), M("t2t", m_t2t), M("gate", m_gate),
    M("scatter", m_scatter), M("scatter_fp8", m_scatter8), M("embed", m_embed), M("lm_head", m_head),
    M("attn_static", m_static), {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_marshal", "argument marshalling of the binding", -1, methods,
                                    NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__marshal(void) {
  if (!(s_data_ptr = PyUnicode_InternFromString("data_ptr"))) return NULL;
  for (int i = 0; i < 7; ++i) if (!(s_state[i] = PyUnicode_InternFromString(k_state[i]))) return NULL;
  for (int i = 0; i < 9; ++i) if (!(s_pack[i] = PyUnicode_InternFromString(k_pack[i]))) return NULL;
  return PyModule_Create(&module);
}
