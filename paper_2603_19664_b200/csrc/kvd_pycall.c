/* Argument marshalling of the calls that a decode step makes, in C.
 *
 * binding.py converts Python arguments for ctypes; for the small layers that costs more time than the GPU needs (a step of
 * four calls: 8.6 us in Python, 2.9 here).  Every function below takes the arguments of the Kvd method of its name, as they
 * are, behind the context's address, and returns the library's status -- or -1, before anything has been called, if an
 * argument is not of the plain kind it knows (tensors, exact ints in range, lists and tuples): binding.py then marshals the
 * call itself, with whatever conversion or exception that brings.  (What is no Exception -- an interrupt, an exit -- is not an
 * argument's fault and passes through.)  The library runs without the interpreter lock, as under
 * ctypes.
 */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <limits.h>
#include <stdint.h>

#include "../../include/kvd.h"

#define MAX_ENTRIES 256 /* segments or ranges marshalled on the stack */

static PyObject *s_data_ptr;
static kvd_status (*p_reset_sequence)(kvd_ctx *, int);
static kvd_status (*p_checkpoint_residual)(kvd_ctx *, int, int, const void *, const int32_t *, int, void *);
static kvd_status (*p_recompute_kv)(kvd_ctx *, int, const void *, const int32_t *, int, int, int, void *, void *, int64_t, void *);
static kvd_status (*p_recompute_kv_step)(kvd_ctx *, int, const kvd_store_range *, int, const void *, const int32_t *, int, void *, void *, int64_t, void *);
static kvd_status (*p_decode_step_kv)(kvd_ctx *, int, const kvd_store_range *, int, int64_t, const void *, const int32_t *, int, const int32_t *, void *,
                                      void *, int64_t, void *);
static kvd_status (*p_decode_attention)(kvd_ctx *, int, int, const void *, const int32_t *, const kvd_kv_segment *, int, float, void *, void *);
static kvd_status (*p_prefill_attention)(kvd_ctx *, int, int, const void *, const int32_t *, const kvd_kv_segment *, int, float, void *, void *);

static const struct {
  const char *name;
  void **slot;
} k_entries[] = {
    {"kvd_reset_sequence", (void **)&p_reset_sequence},       {"kvd_checkpoint_residual", (void **)&p_checkpoint_residual},
    {"kvd_recompute_kv", (void **)&p_recompute_kv},           {"kvd_recompute_kv_step", (void **)&p_recompute_kv_step},
    {"kvd_decode_step_kv", (void **)&p_decode_step_kv},       {"kvd_decode_attention", (void **)&p_decode_attention},
    {"kvd_prefill_attention", (void **)&p_prefill_attention},
};

static int as_i64(PyObject *o, int64_t *out) {
  int over = 0;
  if (!PyLong_CheckExact(o)) return 0;
  *out = PyLong_AsLongLongAndOverflow(o, &over);
  return over == 0;
}
static int as_int(PyObject *o, int *out) {
  int64_t v;
  if (!as_i64(o, &v) || v < INT_MIN || v > INT_MAX) return 0;
  *out = (int)v;
  return 1;
}
/* an address handed over by binding.py (context, stream) */
static int as_handle(PyObject *o, void **out) {
  if (o == Py_None) {
    *out = NULL;
    return 1;
  }
  if (!PyLong_CheckExact(o)) return 0;
  *out = PyLong_AsVoidPtr(o);
  if (*out == NULL && PyErr_Occurred()) {
    PyErr_Clear();
    return 0;
  }
  return 1;
}
/* the address of a tensor; None is NULL where `optional` says so */
static int as_tensor(PyObject *o, void **out, int optional) {
  PyObject *r;
  int ok;
  if (o == Py_None && optional) {
    *out = NULL;
    return 1;
  }
  if (o == Py_None || PyLong_Check(o)) return 0;
  r = PyObject_CallMethodNoArgs(o, s_data_ptr);
  if (r == NULL) {
    if (PyErr_ExceptionMatches(PyExc_Exception)) PyErr_Clear();
    return 0;
  }
  ok = as_handle(r, out) && r != Py_None;
  Py_DECREF(r);
  return ok;
}
/* items and length of a list or tuple */
static PyObject **items_of(PyObject *o, Py_ssize_t *n) {
  if (!PyList_CheckExact(o) && !PyTuple_CheckExact(o)) return NULL;
  *n = PySequence_Fast_GET_SIZE(o);
  return PySequence_Fast_ITEMS(o);
}
static int as_ints(PyObject *o, Py_ssize_t want, int32_t *out) {
  Py_ssize_t n, i;
  PyObject **it = items_of(o, &n);
  if (it == NULL || n != want || n > MAX_ENTRIES) return 0;
  for (i = 0; i < n; ++i) {
    int v;
    if (!as_int(it[i], &v)) return 0;
    out[i] = v;
  }
  return 1;
}
/* Objects reached through a list stay alive only as long as the list holds them, and data_ptr() runs Python code: every
 * entry is kept over its own conversion. */
static int as_segment(PyObject *o, kvd_kv_segment *e) {
  Py_ssize_t n;
  int64_t stride;
  int first, len, ok;
  void *k, *v;
  PyObject **it;
  Py_INCREF(o);
  it = items_of(o, &n);
  ok = it != NULL && PyTuple_CheckExact(o) && n == 5 && as_tensor(it[0], &k, 0) && as_tensor(it[1], &v, 0) && as_i64(it[2], &stride) &&
       as_int(it[3], &first) && as_int(it[4], &len);
  if (ok) {
    e->k = k;
    e->v = v;
    e->row_stride = stride;
    e->first_pos = first;
    e->len = len;
  }
  Py_DECREF(o);
  return ok;
}
static int as_range(PyObject *o, kvd_store_range *e) {
  Py_ssize_t n;
  int seq, first, rows, ok;
  void *k, *v;
  PyObject **it;
  Py_INCREF(o);
  it = items_of(o, &n);
  ok = it != NULL && PyTuple_CheckExact(o) && n == 5 && as_int(it[0], &seq) && as_int(it[1], &first) && as_int(it[2], &rows) &&
       as_tensor(it[3], &k, 0) && as_tensor(it[4], &v, 0);
  if (ok) {
    e->seq = seq;
    e->first_row = first;
    e->n = rows;
    e->reserved = 0;
    e->k_out = k;
    e->v_out = v;
  }
  Py_DECREF(o);
  return ok;
}
/* a list may change while data_ptr() runs: its length is read again for every entry */
static int as_ranges(PyObject *o, kvd_store_range *out, int *count) {
  Py_ssize_t n, i;
  if (items_of(o, &n) == NULL || n > MAX_ENTRIES) return 0;
  *count = (int)n;
  for (i = 0; i < n; ++i) {
    Py_ssize_t now;
    PyObject **it = items_of(o, &now);
    if (now != n || !as_range(it[i], &out[i])) return 0;
  }
  return 1;
}
/* `rows` lists of segments, of up to *count segments each, absent ones zero */
static int as_segments(PyObject *const *lists, Py_ssize_t rows, kvd_kv_segment *out, int *count) {
  Py_ssize_t most = 0, r, i, n;
  for (r = 0; r < rows; ++r) {
    if (items_of(lists[r], &n) == NULL) return 0;
    if (n > most) most = n;
  }
  if (most * rows > MAX_ENTRIES) return 0;
  for (r = 0; r < rows; ++r) {
    PyObject *list = lists[r];
    Py_INCREF(list);
    for (i = 0; i < most; ++i) {
      PyObject **it = items_of(list, &n);
      kvd_kv_segment *e = &out[r * most + i];
      if (n > most || (i < n && !as_segment(it[i], e))) {
        Py_DECREF(list);
        return 0;
      }
      if (i >= n) *e = (kvd_kv_segment){0};
    }
    Py_DECREF(list);
  }
  *count = (int)most;
  return 1;
}

#define UNUSUAL return PyErr_Occurred() ? NULL : PyLong_FromLong(-1)
#define CALL(expr)                    \
  do {                                \
    kvd_status st_;                   \
    Py_BEGIN_ALLOW_THREADS st_ = expr; \
    Py_END_ALLOW_THREADS return PyLong_FromLong((long)st_); \
  } while (0)

static PyObject *py_reset_sequence(PyObject *self, PyObject *const *a, Py_ssize_t n) {
  void *h;
  int seq;
  (void)self;
  if (n != 2 || !as_handle(a[0], &h) || !as_int(a[1], &seq)) UNUSUAL;
  CALL(p_reset_sequence(h, seq));
}
/* (ctx, seq, layer, rows, positions, n, stream) */
static PyObject *py_checkpoint_residual(PyObject *self, PyObject *const *a, Py_ssize_t n) {
  void *h, *rows, *pos, *stream;
  int seq, layer, count;
  (void)self;
  if (n != 7 || !as_handle(a[0], &h) || !as_int(a[1], &seq) || !as_int(a[2], &layer) || !as_tensor(a[3], &rows, 1) || !as_tensor(a[4], &pos, 1) ||
      !as_int(a[5], &count) || !as_handle(a[6], &stream))
    UNUSUAL;
  CALL(p_checkpoint_residual(h, seq, layer, rows, pos, count, stream));
}
/* (ctx, layer, rows, positions, n, k_out, v_out, out_row_stride, seq, first_row, stream) */
static PyObject *py_recompute_kv(PyObject *self, PyObject *const *a, Py_ssize_t n) {
  void *h, *rows, *pos, *k, *v, *stream;
  int layer, count, seq, first;
  int64_t stride;
  (void)self;
  if (n != 11 || !as_handle(a[0], &h) || !as_int(a[1], &layer) || !as_tensor(a[2], &rows, 1) || !as_tensor(a[3], &pos, 1) || !as_int(a[4], &count) ||
      !as_tensor(a[5], &k, 1) || !as_tensor(a[6], &v, 1) || !as_i64(a[7], &stride) || !as_int(a[8], &seq) || !as_int(a[9], &first) ||
      !as_handle(a[10], &stream))
    UNUSUAL;
  CALL(p_recompute_kv(h, layer, rows, pos, count, seq, first, k, v, stride, stream));
}
/* (ctx, layer, ranges, rows, positions, n_rows, k_rows_out, v_rows_out, out_row_stride, stream) */
static PyObject *py_recompute_kv_step(PyObject *self, PyObject *const *a, Py_ssize_t n) {
  void *h, *rows, *pos, *k, *v, *stream;
  int layer, count, n_ranges;
  int64_t stride;
  kvd_store_range ranges[MAX_ENTRIES];
  (void)self;
  if (n != 10 || !as_handle(a[0], &h) || !as_int(a[1], &layer) || !as_ranges(a[2], ranges, &n_ranges) || !as_tensor(a[3], &rows, 1) ||
      !as_tensor(a[4], &pos, 1) || !as_int(a[5], &count) || !as_tensor(a[6], &k, 1) || !as_tensor(a[7], &v, 1) || !as_i64(a[8], &stride) ||
      !as_handle(a[9], &stream))
    UNUSUAL;
  CALL(p_recompute_kv_step(h, layer, ranges, n_ranges, rows, pos, count, k, v, stride, stream));
}
/* (ctx, layer, ranges, out_row_stride, rows, positions, n_rows, append_seqs, k_rows_out, v_rows_out, rows_out_row_stride, stream) */
static PyObject *py_decode_step_kv(PyObject *self, PyObject *const *a, Py_ssize_t n) {
  void *h, *rows, *pos, *k, *v, *stream;
  int layer, count, n_ranges;
  int64_t stride, rows_stride;
  kvd_store_range ranges[MAX_ENTRIES];
  int32_t seqs[MAX_ENTRIES];
  (void)self;
  if (n != 12 || !as_handle(a[0], &h) || !as_int(a[1], &layer) || !as_ranges(a[2], ranges, &n_ranges) || !as_i64(a[3], &stride) ||
      !as_tensor(a[4], &rows, 1) || !as_tensor(a[5], &pos, 1) || !as_int(a[6], &count) || (a[7] != Py_None && !as_ints(a[7], count, seqs)) ||
      !as_tensor(a[8], &k, 1) || !as_tensor(a[9], &v, 1) || !as_i64(a[10], &rows_stride) || !as_handle(a[11], &stream))
    UNUSUAL;
  CALL(p_decode_step_kv(h, layer, ranges, n_ranges, stride, rows, pos, count, a[7] == Py_None ? NULL : seqs, k, v, rows_stride, stream));
}
/* (ctx, layer, batch, q, q_pos, segs, scale, out, stream) */
static PyObject *py_decode_attention(PyObject *self, PyObject *const *a, Py_ssize_t n) {
  void *h, *q, *out, *stream;
  int layer, batch, n_segs;
  Py_ssize_t lists;
  PyObject **segs;
  int32_t pos[MAX_ENTRIES];
  kvd_kv_segment seg[MAX_ENTRIES];
  (void)self;
  if (n != 9 || !as_handle(a[0], &h) || !as_int(a[1], &layer) || !as_int(a[2], &batch) || batch < 1 || !as_tensor(a[3], &q, 1) ||
      !as_ints(a[4], batch, pos) || !PyFloat_CheckExact(a[6]) || !as_tensor(a[7], &out, 1) || !as_handle(a[8], &stream))
    UNUSUAL;
  /* (a copy of the outer list: the inner ones are held one by one) */
  segs = items_of(a[5], &lists);
  if (segs == NULL || lists != batch) UNUSUAL;
  {
    PyObject *held = PySequence_Tuple(a[5]);
    int ok;
    if (held == NULL) return NULL;
    ok = PyTuple_GET_SIZE(held) == batch && as_segments(PySequence_Fast_ITEMS(held), batch, seg, &n_segs);
    Py_DECREF(held);
    if (!ok) UNUSUAL;
  }
  CALL(p_decode_attention(h, layer, batch, q, pos, seg, n_segs, (float)PyFloat_AS_DOUBLE(a[6]), out, stream));
}
/* (ctx, layer, n_rows, q, q_pos, segs, scale, out, stream): q_pos a device tensor, segs of one sequence */
static PyObject *py_prefill_attention(PyObject *self, PyObject *const *a, Py_ssize_t n) {
  void *h, *q, *pos, *out, *stream;
  int layer, rows, n_segs;
  kvd_kv_segment seg[MAX_ENTRIES];
  (void)self;
  if (n != 9 || !as_handle(a[0], &h) || !as_int(a[1], &layer) || !as_int(a[2], &rows) || !as_tensor(a[3], &q, 1) || !as_tensor(a[4], &pos, 1) ||
      !as_segments(&a[5], 1, seg, &n_segs) || !PyFloat_CheckExact(a[6]) || !as_tensor(a[7], &out, 1) || !as_handle(a[8], &stream))
    UNUSUAL;
  CALL(p_prefill_attention(h, layer, rows, q, pos, seg, n_segs, (float)PyFloat_AS_DOUBLE(a[6]), out, stream));
}

/* bind(name, address): the library's entry point of that name */
static PyObject *py_bind(PyObject *self, PyObject *const *a, Py_ssize_t n) {
  const char *name;
  void *address;
  size_t i;
  (void)self;
  if (n != 2 || (name = PyUnicode_AsUTF8(a[0])) == NULL || !as_handle(a[1], &address)) {
    if (!PyErr_Occurred()) PyErr_SetString(PyExc_TypeError, "bind(name, address)");
    return NULL;
  }
  for (i = 0; i < sizeof(k_entries) / sizeof(k_entries[0]); ++i)
    if (strcmp(name, k_entries[i].name) == 0) {
      *k_entries[i].slot = address;
      Py_RETURN_NONE;
    }
  PyErr_SetString(PyExc_KeyError, name);
  return NULL;
}

#define FAST(name) {"kvd_" #name, (PyCFunction)(void (*)(void))py_##name, METH_FASTCALL, NULL}
static PyMethodDef k_methods[] = {FAST(reset_sequence),   FAST(checkpoint_residual), FAST(recompute_kv),      FAST(recompute_kv_step),
                                  FAST(decode_step_kv),   FAST(decode_attention),    FAST(prefill_attention), {"bind", (PyCFunction)(void (*)(void))py_bind, METH_FASTCALL, NULL},
                                  {NULL, NULL, 0, NULL}};
static struct PyModuleDef k_module = {PyModuleDef_HEAD_INIT, "_kvdcall", NULL, -1, k_methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__kvdcall(void) {
  s_data_ptr = PyUnicode_InternFromString("data_ptr");
  return s_data_ptr == NULL ? NULL : PyModule_Create(&k_module);
}
