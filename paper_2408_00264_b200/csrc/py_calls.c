/* CPython entry points of the calls of libclv that a decode loop makes: argument marshalling only.
 *
 * A verify step of a single user keeps the GPU busy for some 15 microseconds in three calls.  Through
 * ctypes a call of 16 arguments took 12 us of host time (every pointer becomes a c_void_p object, the
 * stream a torch Stream object), so the host and not the GPU set the pace.  Here a tensor's address is
 * one bound call of its data_ptr(), a descriptor is read through the buffer protocol of its ctypes
 * structure, and the stream is the current one's raw handle.  No header of torch is used.
 * Every function returns the library's status code; the Python side turns it into an exception.
 * The interpreter lock is released while the library runs. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>

#include "clv.h"

static PyObject *s_data_ptr, *s_nbytes, *s_cuda_stream;   /* interned attribute names */
static PyObject *g_get_device, *g_get_raw_stream;          /* torch._C functions, set by init() */

/* address of a tensor's first element; NULL for None */
static int get_ptr(PyObject *o, void **out) {
  if (o == Py_None) {
    *out = NULL;
    return 0;
  }
  PyObject *v = PyObject_CallMethodNoArgs(o, s_data_ptr);
  if (!v) return -1;
  *out = PyLong_AsVoidPtr(v);
  Py_DECREF(v);
  return (*out == NULL && PyErr_Occurred()) ? -1 : 0;
}
/* size in bytes of a tensor; 0 for None */
static int get_bytes(PyObject *o, size_t *out) {
  *out = 0;
  if (o == Py_None) return 0;
  PyObject *v = PyObject_GetAttr(o, s_nbytes);
  if (!v) return -1;
  *out = PyLong_AsSize_t(v);
  Py_DECREF(v);
  return (*out == (size_t)-1 && PyErr_Occurred()) ? -1 : 0;
}
/* address of a ctypes structure of at least `size` bytes (the caller's argument keeps it alive) */
static int get_struct(PyObject *o, size_t size, void **out) {
  Py_buffer b;
  if (PyObject_GetBuffer(o, &b, PyBUF_SIMPLE) != 0) return -1;
  *out = b.buf;
  const int short_ = (size_t)b.len < size;
  PyBuffer_Release(&b);
  if (short_) {
    PyErr_SetString(PyExc_TypeError, "descriptor structure is too small");
    return -1;
  }
  return 0;
}
static int get_i64(PyObject *o, int64_t *out) {
  if (PyLong_Check(o)) {
    *out = PyLong_AsLongLong(o);
  } else { /* anything int() takes */
    PyObject *v = PyNumber_Long(o);
    if (!v) return -1;
    *out = PyLong_AsLongLong(v);
    Py_DECREF(v);
  }
  return (*out == -1 && PyErr_Occurred()) ? -1 : 0;
}
static int get_i32(PyObject *o, int32_t *out) {
  int64_t v;
  if (get_i64(o, &v)) return -1;
  *out = (int32_t)v;
  return 0;
}
static int get_f32(PyObject *o, float *out) {
  const double v = PyFloat_AsDouble(o);
  *out = (float)v;
  return (v == -1.0 && PyErr_Occurred()) ? -1 : 0;
}
/* raw handle of a torch stream; None = the current stream of the current device */
static int get_stream(PyObject *o, void **out) {
  PyObject *v;
  if (o == Py_None) {
    PyObject *dev = PyObject_CallNoArgs(g_get_device);
    if (!dev) return -1;
    v = PyObject_CallOneArg(g_get_raw_stream, dev);
    Py_DECREF(dev);
  } else {
    v = PyObject_GetAttr(o, s_cuda_stream);
  }
  if (!v) return -1;
  *out = PyLong_AsVoidPtr(v);
  Py_DECREF(v);
  return (*out == NULL && PyErr_Occurred()) ? -1 : 0;
}

#define ARGS PyObject *self, PyObject *const *a, Py_ssize_t n
#define NEED(count)                                                                   \
  (void)self;                                                                         \
  if (n != (count)) return PyErr_Format(PyExc_TypeError, "%d arguments expected", (int)(count))
#define TRY(expr) \
  if (expr) return NULL
/* the tensors a[first .. first + count) to p[] */
static int get_ptrs(PyObject *const *a, int first, int count, void **p) {
  for (int i = 0; i < count; ++i)
    if (get_ptr(a[first + i], p + i)) return -1;
  return 0;
}
#define CALL(expr)            \
  int32_t code;               \
  Py_BEGIN_ALLOW_THREADS;     \
  code = (expr);              \
  Py_END_ALLOW_THREADS;       \
  return PyLong_FromLong(code)

static PyObject *tree_attn(ARGS) { /* shape cache q k_tree v_tree parent ctx_len max_ctx scale out lse status ws stream */
  NEED(14);
  void *shape, *cache, *p[5], *o[4], *st;
  int32_t max_ctx;
  float scale;
  size_t ws_bytes;
  TRY(get_struct(a[0], sizeof(clv_shape), &shape) || get_struct(a[1], sizeof(clv_kv_cache), &cache));
  TRY(get_ptrs(a, 2, 5, p) || get_i32(a[7], &max_ctx) || get_f32(a[8], &scale));
  TRY(get_ptrs(a, 9, 4, o) || get_bytes(a[12], &ws_bytes) || get_stream(a[13], &st));
  CALL(clv_tree_attn(shape, cache, p[0], p[1], p[2], p[3], p[4], max_ctx, scale, o[0], o[1], o[2], o[3], ws_bytes, st));
}

static PyObject *accept_argmax(ARGS) { /* shape logits ld ids ws stream */
  NEED(6);
  void *shape, *lg, *o[2], *st;
  int64_t ld;
  size_t ws_bytes;
  TRY(get_struct(a[0], sizeof(clv_shape), &shape) || get_ptr(a[1], &lg) || get_i64(a[2], &ld));
  TRY(get_ptrs(a, 3, 2, o) || get_bytes(a[4], &ws_bytes) || get_stream(a[5], &st));
  CALL(clv_accept_argmax(shape, lg, ld, o[0], o[1], ws_bytes, st));
}

static PyObject *accept_argmax_noalloc(ARGS) { /* shape logits ld ids stream */
  NEED(5);
  void *shape, *lg, *ids, *st;
  int64_t ld;
  TRY(get_struct(a[0], sizeof(clv_shape), &shape) || get_ptr(a[1], &lg) || get_i64(a[2], &ld));
  TRY(get_ptr(a[3], &ids) || get_stream(a[4], &st));
  CALL(clv_accept_argmax_noalloc(shape, lg, ld, ids, st));
}

static PyObject *accept_walk(ARGS) { /* shape, 7 tensors, stream */
  NEED(9);
  void *shape, *p[7], *st;
  TRY(get_struct(a[0], sizeof(clv_shape), &shape) || get_ptrs(a, 1, 7, p) || get_stream(a[8], &st));
  CALL(clv_accept_walk(shape, p[0], p[1], p[2], p[3], p[4], p[5], p[6], st));
}

static PyObject *kv_commit(ARGS) { /* shape cache, 7 tensors, stream */
  NEED(10);
  void *shape, *cache, *p[7], *st;
  TRY(get_struct(a[0], sizeof(clv_shape), &shape) || get_struct(a[1], sizeof(clv_kv_cache), &cache));
  TRY(get_ptrs(a, 2, 7, p) || get_stream(a[9], &st));
  CALL(clv_kv_commit(shape, cache, p[0], p[1], p[2], p[3], p[4], p[5], p[6], st));
}

static PyObject *accept_walk_commit(ARGS) { /* shape cache, 12 tensors, stream */
  NEED(15);
  void *shape, *cache, *p[12], *st;
  TRY(get_struct(a[0], sizeof(clv_shape), &shape) || get_struct(a[1], sizeof(clv_kv_cache), &cache));
  TRY(get_ptrs(a, 2, 12, p) || get_stream(a[14], &st));
  CALL(clv_accept_walk_commit(shape, cache, p[0], p[1], p[2], p[3], p[4], p[5], p[6], p[7], p[8], p[9], p[10], p[11], st));
}

static PyObject *accept_sample(ARGS) { /* shape logits ld parent tokens uniforms T len idx next status ws stream */
  NEED(13);
  void *shape, *lg, *p[3], *o[5], *st;
  int64_t ld;
  float temp;
  size_t ws_bytes;
  TRY(get_struct(a[0], sizeof(clv_shape), &shape) || get_ptr(a[1], &lg) || get_i64(a[2], &ld));
  TRY(get_ptrs(a, 3, 3, p) || get_f32(a[6], &temp) || get_ptrs(a, 7, 5, o));
  TRY(get_bytes(a[11], &ws_bytes) || get_stream(a[12], &st));
  CALL(clv_accept_sample(shape, lg, ld, p[0], p[1], p[2], temp, o[0], o[1], o[2], o[3], o[4], ws_bytes, st));
}

static PyObject *tree_to_intervals(ARGS) { /* batch n, 4 tensors, stream */
  NEED(7);
  int32_t b, nn;
  void *p[4], *st;
  TRY(get_i32(a[0], &b) || get_i32(a[1], &nn) || get_ptrs(a, 2, 4, p) || get_stream(a[6], &st));
  CALL(clv_tree_to_intervals(b, nn, p[0], p[1], p[2], p[3], st));
}

static PyObject *tree_from_intervals(ARGS) { /* batch n, 4 tensors, stream */
  NEED(7);
  int32_t b, nn;
  void *p[4], *st;
  TRY(get_i32(a[0], &b) || get_i32(a[1], &nn) || get_ptrs(a, 2, 4, p) || get_stream(a[6], &st));
  CALL(clv_tree_from_intervals(b, nn, p[0], p[1], p[2], p[3], st));
}

static PyObject *kv_commit_layers(ARGS) { /* shape cache layers cache_stride kt vt tree_stride idx len ctx ctx_out status stream */
  NEED(13);
  void *shape, *cache, *t[2], *p[5], *st;
  int32_t layers;
  int64_t cs, ts;
  TRY(get_struct(a[0], sizeof(clv_shape), &shape) || get_struct(a[1], sizeof(clv_kv_cache), &cache));
  TRY(get_i32(a[2], &layers) || get_i64(a[3], &cs) || get_ptrs(a, 4, 2, t) || get_i64(a[6], &ts));
  TRY(get_ptrs(a, 7, 5, p) || get_stream(a[12], &st));
  CALL(clv_kv_commit_layers(shape, cache, layers, cs, t[0], t[1], ts, p[0], p[1], p[2], p[3], p[4], st));
}

static PyObject *draft_head_step(ARGS) { /* head rows h e k_top hidden_out ids logits status ws stream */
  NEED(11);
  void *head, *x[2], *o[5], *st;
  int32_t rows, k;
  size_t ws_bytes;
  TRY(get_struct(a[0], sizeof(clv_draft_head), &head) || get_i32(a[1], &rows) || get_ptrs(a, 2, 2, x));
  TRY(get_i32(a[4], &k) || get_ptrs(a, 5, 5, o) || get_bytes(a[9], &ws_bytes) || get_stream(a[10], &st));
  CALL(clv_draft_head_step(head, rows, x[0], x[1], k, o[0], o[1], o[2], o[3], o[4], ws_bytes, st));
}

static PyObject *build_token_tree(ARGS) { /* batch cand len cap, 8 tensors, stream */
  NEED(13);
  int32_t v[4];
  void *p[8], *st;
  for (int i = 0; i < 4; ++i) TRY(get_i32(a[i], v + i));
  TRY(get_ptrs(a, 4, 8, p) || get_stream(a[12], &st));
  CALL(clv_build_token_tree(v[0], v[1], v[2], v[3], p[0], p[1], p[2], p[3], p[4], p[5], p[6], p[7], st));
}

static PyObject *lm_head_argmax(ARGS) { /* hidden ld weight ld rows hidden_dim vocab ids status ws stream */
  NEED(11);
  void *h, *w, *o[3], *st;
  int64_t ldh, ldw;
  int32_t v[3];
  size_t ws_bytes;
  TRY(get_ptr(a[0], &h) || get_i64(a[1], &ldh) || get_ptr(a[2], &w) || get_i64(a[3], &ldw));
  for (int i = 0; i < 3; ++i) TRY(get_i32(a[4 + i], v + i));
  TRY(get_ptrs(a, 7, 3, o) || get_bytes(a[9], &ws_bytes) || get_stream(a[10], &st));
  CALL(clv_lm_head_argmax(h, ldh, w, ldw, v[0], v[1], v[2], o[0], o[1], o[2], ws_bytes, st));
}

static PyObject *verify_step_host(ARGS) { /* shape cache in out ctx_len max_ctx scale staging ws stream */
  NEED(10);
  void *shape, *cache, *in, *out, *ctx, *stage, *ws, *st;
  int32_t max_ctx;
  float scale;
  size_t stage_bytes, ws_bytes;
  TRY(get_struct(a[0], sizeof(clv_shape), &shape) || get_struct(a[1], sizeof(clv_kv_cache), &cache));
  TRY(get_struct(a[2], sizeof(clv_host_inputs), &in) || get_struct(a[3], sizeof(clv_host_outputs), &out));
  TRY(get_ptr(a[4], &ctx) || get_i32(a[5], &max_ctx) || get_f32(a[6], &scale));
  TRY(get_ptr(a[7], &stage) || get_bytes(a[7], &stage_bytes) || get_ptr(a[8], &ws) || get_bytes(a[8], &ws_bytes));
  TRY(get_stream(a[9], &st));
  CALL(clv_verify_step_host(shape, cache, in, out, ctx, max_ctx, scale, stage, stage_bytes, ws, ws_bytes, st));
}

static PyObject *init(ARGS) { /* the two functions that name the current stream */
  NEED(2);
  Py_INCREF(a[0]);
  Py_INCREF(a[1]);
  Py_XSETREF(g_get_device, a[0]);
  Py_XSETREF(g_get_raw_stream, a[1]);
  Py_RETURN_NONE;
}

#define ENTRY(name) {#name, (PyCFunction)(void (*)(void))name, METH_FASTCALL, NULL}
static PyMethodDef methods[] = {ENTRY(init), ENTRY(tree_attn), ENTRY(accept_argmax), ENTRY(accept_argmax_noalloc),
                                ENTRY(accept_walk), ENTRY(kv_commit), ENTRY(accept_walk_commit), ENTRY(accept_sample),
                                ENTRY(tree_to_intervals), ENTRY(tree_from_intervals), ENTRY(kv_commit_layers),
                                ENTRY(draft_head_step), ENTRY(build_token_tree), ENTRY(lm_head_argmax),
                                ENTRY(verify_step_host), {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_calls", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__calls(void) {
  s_data_ptr = PyUnicode_InternFromString("data_ptr");
  s_nbytes = PyUnicode_InternFromString("nbytes");
  s_cuda_stream = PyUnicode_InternFromString("cuda_stream");
  if (!s_data_ptr || !s_nbytes || !s_cuda_stream) return NULL;
  return PyModule_Create(&module);
}
