/* CPython entry to the device calls of libdasc that sit on a serving engine's path: argument marshalling only, like
 * binding.py, which uses it for these calls.  A ctypes call with ten to twenty-six arguments costs 4 to 8 us of interpreter
 * time on the host of a B200, more than the GPU needs for the smallest calls; here it is under 1 us.
 *
 * Tensors are taken as they are: None is a null pointer, an int an address, anything with a data_ptr() that; what an address
 * is for other objects binding.py says.  `stream` is None (torch's current stream) or has a cuda_stream attribute.  Every function
 * returns the dasc_status_t. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>

#include "dasc.h"

static PyObject *s_data_ptr, *s_numel, *s_element_size, *s_cuda_stream, *s_dtype;
static PyObject *g_raw_stream, *g_device, *g_bf16, *g_address; /* set by init() */

static int as_ptr(PyObject *o, void **out) {
  if (o == Py_None) {
    *out = NULL;
    return 0;
  }
  PyObject *v;
  if (PyLong_Check(o)) {
    v = Py_NewRef(o);
  } else {
    v = PyObject_CallMethodNoArgs(o, s_data_ptr);
    if (!v && PyErr_ExceptionMatches(PyExc_AttributeError)) {
      PyErr_Clear();
      v = PyObject_CallOneArg(g_address, o);
    }
    if (!v) return -1;
  }
  *out = PyLong_AsVoidPtr(v);
  Py_DECREF(v);
  return *out == NULL && PyErr_Occurred() ? -1 : 0;
}

/* A stride, a layer, an enumerator: whole numbers only, a float is an error and not cut off. */
static int as_index(PyObject *o, int64_t *out) {
  if (PyLong_Check(o)) {
    *out = PyLong_AsLongLong(o);
  } else {
    PyObject *v = PyNumber_Index(o);
    if (!v) return -1;
    *out = PyLong_AsLongLong(v);
    Py_DECREF(v);
  }
  return *out == -1 && PyErr_Occurred() ? -1 : 0;
}

/* A token count: whatever int() takes. */
static int as_count(PyObject *o, int64_t *out) {
  if (PyLong_Check(o)) {
    *out = PyLong_AsLongLong(o);
  } else {
    PyObject *v = PyNumber_Long(o);
    if (!v) return -1;
    *out = PyLong_AsLongLong(v);
    Py_DECREF(v);
  }
  return *out == -1 && PyErr_Occurred() ? -1 : 0;
}

static int method_i64(PyObject *o, PyObject *name, int64_t *out) {
  PyObject *v = PyObject_CallMethodNoArgs(o, name);
  if (!v) return -1;
  const int r = as_index(v, out);
  Py_DECREF(v);
  return r;
}

static int as_stream(PyObject *o, void **out) {
  PyObject *v;
  if (o == Py_None) {
    PyObject *dev = PyObject_CallNoArgs(g_device);
    if (!dev) return -1;
    v = PyObject_CallOneArg(g_raw_stream, dev);
    Py_DECREF(dev);
  } else {
    v = PyObject_GetAttr(o, s_cuda_stream);
  }
  if (!v) return -1;
  *out = PyLong_AsVoidPtr(v);
  Py_DECREF(v);
  return *out == NULL && PyErr_Occurred() ? -1 : 0;
}

/* DASC_IO_BF16 or DASC_IO_FP32 */
static int as_io(PyObject *o, int32_t *out) {
  *out = DASC_IO_FP32;
  if (o == Py_None) return 0;
  PyObject *v = PyObject_GetAttr(o, s_dtype);
  if (!v) return -1;
  if (v == g_bf16) *out = DASC_IO_BF16;
  Py_DECREF(v);
  return 0;
}

static int nbytes(PyObject *o, size_t *out) {
  *out = 0;
  if (o == Py_None) return 0;
  int64_t n, e;
  if (method_i64(o, s_numel, &n) || method_i64(o, s_element_size, &e)) return -1;
  *out = (size_t)(n * e);
  return 0;
}

static int arg_count(Py_ssize_t n, Py_ssize_t want) {
  if (n == want) return 0;
  PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, n);
  return -1;
}

/* raw_stream(device) -> cudaStream_t of torch's current stream, device() -> current device, torch.bfloat16, address(object) */
static PyObject *py_init(PyObject *self, PyObject *const *a, Py_ssize_t n) {
  if (arg_count(n, 4)) return NULL;
  Py_XSETREF(g_raw_stream, Py_NewRef(a[0]));
  Py_XSETREF(g_device, Py_NewRef(a[1]));
  Py_XSETREF(g_bf16, Py_NewRef(a[2]));
  Py_XSETREF(g_address, Py_NewRef(a[3]));
  Py_RETURN_NONE;
}

/* plan, state, layer_stride, req_stride, src_req, pool, pool_arg, dst_slot, stream; pool_arg: slot stride or slot count */
typedef dasc_status_t (*store_fn)(const dasc_plan_t *, const float *, int64_t, int64_t, const int32_t *, void *, int64_t,
                                  const int32_t *, int32_t, void *);
static PyObject *store_call(store_fn fn, PyObject *const *a, Py_ssize_t n) {
  void *plan, *state, *src, *pool, *dst, *stream;
  int64_t ls, rs, arg, pairs;
  if (arg_count(n, 9) || as_ptr(a[0], &plan) || as_ptr(a[1], &state) || as_index(a[2], &ls) || as_index(a[3], &rs) ||
      as_ptr(a[4], &src) || as_ptr(a[5], &pool) || as_index(a[6], &arg) || as_ptr(a[7], &dst) ||
      method_i64(a[4], s_numel, &pairs) || as_stream(a[8], &stream))
    return NULL;
  dasc_status_t st;
  Py_BEGIN_ALLOW_THREADS
  st = fn(plan, state, ls, rs, src, pool, arg, dst, (int32_t)pairs, stream);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(st);
}

/* plan, pool, pool_arg, src_slot, state, layer_stride, req_stride, dst_req, stream */
typedef dasc_status_t (*load_fn)(const dasc_plan_t *, const void *, int64_t, const int32_t *, float *, int64_t, int64_t,
                                 const int32_t *, int32_t, void *);
static PyObject *load_call(load_fn fn, PyObject *const *a, Py_ssize_t n) {
  void *plan, *state, *src, *pool, *dst, *stream;
  int64_t ls, rs, arg, pairs;
  if (arg_count(n, 9) || as_ptr(a[0], &plan) || as_ptr(a[1], &pool) || as_index(a[2], &arg) || as_ptr(a[3], &src) ||
      as_ptr(a[4], &state) || as_index(a[5], &ls) || as_index(a[6], &rs) || as_ptr(a[7], &dst) ||
      method_i64(a[3], s_numel, &pairs) || as_stream(a[8], &stream))
    return NULL;
  dasc_status_t st;
  Py_BEGIN_ALLOW_THREADS
  st = fn(plan, pool, arg, src, state, ls, rs, dst, (int32_t)pairs, stream);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(st);
}

#define COPY_CALL(name, kind, fn) \
  static PyObject *name(PyObject *self, PyObject *const *a, Py_ssize_t n) { return kind##_call((kind##_fn)fn, a, n); }
COPY_CALL(py_pack, store, dasc_pack)
COPY_CALL(py_pack_padded, store, dasc_pack_padded)
COPY_CALL(py_pack_int8, store, dasc_pack_int8)
COPY_CALL(py_restore, load, dasc_restore)
COPY_CALL(py_restore_padded, load, dasc_restore_padded)
COPY_CALL(py_restore_int8, load, dasc_restore_int8)

/* What the two refresh calls share: plan, state, layer_stride, req_stride, req_idx, q, k, v, g, beta, cu_seqlens, total_tokens,
 * bound (longest request or window), layer_begin, layer_end, q_scale, o, algo, workspace, stream */
struct refresh_args {
  void *plan, *state, *req, *q, *k, *v, *g, *beta, *cu, *o, *ws, *stream;
  int64_t ls, rs, total, bound, lb, le, algo, n_cu;
  int32_t io, o_io;
  float q_scale;
  size_t ws_bytes;
};
static int refresh_parse(struct refresh_args *r, PyObject *const *a, PyObject *io_from) {
  if (as_ptr(a[0], &r->plan) || as_ptr(a[1], &r->state) || as_index(a[2], &r->ls) || as_index(a[3], &r->rs) ||
      as_ptr(a[4], &r->req) || as_ptr(a[5], &r->q) || as_ptr(a[6], &r->k) || as_ptr(a[7], &r->v) || as_ptr(a[8], &r->g) ||
      as_ptr(a[9], &r->beta) || as_ptr(a[10], &r->cu) || method_i64(a[10], s_numel, &r->n_cu) || as_count(a[11], &r->total) ||
      as_count(a[12], &r->bound) || as_index(a[13], &r->lb) || as_index(a[14], &r->le) || as_ptr(a[16], &r->o) ||
      as_index(a[17], &r->algo) || as_ptr(a[18], &r->ws) || nbytes(a[18], &r->ws_bytes) || as_stream(a[19], &r->stream) ||
      as_io(io_from, &r->io) || as_io(a[16], &r->o_io))
    return -1;
  PyObject *s = PyNumber_Float(a[15]);
  if (!s) return -1;
  r->q_scale = (float)PyFloat_AS_DOUBLE(s);
  Py_DECREF(s);
  return 0;
}

/* the arguments above, then mode */
static PyObject *py_refresh(PyObject *self, PyObject *const *a, Py_ssize_t n) {
  struct refresh_args r;
  int64_t mode;
  if (arg_count(n, 21) || refresh_parse(&r, a, a[5]) || as_index(a[20], &mode)) return NULL;
  dasc_status_t st;
  Py_BEGIN_ALLOW_THREADS
  st = dasc_refresh(r.plan, r.state, r.ls, r.rs, r.req, r.q, r.k, r.v, r.io, r.g, r.beta, r.cu, (int32_t)(r.n_cu - 1), r.total,
                    (int32_t)r.bound, (int32_t)r.lb, (int32_t)r.le, r.q_scale, r.o, r.o_io, (int32_t)mode, (int32_t)r.algo, r.ws,
                    r.ws_bytes, r.stream);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(st);
}

/* the arguments above, then window_begin */
static PyObject *py_refresh_window(PyObject *self, PyObject *const *a, Py_ssize_t n) {
  struct refresh_args r;
  void *wb;
  if (arg_count(n, 21) || refresh_parse(&r, a, a[6]) || as_ptr(a[20], &wb)) return NULL;
  dasc_status_t st;
  Py_BEGIN_ALLOW_THREADS
  st = dasc_refresh_window(r.plan, r.state, r.ls, r.rs, r.req, r.q, r.k, r.v, r.io, r.g, r.beta, r.cu, (int32_t)(r.n_cu - 1),
                           r.total, r.bound, (int32_t)r.lb, (int32_t)r.le, r.q_scale, r.o, r.o_io, (int32_t)r.algo, wb, r.ws,
                           r.ws_bytes, r.stream);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(st);
}

#define M(name, fn) {name, (PyCFunction)(void (*)(void))fn, METH_FASTCALL, NULL}
static PyMethodDef methods[] = {
    M("init", py_init), M("pack", py_pack), M("pack_padded", py_pack_padded), M("pack_int8", py_pack_int8),
    M("restore", py_restore), M("restore_padded", py_restore_padded), M("restore_int8", py_restore_int8),
    M("refresh", py_refresh), M("refresh_window", py_refresh_window), {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_dasccall", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__dasccall(void) {
  s_data_ptr = PyUnicode_InternFromString("data_ptr");
  s_numel = PyUnicode_InternFromString("numel");
  s_element_size = PyUnicode_InternFromString("element_size");
  s_cuda_stream = PyUnicode_InternFromString("cuda_stream");
  s_dtype = PyUnicode_InternFromString("dtype");
  if (!s_data_ptr || !s_numel || !s_element_size || !s_cuda_stream || !s_dtype) return NULL;
  return PyModule_Create(&module);
}
