/* Argument marshalling of the calls a training loop makes every tick, as a CPython extension: snapshots in and out of their
 * ctypes structures, numpy arrays by the buffer protocol, the results as Python objects.  Through ctypes alone these calls
 * cost the host more than the library's own work (measured per call, ctypes -> here: pull 0.9 -> 0.3 us, reserve 3.6 -> 0.9,
 * enqueue 9 -> 2, apply 5 -> 1.5, the grad step's arguments 20 -> 8).  Arrays that already have their type and layout are read
 * where they lie, and a list of versions is read element by element: only the rest goes through numpy.  No step of the method
 * happens here. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>
#include <string.h>

#include "ps.h"

static int32_t (*f_pull)(ps_ctx*, int32_t, int32_t, ps_snapshot*);
static int32_t (*f_reserve)(ps_ctx*, int32_t, int64_t*);
static int32_t (*f_grad)(ps_ctx*, int32_t, int32_t, const ps_snapshot*, const int32_t*, const float*, const int32_t*, uint64_t,
                         uint64_t, const int64_t*, float*, float*, int32_t*);
static int32_t (*f_summed)(ps_ctx*, int32_t, int32_t, const ps_snapshot*, const int32_t*, const float*, const int32_t*, uint64_t,
                           uint64_t, float*, float*, int32_t*);
static int32_t (*f_eval)(ps_ctx*, int32_t, int32_t, const ps_snapshot*, const float*, const int32_t*, float*, int32_t*, int32_t*);
static int32_t (*f_enqueue)(ps_ctx*, int32_t, const int64_t*, const float*, const int32_t*, const uint64_t*, uint64_t);
static int32_t (*f_apply)(ps_ctx*, ps_mode, float, float, const int32_t*, ps_apply_result*);
static int32_t (*f_apply_stale)(ps_ctx*, ps_mode, float, float, const int32_t*, float, float, ps_apply_result*);
static int32_t (*f_apply_summed)(ps_ctx*, const float*, int32_t, float, float, ps_apply_result*);
static const char* (*f_error)(ps_ctx*);
static PyObject *snapshot_type, *error_type;
static PyObject *as_array;       /* as_array(object, kind): numpy's conversion to a contiguous array */
static PyObject *as_snapshots;   /* as_snapshots(sequence, n): ctypes' conversion to an array of n structures */
static PyObject *k_applied, *k_version, *k_checkpointed, *k_replicated;

static PyObject* raise(int32_t rc) {
  PyObject* e = PyObject_CallFunction(error_type, "is", (int)rc, f_error(NULL));
  if (e) { PyErr_SetObject(error_type, e); Py_DECREF(e); }
  return NULL;
}

/* Integer arguments: anything int() takes, wrapped like a C conversion, as ctypes does it. */
static int as_u64(PyObject* o, uint64_t* v) {
  PyObject* i = PyNumber_Long(o);
  if (!i) return -1;
  *v = PyLong_AsUnsignedLongLongMask(i);
  Py_DECREF(i);
  return PyErr_Occurred() ? -1 : 0;
}
static int i32(PyObject* o, int32_t* v) {
  uint64_t w;
  if (as_u64(o, &w)) return -1;
  *v = (int32_t)(uint32_t)w;
  return 0;
}
static int as_ptr(PyObject* o, void** p) {         /* None or an address */
  if (o == Py_None) { *p = NULL; return 0; }
  *p = PyLong_AsVoidPtr(o);
  return !*p && PyErr_Occurred() ? -1 : 0;
}
static int as_float(PyObject* o, float* v) {       /* anything float() takes */
  PyObject* f = PyNumber_Float(o);
  if (!f) return -1;
  *v = (float)PyFloat_AS_DOUBLE(f);
  Py_DECREF(f);
  return 0;
}

/* The types of the library's integer arrays. */
enum { I32, I64, U64 };

/* A contiguous one-dimensional array of the given type, or None.  The buffer keeps whatever holds the items alive. */
static int array(PyObject* o, Py_buffer* b, int kind) {
  b->obj = NULL;
  b->buf = NULL;
  b->len = 0;
  if (o == Py_None) return 0;
  if (PyObject_CheckBuffer(o)) {
    if (PyObject_GetBuffer(o, b, PyBUF_C_CONTIGUOUS | PyBUF_FORMAT) == 0) {
      const char f = b->ndim == 1 && b->format && b->format[0] && !b->format[1] ? b->format[0] : 0;
      if (b->itemsize == (kind == I32 ? 4 : 8) && (kind == U64 ? f == 'L' || f == 'Q' : f == 'i' || f == 'l' || f == 'q')) return 0;
      PyBuffer_Release(b);
    } else PyErr_Clear();
  }
  PyObject* c = PyObject_CallFunction(as_array, "Oi", o, kind);
  if (!c) { b->obj = NULL; return -1; }
  const int rc = PyObject_GetBuffer(c, b, PyBUF_C_CONTIGUOUS);
  Py_DECREF(c);
  return rc;
}
static void done(Py_buffer* b) { if (b->obj) PyBuffer_Release(b); }

static int long_enough(const Py_buffer* b, Py_ssize_t n, Py_ssize_t item) {
  if (!b->obj || b->len >= n * item) return 1;
  PyErr_SetString(PyExc_ValueError, "array is too short");
  return 0;
}

/* The snapshots of a call, out of their structures.  Anything but a list or tuple of n Snapshots goes through ctypes, which
 * converts or refuses it. */
static int snapshots(PyObject* seq, Py_ssize_t n, ps_snapshot* out) {
  Py_buffer b;
  Py_ssize_t i = 0;
  if ((PyList_CheckExact(seq) || PyTuple_CheckExact(seq)) && PySequence_Fast_GET_SIZE(seq) == n) {
    for (; i < n; ++i) {
      PyObject* o = PySequence_Fast_GET_ITEM(seq, i);
      if ((PyObject*)Py_TYPE(o) != snapshot_type) break;
      if (PyObject_GetBuffer(o, &b, PyBUF_SIMPLE)) return -1;
      out[i] = *(const ps_snapshot*)b.buf;
      PyBuffer_Release(&b);
    }
    if (i == n) return 0;
  }
  PyObject* c = PyObject_CallFunction(as_snapshots, "On", seq, n);
  if (!c) return -1;
  const int rc = PyObject_GetBuffer(c, &b, PyBUF_SIMPLE);
  Py_DECREF(c);
  if (rc) return -1;
  memcpy(out, b.buf, (size_t)n * sizeof(ps_snapshot));
  PyBuffer_Release(&b);
  return 0;
}

static PyObject* result(const ps_apply_result* r) {
  PyObject* d = PyDict_New();
  PyObject* v[4] = {PyLong_FromLongLong(r->applied), PyLong_FromUnsignedLongLong(r->new_version), PyLong_FromLong(r->checkpointed), PyLong_FromLong(r->replicated)};
  PyObject* k[4] = {k_applied, k_version, k_checkpointed, k_replicated};
  int bad = !d;
  for (int i = 0; i < 4; ++i) {
    if (!v[i] || bad || PyDict_SetItem(d, k[i], v[i])) bad = 1;
    Py_XDECREF(v[i]);
  }
  if (bad) { Py_XDECREF(d); return NULL; }
  return d;
}

/* The other threads run while the library works (it may wait for room in a stream). */
#define CALL(expr) Py_BEGIN_ALLOW_THREADS rc = (expr); Py_END_ALLOW_THREADS
#define WANT(n) if (nargs != (n)) { PyErr_SetString(PyExc_TypeError, "wrong number of arguments"); return NULL; }

static PyObject* bind(PyObject* m, PyObject* const* a, Py_ssize_t nargs) {
  WANT(5)
  static const struct { const char* name; void** f; } table[] = {
      {"ps_pull_snapshot", (void**)&f_pull}, {"ps_queue_reserve", (void**)&f_reserve}, {"workers_grad_step", (void**)&f_grad},
      {"workers_grad_step_summed", (void**)&f_summed}, {"workers_eval", (void**)&f_eval}, {"ps_enqueue", (void**)&f_enqueue},
      {"ps_apply", (void**)&f_apply}, {"ps_apply_stale", (void**)&f_apply_stale}, {"ps_apply_summed", (void**)&f_apply_summed}, {"ps_last_error", (void**)&f_error}};
  for (size_t i = 0; i < sizeof(table) / sizeof(table[0]); ++i) {
    PyObject* addr = PyDict_GetItemString(a[0], table[i].name);
    if (!addr) { PyErr_SetString(PyExc_KeyError, table[i].name); return NULL; }
    *table[i].f = PyLong_AsVoidPtr(addr);
    if (!*table[i].f) { if (!PyErr_Occurred()) PyErr_SetString(PyExc_ValueError, table[i].name); return NULL; }
  }
  Py_INCREF(a[1]);
  Py_XSETREF(snapshot_type, a[1]);
  Py_INCREF(a[2]);
  Py_XSETREF(error_type, a[2]);
  Py_INCREF(a[3]);
  Py_XSETREF(as_array, a[3]);
  Py_INCREF(a[4]);
  Py_XSETREF(as_snapshots, a[4]);
  Py_RETURN_NONE;
}

/* (ctx, worker, lag) -> Snapshot */
static PyObject* pull(PyObject* m, PyObject* const* a, Py_ssize_t nargs) {
  WANT(3)
  void* ctx;
  int32_t worker, lag;
  if (as_ptr(a[0], &ctx) || i32(a[1], &worker) || i32(a[2], &lag)) return NULL;
  PyObject* s = PyObject_CallNoArgs(snapshot_type);
  if (!s) return NULL;
  Py_buffer b;
  if (PyObject_GetBuffer(s, &b, PyBUF_WRITABLE)) { Py_DECREF(s); return NULL; }
  const int32_t rc = f_pull((ps_ctx*)ctx, worker, lag, (ps_snapshot*)b.buf);
  PyBuffer_Release(&b);
  if (rc) { Py_DECREF(s); return raise(rc); }
  return s;
}

/* (ctx, n, ids int64[n]) */
static PyObject* reserve(PyObject* m, PyObject* const* a, Py_ssize_t nargs) {
  WANT(3)
  void* ctx;
  int32_t n;
  Py_buffer b;
  if (as_ptr(a[0], &ctx) || i32(a[1], &n) || PyObject_GetBuffer(a[2], &b, PyBUF_WRITABLE)) return NULL;
  const int32_t rc = f_reserve((ps_ctx*)ctx, n, (int64_t*)b.buf);
  PyBuffer_Release(&b);
  if (rc) return raise(rc);
  Py_RETURN_NONE;
}

/* (ctx, W, b, snaps, worker_ids int32[W], x, y, seed, step, slot_ids int64[W] | None, grads | None, loss, argmax) */
static PyObject* grad_step(PyObject* m, PyObject* const* a, Py_ssize_t nargs) {
  WANT(13)
  void *ctx, *x, *y, *grads, *loss, *argmax;
  int32_t W, b;
  uint64_t seed, step;
  ps_snapshot snaps[PS_MAX_WORKERS];
  Py_buffer ids, slots;
  if (as_ptr(a[0], &ctx) || i32(a[1], &W) || i32(a[2], &b) || as_ptr(a[5], &x) || as_ptr(a[6], &y) || as_u64(a[7], &seed) ||
      as_u64(a[8], &step) || as_ptr(a[10], &grads) || as_ptr(a[11], &loss) || as_ptr(a[12], &argmax))
    return NULL;
  if (W <= PS_MAX_WORKERS && snapshots(a[3], W, snaps)) return NULL;      /* of more workers the library reads nothing: it refuses the call */
  if (array(a[4], &ids, I32)) return NULL;
  if (array(a[9], &slots, I64)) { done(&ids); return NULL; }
  if (!ids.obj || ids.ndim != 1 || ids.len != (Py_ssize_t)W * 4) PyErr_SetString(PyExc_AssertionError, "one worker id per worker is wanted");
  else long_enough(&slots, W, 8);
  if (PyErr_Occurred()) { done(&ids); done(&slots); return NULL; }
  int32_t rc;
  CALL(f_grad((ps_ctx*)ctx, W, b, snaps, (const int32_t*)ids.buf, (const float*)x, (const int32_t*)y, seed, step,
                            (const int64_t*)slots.buf, (float*)grads, (float*)loss, (int32_t*)argmax))
  done(&ids);
  done(&slots);
  if (rc) return raise(rc);
  Py_RETURN_NONE;
}

/* (ctx, W, b, snaps, worker_ids, x, y, seed, step, grad_sum, loss, argmax) */
static PyObject* grad_step_summed(PyObject* m, PyObject* const* a, Py_ssize_t nargs) {
  WANT(12)
  void *ctx, *x, *y, *sum, *loss, *argmax;
  int32_t W, b;
  uint64_t seed, step;
  ps_snapshot snaps[PS_MAX_WORKERS];
  Py_buffer ids;
  if (as_ptr(a[0], &ctx) || i32(a[1], &W) || i32(a[2], &b) || as_ptr(a[5], &x) || as_ptr(a[6], &y) || as_u64(a[7], &seed) ||
      as_u64(a[8], &step) || as_ptr(a[9], &sum) || as_ptr(a[10], &loss) || as_ptr(a[11], &argmax))
    return NULL;
  if (W <= PS_MAX_WORKERS && snapshots(a[3], W, snaps)) return NULL;
  if (array(a[4], &ids, I32)) return NULL;
  if (!long_enough(&ids, W, 4)) { done(&ids); return NULL; }
  int32_t rc;
  CALL(f_summed((ps_ctx*)ctx, W, b, snaps, (const int32_t*)ids.buf, (const float*)x, (const int32_t*)y, seed, step,
                              (float*)sum, (float*)loss, (int32_t*)argmax))
  done(&ids);
  if (rc) return raise(rc);
  Py_RETURN_NONE;
}

/* (ctx, W, b, snaps, x, y, loss, argmax, correct) */
static PyObject* eval(PyObject* m, PyObject* const* a, Py_ssize_t nargs) {
  WANT(9)
  void *ctx, *x, *y, *loss, *argmax, *correct;
  int32_t W, b;
  ps_snapshot snaps[PS_MAX_WORKERS];
  if (as_ptr(a[0], &ctx) || i32(a[1], &W) || i32(a[2], &b) || as_ptr(a[4], &x) || as_ptr(a[5], &y) || as_ptr(a[6], &loss) ||
      as_ptr(a[7], &argmax) || as_ptr(a[8], &correct))
    return NULL;
  if (W <= PS_MAX_WORKERS && snapshots(a[3], W, snaps)) return NULL;
  int32_t rc;
  CALL(f_eval((ps_ctx*)ctx, W, b, snaps, (const float*)x, (const int32_t*)y, (float*)loss, (int32_t*)argmax, (int32_t*)correct))
  if (rc) return raise(rc);
  Py_RETURN_NONE;
}

/* A list of versions, read without an array in between; NULL without an error if it is anything else. */
static uint64_t* version_list(PyObject* o, Py_ssize_t n) {
  if (!PyList_CheckExact(o) || PyList_GET_SIZE(o) < n) return NULL;
  uint64_t* v = PyMem_Malloc((size_t)(n ? n : 1) * sizeof(uint64_t));
  for (Py_ssize_t i = 0; v && i < n; ++i) {
    PyObject* e = PyList_GET_ITEM(o, i);
    v[i] = PyLong_CheckExact(e) ? PyLong_AsUnsignedLongLong(e) : (uint64_t)-1;
    if (v[i] == (uint64_t)-1) { PyErr_Clear(); PyMem_Free(v); return NULL; }
  }
  return v;
}

/* (ctx, slot_ids int64[n] | None, grads | None, worker_ids int32[n], base_versions uint64[n], step) */
static PyObject* enqueue(PyObject* m, PyObject* const* a, Py_ssize_t nargs) {
  WANT(6)
  void *ctx, *grads;
  uint64_t step;
  Py_buffer slots = {0}, ids = {0}, base = {0};
  uint64_t* list = NULL;
  PyObject* ret = NULL;
  if (as_ptr(a[0], &ctx) || as_ptr(a[2], &grads) || as_u64(a[5], &step)) return NULL;
  if (a[3] == Py_None || a[4] == Py_None) { PyErr_SetString(PyExc_TypeError, "worker_ids and base_versions are wanted"); return NULL; }
  if (array(a[3], &ids, I32) || array(a[1], &slots, I64)) goto end;
  const Py_ssize_t n = ids.shape[0];
  if (!(list = version_list(a[4], n)) && array(a[4], &base, U64)) goto end;
  if (!long_enough(&slots, n, 8) || !long_enough(&base, n, 8)) goto end;
  int32_t rc;
  CALL(f_enqueue((ps_ctx*)ctx, (int32_t)n, (const int64_t*)slots.buf, (const float*)grads, (const int32_t*)ids.buf,
                 list ? list : (const uint64_t*)base.buf, step))
  ret = rc ? raise(rc) : Py_NewRef(Py_None);
end:
  PyMem_Free(list);
  done(&slots);
  done(&ids);
  done(&base);
  return ret;
}

/* (ctx, mode, lr, scale, order int32[K] | None) -> dict */
static PyObject* apply(PyObject* m, PyObject* const* a, Py_ssize_t nargs) {
  WANT(5)
  void* ctx;
  int32_t mode;
  float lr, scale;
  Py_buffer order;
  ps_apply_result r = {0, 0, 0, 0};
  if (as_ptr(a[0], &ctx) || i32(a[1], &mode) || as_float(a[2], &lr) || as_float(a[3], &scale) || array(a[4], &order, I32)) return NULL;
  int32_t rc;
  CALL(f_apply((ps_ctx*)ctx, (ps_mode)mode, lr, scale, (const int32_t*)order.buf, &r))
  done(&order);
  return rc ? raise(rc) : result(&r);
}

/* (ctx, mode, lr, scale, order int32[K] | None, clip_norm, staleness_alpha) -> dict */
static PyObject* apply_stale(PyObject* m, PyObject* const* a, Py_ssize_t nargs) {
  WANT(7)
  void* ctx;
  int32_t mode;
  float lr, scale, clip, alpha;
  Py_buffer order;
  ps_apply_result r = {0, 0, 0, 0};
  if (as_ptr(a[0], &ctx) || i32(a[1], &mode) || as_float(a[2], &lr) || as_float(a[3], &scale) || as_float(a[5], &clip) ||
      as_float(a[6], &alpha) || array(a[4], &order, I32))
    return NULL;
  int32_t rc;
  CALL(f_apply_stale((ps_ctx*)ctx, (ps_mode)mode, lr, scale, (const int32_t*)order.buf, clip, alpha, &r))
  done(&order);
  return rc ? raise(rc) : result(&r);
}

/* (ctx, grad_sum, n_workers, lr, scale) -> dict */
static PyObject* apply_summed(PyObject* m, PyObject* const* a, Py_ssize_t nargs) {
  WANT(5)
  void *ctx, *sum;
  int32_t n;
  float lr, scale;
  ps_apply_result r = {0, 0, 0, 0};
  if (as_ptr(a[0], &ctx) || as_ptr(a[1], &sum) || i32(a[2], &n) || as_float(a[3], &lr) || as_float(a[4], &scale)) return NULL;
  int32_t rc;
  CALL(f_apply_summed((ps_ctx*)ctx, (const float*)sum, n, lr, scale, &r))
  return rc ? raise(rc) : result(&r);
}

#define FAST(f) {#f, (PyCFunction)(void (*)(void))f, METH_FASTCALL, NULL}
static PyMethodDef methods[] = {FAST(bind), FAST(pull), FAST(reserve), FAST(grad_step), FAST(grad_step_summed), FAST(eval),
                                FAST(enqueue), FAST(apply), FAST(apply_stale), FAST(apply_summed), {NULL, NULL, 0, NULL}};
static struct PyModuleDef def = {PyModuleDef_HEAD_INIT, "_marshal", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__marshal(void) {
  k_applied = PyUnicode_InternFromString("applied");
  k_version = PyUnicode_InternFromString("new_version");
  k_checkpointed = PyUnicode_InternFromString("checkpointed");
  k_replicated = PyUnicode_InternFromString("replicated");
  return PyModule_Create(&def);
}
