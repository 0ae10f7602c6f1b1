/* The binding's hot calls without ctypes: Python objects -> C structs -> libpard, in native code.
 *
 * A planning call of one small pipeline runs for some 25 us on the device; marshalling its 26
 * pointers through ctypes took 5.5 us of host time and the goodput call behind it 5.7.  Here an
 * attribute lookup and a data_ptr() call per array are left: about 1.5 us and 1 us.
 * The library is the one binding.py has loaded (same path, looked up with dlopen/dlsym); the global
 * interpreter lock is released while it runs. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <dlfcn.h>
#include <stdint.h>

#include "pard.h"

static __typeof__(&pard_plan) f_plan;
static __typeof__(&pard_plan_host) f_plan_host;
static __typeof__(&pard_plan_policy) f_plan_policy;
static __typeof__(&pard_plan_static) f_plan_static;
static __typeof__(&pard_plan_status) f_plan_status;
static __typeof__(&pard_goodput) f_goodput;
static __typeof__(&pard_estimate_w) f_estimate_w;
static __typeof__(&pard_update_priority) f_update_priority;
static __typeof__(&pard_update_queue_delay) f_update_queue_delay;
static __typeof__(&pard_advance_state) f_advance_state;

static PyObject *s_data_ptr, *s_addr, *s_numel, *s_element_size;
enum { kStateArrays = 8, kOutArrays = 7 };
static const char* const kStateNames[kStateArrays] = {"pipeline_of_ctx", "now_us", "batch", "free_at_us",
                                                      "q_us", "w_us", "workers", "priority"};
static const char* const kOutNames[kOutArrays] = {"keep", "est_us", "perm", "kept_idx", "n_kept", "seg_offsets", "seg_kept"};
static PyObject *s_state[kStateArrays], *s_out[kOutArrays], *s_stage_stride, *s_slot_stride;

/* address of a torch tensor or numpy array; None is NULL */
static int ptr_of(PyObject* o, void** p) {
  *p = NULL;
  if (o == Py_None) return 0;
  if (PyObject_CheckBuffer(o)) {
    Py_buffer b;
    if (PyObject_GetBuffer(o, &b, PyBUF_STRIDES)) return -1;
    *p = b.buf;
    PyBuffer_Release(&b);
    return 0;
  }
  PyObject* r = PyObject_CallMethodNoArgs(o, s_data_ptr);
  if (!r) return -1;
  *p = PyLong_AsVoidPtr(r);
  Py_DECREF(r);
  return *p == NULL && PyErr_Occurred() ? -1 : 0;
}

static int ptr_attr(PyObject* o, PyObject* name, void* field) {
  PyObject* a = PyObject_GetAttr(o, name);
  if (!a) return -1;
  const int rc = ptr_of(a, (void**)field);
  Py_DECREF(a);
  return rc;
}

static int int_attr(PyObject* o, PyObject* name, int32_t* field) {
  PyObject* a = PyObject_GetAttr(o, name);
  if (!a) return -1;
  *field = (int32_t)PyLong_AsLong(a);
  Py_DECREF(a);
  return PyErr_Occurred() ? -1 : 0;
}

static int state_of(PyObject* o, pard_queue_state_t* st) {
  void* const to[kStateArrays] = {&st->d_pipeline_of_ctx, &st->d_now_us, &st->d_batch, &st->d_free_at_us,
                                  &st->d_q_us, &st->d_w_us, &st->d_workers, &st->d_priority};
  if (int_attr(o, s_stage_stride, &st->stage_stride) || int_attr(o, s_slot_stride, &st->slot_stride)) return -1;
  for (int i = 0; i < kStateArrays; ++i)
    if (ptr_attr(o, s_state[i], to[i])) return -1;
  return 0;
}

static int out_of(PyObject* o, pard_plan_out_t* out) {
  void* const to[kOutArrays] = {&out->d_keep, &out->d_est_us, &out->d_perm, &out->d_kept_idx,
                                &out->d_n_kept, &out->d_seg_offsets, &out->d_seg_kept};
  for (int i = 0; i < kOutArrays; ++i)
    if (ptr_attr(o, s_out[i], to[i])) return -1;
  return 0;
}

/* the handles of a sequence of pipelines; up to kOnStack need no allocation */
enum { kOnStack = 64 };
typedef struct {
  const pard_pipeline_t* few[kOnStack];
  const pard_pipeline_t** h;
  uint32_t n;
} handles_t;

static int handles_of(PyObject* seq, handles_t* out) {
  PyObject* fast = PySequence_Fast(seq, "pipelines: a sequence is wanted");
  out->h = out->few;
  if (!fast) return -1;
  const Py_ssize_t n = PySequence_Fast_GET_SIZE(fast);
  out->n = (uint32_t)n;
  if (n > kOnStack && !(out->h = PyMem_Malloc(sizeof(*out->h) * (size_t)n))) {
    out->h = out->few;
    Py_DECREF(fast);
    PyErr_NoMemory();
    return -1;
  }
  for (Py_ssize_t i = 0; i < n; ++i) {
    PyObject* a = PyObject_GetAttr(PySequence_Fast_GET_ITEM(fast, i), s_addr);
    if (!a) break;
    out->h[i] = PyLong_AsVoidPtr(a);
    Py_DECREF(a);
  }
  Py_DECREF(fast);
  return PyErr_Occurred() ? -1 : 0;
}

static void handles_free(handles_t* h) {
  if (h->h != h->few) PyMem_Free(h->h);
}

/* an integer argument, reduced modulo 2^64 as ctypes does */
static uint64_t u64(PyObject* o) { return PyLong_AsUnsignedLongLongMask(o); }

/* size of the workspace: given, or that of the tensor */
static int bytes_of(PyObject* given, PyObject* ws, uint64_t* n) {
  if (given != Py_None) { *n = u64(given); return PyErr_Occurred() ? -1 : 0; }
  PyObject* a = PyObject_CallMethodNoArgs(ws, s_numel);
  PyObject* b = a ? PyObject_CallMethodNoArgs(ws, s_element_size) : NULL;
  if (b) *n = u64(a) * u64(b);
  Py_XDECREF(a);
  Py_XDECREF(b);
  return b && !PyErr_Occurred() ? 0 : -1;
}

#define WANT(k) \
  if (n != (k)) { PyErr_SetString(PyExc_TypeError, "wrong number of arguments"); return NULL; }
#define RUN(call)          \
  int rc;                  \
  Py_BEGIN_ALLOW_THREADS;  \
  rc = (call);             \
  Py_END_ALLOW_THREADS

/* (which, pipelines, requests, arrivals, n, state, n_ctx, mode, out, workspace, workspace_bytes, stream);
 * which: 0 pard_plan, 1 pard_plan_policy, 2 pard_plan_host, 3 pard_plan_static */
static PyObject* py_plan(PyObject* self, PyObject* const* v, Py_ssize_t n) {
  (void)self;
  WANT(12);
  handles_t h;
  pard_queue_state_t st;
  pard_plan_out_t out;
  void *req, *arr, *ws;
  uint64_t wb = 0;
  const long which = PyLong_AsLong(v[0]);
  if (handles_of(v[1], &h) || ptr_of(v[2], &req) || ptr_of(v[3], &arr) || state_of(v[5], &st) || out_of(v[8], &out) ||
      ptr_of(v[9], &ws) || (which != 3 && bytes_of(v[10], v[9], &wb))) {
    handles_free(&h);
    return NULL;
  }
  const uint64_t count = u64(v[4]);
  const uint32_t n_ctx = (uint32_t)u64(v[6]), mode = (uint32_t)u64(v[7]);
  void* stream = (void*)(uintptr_t)u64(v[11]);
  if (PyErr_Occurred()) { handles_free(&h); return NULL; }
  RUN(which == 0   ? f_plan(h.h, h.n, req, count, &st, n_ctx, mode, &out, ws, wb, stream)
      : which == 1 ? f_plan_policy(h.h, h.n, req, arr, count, &st, n_ctx, mode, &out, ws, wb, stream)
      : which == 2 ? f_plan_host(h.h, h.n, req, count, &st, n_ctx, mode, &out, ws, wb, stream)
                   : f_plan_static(h.h, h.n, req, count, &st, n_ctx, mode, &out, stream));
  handles_free(&h);
  return PyLong_FromLong(rc);
}

/* (workspace, stream) */
static PyObject* py_status(PyObject* self, PyObject* const* v, Py_ssize_t n) {
  (void)self;
  WANT(2);
  void* ws;
  if (ptr_of(v[0], &ws)) return NULL;
  void* stream = (void*)(uintptr_t)u64(v[1]);
  if (PyErr_Occurred()) return NULL;
  RUN(f_plan_status(ws, stream));
  return PyLong_FromLong(rc);
}

/* (keep, seg_offsets, seg_kept, n, n_ctx, stage_stride, out_total, out_kept, stream) */
static PyObject* py_goodput(PyObject* self, PyObject* const* v, Py_ssize_t n) {
  (void)self;
  WANT(9);
  void *keep, *off, *kept, *total, *out;
  if (ptr_of(v[0], &keep) || ptr_of(v[1], &off) || ptr_of(v[2], &kept) || ptr_of(v[6], &total) || ptr_of(v[7], &out)) return NULL;
  const uint64_t count = u64(v[3]);
  const uint32_t n_ctx = (uint32_t)u64(v[4]);
  const int32_t S = (int32_t)u64(v[5]);
  void* stream = (void*)(uintptr_t)u64(v[8]);
  if (PyErr_Occurred()) return NULL;
  RUN(f_goodput(keep, off, kept, count, n_ctx, S, total, out, stream));
  return PyLong_FromLong(rc);
}

/* (pipelines, pipeline_of_ctx, n_ctx, stage_stride, slot_stride, samples, n_samples, lambda_num, lambda_den, seed,
 *  mode, w, workspace, workspace_bytes, stream) */
static PyObject* py_estimate_w(PyObject* self, PyObject* const* v, Py_ssize_t n) {
  (void)self;
  WANT(15);
  handles_t h;
  void *poc, *samples, *w, *ws;
  uint64_t wb, x[15];
  if (handles_of(v[0], &h) || ptr_of(v[1], &poc) || ptr_of(v[5], &samples) || ptr_of(v[11], &w) || ptr_of(v[12], &ws) ||
      bytes_of(v[13], v[12], &wb)) {
    handles_free(&h);
    return NULL;
  }
  static const int at[] = {2, 3, 4, 6, 7, 8, 9, 10, 14};
  for (unsigned i = 0; i < sizeof(at) / sizeof(at[0]); ++i) x[at[i]] = u64(v[at[i]]);
  if (PyErr_Occurred()) { handles_free(&h); return NULL; }
  RUN(f_estimate_w(h.h, h.n, poc, (uint32_t)x[2], (int32_t)x[3], (int32_t)x[4], samples, (uint32_t)x[6], (uint32_t)x[7],
                   (uint32_t)x[8], x[9], (uint32_t)x[10], w, ws, wb, (void*)(uintptr_t)x[14]));
  handles_free(&h);
  return PyLong_FromLong(rc);
}

/* (pipelines, pipeline_of_ctx, n_ctx, stage_stride, batch, workers, arrivals, n_hist, window, interval_us, mode,
 *  priority, workspace, workspace_bytes, stream) */
static PyObject* py_update_priority(PyObject* self, PyObject* const* v, Py_ssize_t n) {
  (void)self;
  WANT(15);
  handles_t h;
  void *poc, *batch, *workers, *arrivals, *priority, *ws;
  uint64_t wb, x[15];
  if (handles_of(v[0], &h) || ptr_of(v[1], &poc) || ptr_of(v[4], &batch) || ptr_of(v[5], &workers) ||
      ptr_of(v[6], &arrivals) || ptr_of(v[11], &priority) || ptr_of(v[12], &ws) || bytes_of(v[13], v[12], &wb)) {
    handles_free(&h);
    return NULL;
  }
  static const int at[] = {2, 3, 7, 8, 9, 10, 14};
  for (unsigned i = 0; i < sizeof(at) / sizeof(at[0]); ++i) x[at[i]] = u64(v[at[i]]);
  if (PyErr_Occurred()) { handles_free(&h); return NULL; }
  RUN(f_update_priority(h.h, h.n, poc, (uint32_t)x[2], (int32_t)x[3], batch, workers, arrivals, (uint32_t)x[7], (uint32_t)x[8],
                        (uint32_t)x[9], (uint32_t)x[10], priority, ws, wb, (void*)(uintptr_t)x[14]));
  handles_free(&h);
  return PyLong_FromLong(rc);
}

/* (n_ctx, stage_stride, now, sample_time, sample_delay, n_samples, window_us, mode, q, workspace, workspace_bytes, stream) */
static PyObject* py_update_queue_delay(PyObject* self, PyObject* const* v, Py_ssize_t n) {
  (void)self;
  WANT(12);
  void *now, *t, *d, *q, *ws;
  uint64_t wb, x[12];
  if (ptr_of(v[2], &now) || ptr_of(v[3], &t) || ptr_of(v[4], &d) || ptr_of(v[8], &q) || ptr_of(v[9], &ws) ||
      bytes_of(v[10], v[9], &wb))
    return NULL;
  static const int at[] = {0, 1, 5, 6, 7, 11};
  for (unsigned i = 0; i < sizeof(at) / sizeof(at[0]); ++i) x[at[i]] = u64(v[at[i]]);
  if (PyErr_Occurred()) return NULL;
  RUN(f_update_queue_delay((uint32_t)x[0], (int32_t)x[1], now, t, d, (uint32_t)x[5], (uint32_t)x[6], (uint32_t)x[7], q, ws, wb,
                           (void*)(uintptr_t)x[11]));
  return PyLong_FromLong(rc);
}

/* (pipelines, pipeline_of_ctx, n_ctx, stage_stride, now, batch, workers, seg_kept, free_at, sample_time, sample_delay,
 *  n_samples, slot, mode, workspace, workspace_bytes, stream) */
static PyObject* py_advance_state(PyObject* self, PyObject* const* v, Py_ssize_t n) {
  (void)self;
  WANT(17);
  handles_t h;
  void *poc, *now, *batch, *workers, *kept, *free_at, *t, *d, *ws;
  uint64_t wb, x[17];
  if (handles_of(v[0], &h) || ptr_of(v[1], &poc) || ptr_of(v[4], &now) || ptr_of(v[5], &batch) || ptr_of(v[6], &workers) ||
      ptr_of(v[7], &kept) || ptr_of(v[8], &free_at) || ptr_of(v[9], &t) || ptr_of(v[10], &d) || ptr_of(v[14], &ws) ||
      bytes_of(v[15], v[14], &wb)) {
    handles_free(&h);
    return NULL;
  }
  static const int at[] = {2, 3, 11, 12, 13, 16};
  for (unsigned i = 0; i < sizeof(at) / sizeof(at[0]); ++i) x[at[i]] = u64(v[at[i]]);
  if (PyErr_Occurred()) { handles_free(&h); return NULL; }
  RUN(f_advance_state(h.h, h.n, poc, (uint32_t)x[2], (int32_t)x[3], now, batch, workers, kept, free_at, t, d, (uint32_t)x[11],
                      (uint32_t)x[12], (uint32_t)x[13], ws, wb, (void*)(uintptr_t)x[16]));
  handles_free(&h);
  return PyLong_FromLong(rc);
}

/* (path of libpard.so): the entry points, from the library as it is already loaded */
static PyObject* py_bind(PyObject* self, PyObject* path) {
  (void)self;
  const char* p = PyUnicode_AsUTF8(path);
  if (!p) return NULL;
  void* lib = dlopen(p, RTLD_NOW);
  if (!lib) return PyErr_Format(PyExc_RuntimeError, "%s", dlerror());
#define GET(f, name)                                        \
  if (!(*(void**)&f = dlsym(lib, #name)))                   \
    return PyErr_Format(PyExc_RuntimeError, "%s lacks %s", p, #name)
  GET(f_plan, pard_plan);
  GET(f_plan_host, pard_plan_host);
  GET(f_plan_policy, pard_plan_policy);
  GET(f_plan_static, pard_plan_static);
  GET(f_plan_status, pard_plan_status);
  GET(f_goodput, pard_goodput);
  GET(f_estimate_w, pard_estimate_w);
  GET(f_update_priority, pard_update_priority);
  GET(f_update_queue_delay, pard_update_queue_delay);
  GET(f_advance_state, pard_advance_state);
#undef GET
  Py_RETURN_NONE;
}

#define FAST(name, f) {name, (PyCFunction)(void (*)(void))f, METH_FASTCALL, NULL}
static PyMethodDef methods[] = {{"bind", py_bind, METH_O, NULL},
                                FAST("plan", py_plan),
                                FAST("status", py_status),
                                FAST("goodput", py_goodput),
                                FAST("estimate_w", py_estimate_w),
                                FAST("update_priority", py_update_priority),
                                FAST("update_queue_delay", py_update_queue_delay),
                                FAST("advance_state", py_advance_state),
                                {NULL, NULL, 0, NULL}};

static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_pardcall", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__pardcall(void) {
  s_data_ptr = PyUnicode_InternFromString("data_ptr");
  s_addr = PyUnicode_InternFromString("addr");
  s_numel = PyUnicode_InternFromString("numel");
  s_element_size = PyUnicode_InternFromString("element_size");
  s_stage_stride = PyUnicode_InternFromString("stage_stride");
  s_slot_stride = PyUnicode_InternFromString("slot_stride");
  for (int i = 0; i < kStateArrays; ++i) s_state[i] = PyUnicode_InternFromString(kStateNames[i]);
  for (int i = 0; i < kOutArrays; ++i) s_out[i] = PyUnicode_InternFromString(kOutNames[i]);
  return PyModule_Create(&module);
}
