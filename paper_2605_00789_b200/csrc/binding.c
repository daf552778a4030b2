/* Argument marshalling of the Python binding (module _binding): tensors, views and plain values of one call go straight
 * into the C ABI's argument structs.  A call used to fill them field by field through ctypes (9 us for
 * lightkv_compress_layer, 6 for lightkv_compact_kv, more than the launches behind them take); here a tensor costs a
 * data_ptr() and a stride() call.  Needs no header of torch: tensors are Python objects with those two methods. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>
#include <string.h>

#include "lightkv.h"

typedef int (*layer_fn)(const lightkv_plan_t*, const lightkv_layer_args_t*);
typedef int (*kv_fn)(const lightkv_plan_t*, const lightkv_kv_args_t*);
static layer_fn g_layer, g_layer_builtin;
static kv_fn g_kv;
static PyObject *g_fail, *g_fork_join, *g_raw_stream, *g_device;   /* Python callables, see bind() */

/* names used as keywords, attributes or methods, interned once */
#define NAMES(X) \
  X(plan) X(stage) X(hidden) X(out) X(vis_begin) X(n_text_after) X(text_begin) X(text_end) X(q) X(k) X(lse) X(xi) \
  X(n_vis) X(pos) X(stream) X(trace_events) X(aux_stream) X(map_event) X(fork_event) X(join_event) X(text_ranges) \
  X(bidirectional) X(lse_out) X(seq_start) X(seq_start_out) X(hidden_out) X(k_src) X(v_src) X(k_dst) X(v_dst) X(mode) \
  X(page_size) X(src_block_table) X(dst_block_table) X(src_seq_start) X(dst_seq_start) X(data_ptr) X(size) \
  X(handle) X(value) X(n_vis_out) X(pos_out) X(dst) X(weight) X(grp_off) X(grp_src) X(xi_out) X(status) X(workspace) \
  X(info) X(workspace_bytes) X(cuda_stream) X(cuda_event)
enum {
#define X(n) N_##n,
  NAMES(X)
#undef X
  N_COUNT
};
static PyObject* g_name[N_COUNT];
static PyObject* g_stride;   /* "stride" */

/* value of keyword / positional argument `id`, NULL when absent or None */
typedef struct { PyObject* v[N_COUNT]; } Args;
static PyObject* get(const Args* a, int id) { return a->v[id] == Py_None ? NULL : a->v[id]; }

static int parse(Args* a, const char* fn, PyObject* const* args, Py_ssize_t nargs, PyObject* kwnames,
                 const int* positional, int n_pos, int n_required, const int* keywords, int n_kw) {
  memset(a, 0, sizeof(*a));
  if (nargs > n_pos) { PyErr_Format(PyExc_TypeError, "%s() takes %d positional arguments but %zd were given", fn, n_pos, nargs); return -1; }
  for (Py_ssize_t i = 0; i < nargs; ++i) a->v[positional[i]] = args[i];
  const Py_ssize_t n = kwnames ? PyTuple_GET_SIZE(kwnames) : 0;
  for (Py_ssize_t i = 0; i < n; ++i) {
    PyObject* name = PyTuple_GET_ITEM(kwnames, i);
    int id = -1;
    for (int pass = 0; pass < 2 && id < 0; ++pass) {          /* interned names are equal as pointers */
      for (int j = 0; j < n_kw + n_pos && id < 0; ++j) {
        const int c = j < n_kw ? keywords[j] : positional[j - n_kw];
        if (pass == 0 ? name == g_name[c] : PyUnicode_Compare(name, g_name[c]) == 0) id = c;
      }
    }
    if (id < 0) { PyErr_Format(PyExc_TypeError, "%s() got an unexpected keyword argument '%U'", fn, name); return -1; }
    if (a->v[id]) { PyErr_Format(PyExc_TypeError, "%s() got multiple values for argument '%U'", fn, name); return -1; }
    a->v[id] = args[nargs + i];
  }
  for (int j = 0; j < n_required; ++j)
    if (!a->v[positional[j]]) { PyErr_Format(PyExc_TypeError, "%s() missing required argument: '%U'", fn, g_name[positional[j]]); return -1; }
  if (!a->v[N_vis_begin]) { PyErr_Format(PyExc_TypeError, "%s() missing 1 required keyword-only argument: 'vis_begin'", fn); return -1; }
  return 0;
}

static int to_i64(PyObject* v, int64_t* r) {
  if (PyLong_CheckExact(v)) { *r = PyLong_AsLongLong(v); return *r == -1 && PyErr_Occurred() ? -1 : 0; }
  PyObject* i = PyNumber_Index(v);                            /* numpy integers and the like */
  if (!i) return -1;
  *r = PyLong_AsLongLong(i);
  Py_DECREF(i);
  return *r == -1 && PyErr_Occurred() ? -1 : 0;
}
static int int_arg(const Args* a, int id, int32_t fallback, int32_t* r) {
  PyObject* v = get(a, id);
  int64_t t = fallback;
  if (v && to_i64(v, &t)) return -1;
  if (t < INT32_MIN || t > INT32_MAX) { PyErr_Format(PyExc_OverflowError, "'%U' is out of range", g_name[id]); return -1; }
  *r = (int32_t)t;
  return 0;
}
/* integer attribute of an object as a pointer (stream and event handles, plan handles) */
static int ptr_attr(PyObject* o, int id, void** r) {
  PyObject* v = PyObject_GetAttr(o, g_name[id]);
  if (!v) return -1;
  *r = v == Py_None ? NULL : PyLong_AsVoidPtr(v);
  Py_DECREF(v);
  return !*r && PyErr_Occurred() ? -1 : 0;
}
/* address of a tensor's data; NULL object: NULL */
static int data(PyObject* t, void* r) {
  void* p = NULL;
  if (t) {
    PyObject* v = PyObject_CallMethodNoArgs(t, g_name[N_data_ptr]);
    if (!v) return -1;
    p = PyLong_AsVoidPtr(v);
    Py_DECREF(v);
    if (!p && PyErr_Occurred()) return -1;
  }
  memcpy(r, &p, sizeof(p));
  return 0;
}
static int data_attr(PyObject* o, int id, void* r) {
  PyObject* t = PyObject_GetAttr(o, g_name[id]);
  if (!t) return -1;
  const int rc = data(t == Py_None ? NULL : t, r);
  Py_DECREF(t);
  return rc;
}
/* the first n strides of a tensor */
static int strides(PyObject* t, int n, int64_t* r) {
  PyObject* v = PyObject_CallMethodNoArgs(t, g_stride);
  if (!v) return -1;
  int rc = PyTuple_Check(v) && PyTuple_GET_SIZE(v) >= n ? 0 : -1;
  if (rc) PyErr_Format(PyExc_IndexError, "a tensor of at least %d dimensions is expected", n);
  for (int i = 0; i < n && !rc; ++i) rc = to_i64(PyTuple_GET_ITEM(v, i), &r[i]);
  Py_DECREF(v);
  return rc;
}
static int size_of(PyObject* t, int dim, int32_t* r) {
  PyObject* d = PyLong_FromLong(dim);
  PyObject* v = d ? PyObject_CallMethodOneArg(t, g_name[N_size], d) : NULL;
  Py_XDECREF(d);
  if (!v) return -1;
  *r = (int32_t)PyLong_AsLong(v);
  Py_DECREF(v);
  return *r == -1 && PyErr_Occurred() ? -1 : 0;
}
static int stream_handle(PyObject* stream, void** r) {
  if (stream) return ptr_attr(stream, N_cuda_stream, r);
  PyObject* dev = PyObject_CallNoArgs(g_device);              /* the current stream of the current device */
  PyObject* v = dev ? PyObject_CallOneArg(g_raw_stream, dev) : NULL;
  Py_XDECREF(dev);
  if (!v) return -1;
  *r = PyLong_AsVoidPtr(v);
  Py_DECREF(v);
  return !*r && PyErr_Occurred() ? -1 : 0;
}
static int plan_handle(PyObject* plan, void** r) {
  PyObject* h = PyObject_GetAttr(plan, g_name[N_handle]);
  if (!h) return -1;
  int rc = 0;
  *r = NULL;
  if (h != Py_None) rc = ptr_attr(h, N_value, r);
  Py_DECREF(h);
  return rc;
}
static PyObject* done(int code, const char* what) {
  if (code == 0) Py_RETURN_NONE;
  return PyObject_CallFunction(g_fail, "is", code, what);     /* raises LightKVError */
}

static const int kLayerPos[] = {N_plan, N_stage, N_hidden, N_out};
static const int kLayerKw[] = {N_vis_begin, N_n_text_after, N_q, N_k, N_n_vis, N_pos, N_lse, N_xi, N_text_begin, N_text_end,
                               N_stream, N_aux_stream, N_map_event, N_fork_event, N_join_event, N_trace_events, N_text_ranges,
                               N_bidirectional, N_lse_out, N_seq_start, N_seq_start_out, N_hidden_out};

static PyObject* layer(const char* fn, layer_fn call, int builtin, PyObject* const* args, Py_ssize_t nargs, PyObject* kwnames) {
  Args in;
  if (parse(&in, fn, args, nargs, kwnames, kLayerPos, 4, 4, kLayerKw, sizeof(kLayerKw) / sizeof(int))) return NULL;
  lightkv_layer_args_t a;
  memset(&a, 0, sizeof(a));
  a.struct_size = sizeof(a);
  PyObject *out = in.v[N_out], *t;
  void* plan;
  int64_t s[3];
  int32_t ranges[2 * LIGHTKV_MAX_TEXT_RANGES];
  void* trace[LIGHTKV_TRACE_EVENTS];
  if (plan_handle(in.v[N_plan], &plan) || int_arg(&in, N_stage, 0, &a.stage) || int_arg(&in, N_vis_begin, 0, &a.vis_begin) ||
      int_arg(&in, N_n_text_after, 0, &a.n_text_after) || int_arg(&in, N_text_begin, 0, &a.text_begin) ||
      int_arg(&in, N_text_end, a.vis_begin, &a.text_end))
    return NULL;
  if (data(in.v[N_hidden], &a.hidden) || strides(in.v[N_hidden], 2, s)) return NULL;
  a.hidden_batch_stride = s[0]; a.hidden_row_stride = s[1];
  t = get(&in, N_hidden_out);
  if (!t) t = PyObject_GetAttr(out, g_name[N_hidden_out]); else Py_INCREF(t);
  if (!t) return NULL;
  int rc = data(t, &a.hidden_out) || strides(t, 2, s);
  Py_DECREF(t);
  if (rc) return NULL;
  a.hidden_out_batch_stride = s[0]; a.hidden_out_row_stride = s[1];
  if ((t = get(&in, N_q))) {
    if (data(t, &a.q) || strides(t, 3, s) || size_of(t, 2, &a.seq_rows)) return NULL;
    a.q_batch_stride = s[0]; a.q_head_stride = s[1]; a.q_row_stride = s[2];
  }
  if ((t = get(&in, N_k))) {
    if (data(t, &a.k) || strides(t, 3, s)) return NULL;
    a.k_batch_stride = s[0]; a.k_head_stride = s[1]; a.k_row_stride = s[2];
  }
  if ((t = get(&in, N_lse))) {
    if (data(t, &a.lse) || strides(t, 2, s)) return NULL;
    a.lse_batch_stride = s[0]; a.lse_head_stride = s[1];
  }
  if ((t = get(&in, N_lse_out))) {
    if (data(t, &a.lse_out) || strides(t, 2, s)) return NULL;
    a.lse_out_batch_stride = s[0]; a.lse_out_head_stride = s[1];
  }
  if (data(get(&in, N_xi), &a.xi) || data(get(&in, N_n_vis), &a.n_vis) || data(get(&in, N_pos), &a.pos) ||
      data_attr(out, N_n_vis_out, &a.n_vis_out) || data_attr(out, N_pos_out, &a.pos_out) || data_attr(out, N_dst, &a.dst) ||
      data_attr(out, N_weight, &a.weight) || data_attr(out, N_grp_off, &a.grp_off) || data_attr(out, N_grp_src, &a.grp_src) ||
      data_attr(out, N_xi_out, &a.xi_out) || data_attr(out, N_status, &a.status))
    return NULL;
  if (!builtin) {
    void* p;
    PyObject* info = PyObject_GetAttr(out, g_name[N_info]);
    PyObject* bytes = info ? PyObject_GetAttr(info, g_name[N_workspace_bytes]) : NULL;
    Py_XDECREF(info);
    if (!bytes) return NULL;
    a.workspace_bytes = PyLong_AsSize_t(bytes);
    Py_DECREF(bytes);
    if (PyErr_Occurred() || data_attr(out, N_workspace, &p)) return NULL;
    a.workspace = (void*)(((uintptr_t)p + 255) / 256 * 256);
  }
  if (stream_handle(get(&in, N_stream), &a.stream)) return NULL;
  if ((t = get(&in, N_aux_stream))) {
    PyObject *fork = get(&in, N_fork_event), *join = get(&in, N_join_event), *pair = NULL;
    if (ptr_attr(t, N_cuda_stream, &a.aux_stream)) return NULL;
    if (!fork || !join) {                                     /* a pair kept with the stage's buffers */
      pair = PyObject_CallOneArg(g_fork_join, out);
      if (!pair) return NULL;
      fork = PyTuple_GET_ITEM(pair, 0); join = PyTuple_GET_ITEM(pair, 1);
    }
    rc = ptr_attr(fork, N_cuda_event, &a.fork_event) || ptr_attr(join, N_cuda_event, &a.join_event);
    Py_XDECREF(pair);
    if (rc) return NULL;
  }
  if ((t = get(&in, N_text_ranges))) {                        /* [(begin, end), ...] */
    PyObject* seq = PySequence_Fast(t, "text_ranges is a sequence of (begin, end)");
    if (!seq) return NULL;
    const Py_ssize_t n = PySequence_Fast_GET_SIZE(seq);
    a.n_text_ranges = (int32_t)n;                             /* too many: the library refuses the count */
    a.text_ranges = ranges;
    for (Py_ssize_t i = 0; i < n && i < LIGHTKV_MAX_TEXT_RANGES && !rc; ++i)
      for (int e = 0; e < 2 && !rc; ++e) {
        PyObject* v = PySequence_GetItem(PySequence_Fast_GET_ITEM(seq, i), e);
        int64_t x = 0;
        rc = !v || to_i64(v, &x);
        Py_XDECREF(v);
        ranges[2 * i + e] = (int32_t)x;
      }
    Py_DECREF(seq);
    if (rc) return NULL;
  }
  if ((t = get(&in, N_bidirectional))) {
    a.bidirectional = PyObject_IsTrue(t);
    if (a.bidirectional < 0) return NULL;
  }
  if ((t = get(&in, N_seq_start))) {
    /* packed batch: tensors of shape [1, rows, ...] hold the samples back to back; sample b starts at row seq_start[b],
     * so the batch strides are 0 and q / k span all rows */
    if (data(t, &a.seq_start) || data(get(&in, N_seq_start_out), &a.seq_start_out)) return NULL;
    a.hidden_batch_stride = a.q_batch_stride = a.k_batch_stride = a.lse_batch_stride = a.lse_out_batch_stride = 0;
    if (a.seq_start_out) a.hidden_out_batch_stride = 0;
  }
  if ((t = get(&in, N_map_event)) && ptr_attr(t, N_cuda_event, &a.map_event)) return NULL;
  if ((t = get(&in, N_trace_events))) {
    PyObject* seq = PySequence_Fast(t, "trace_events is a sequence of events");
    if (!seq) return NULL;
    if (PySequence_Fast_GET_SIZE(seq) != LIGHTKV_TRACE_EVENTS) {
      PyErr_Format(PyExc_AssertionError, "%d trace events are expected", LIGHTKV_TRACE_EVENTS);
      rc = -1;
    }
    for (int i = 0; i < LIGHTKV_TRACE_EVENTS && !rc; ++i) rc = ptr_attr(PySequence_Fast_GET_ITEM(seq, i), N_cuda_event, &trace[i]);
    Py_DECREF(seq);
    if (rc) return NULL;
    a.trace_events = trace;
  }
  Py_BEGIN_ALLOW_THREADS
  rc = call(plan, &a);
  Py_END_ALLOW_THREADS
  return done(rc, builtin ? "lightkv_compress_layer_builtin_ws" : "lightkv_compress_layer");
}

static PyObject* compress_layer(PyObject* self, PyObject* const* args, Py_ssize_t nargs, PyObject* kwnames) {
  return layer("compress_layer", g_layer, 0, args, nargs, kwnames);
}
static PyObject* compress_layer_builtin_ws(PyObject* self, PyObject* const* args, Py_ssize_t nargs, PyObject* kwnames) {
  return layer("compress_layer_builtin_ws", g_layer_builtin, 1, args, nargs, kwnames);
}

static const int kKvPos[] = {N_plan, N_stage, N_out, N_k_src, N_v_src, N_k_dst, N_v_dst, N_vis_begin, N_n_text_after, N_mode,
                             N_n_vis, N_page_size, N_src_block_table, N_dst_block_table, N_stream, N_src_seq_start,
                             N_dst_seq_start};

static PyObject* compact_kv(PyObject* self, PyObject* const* args, Py_ssize_t nargs, PyObject* kwnames) {
  Args in;
  if (parse(&in, "compact_kv", args, nargs, kwnames, kKvPos, sizeof(kKvPos) / sizeof(int), 8, NULL, 0)) return NULL;
  lightkv_kv_args_t a;
  memset(&a, 0, sizeof(a));
  a.struct_size = sizeof(a);
  PyObject* out = in.v[N_out];
  void* plan;
  int64_t s[4][3];
  if (plan_handle(in.v[N_plan], &plan) || int_arg(&in, N_stage, 0, &a.stage) || int_arg(&in, N_vis_begin, 0, &a.vis_begin) ||
      int_arg(&in, N_n_text_after, 0, &a.n_text_after) || int_arg(&in, N_mode, LIGHTKV_KV_MERGE, &a.mode) ||
      int_arg(&in, N_page_size, 0, &a.page_size))
    return NULL;
  if (data(get(&in, N_n_vis), &a.n_vis) || data_attr(out, N_n_vis_out, &a.n_vis_out) || data_attr(out, N_grp_off, &a.grp_off) ||
      data_attr(out, N_grp_src, &a.grp_src) || data_attr(out, N_weight, &a.weight) || data_attr(out, N_status, &a.status) ||
      data(in.v[N_k_src], &a.k_src) || data(in.v[N_v_src], &a.v_src) || data(in.v[N_k_dst], &a.k_dst) ||
      data(in.v[N_v_dst], &a.v_dst) || strides(in.v[N_k_src], 3, s[0]) || strides(in.v[N_v_src], 3, s[1]) ||
      strides(in.v[N_k_dst], 3, s[2]) || strides(in.v[N_v_dst], 3, s[3]))
    return NULL;
  if (memcmp(s[0], s[1], sizeof(s[0])) || memcmp(s[2], s[3], sizeof(s[2]))) {
    PyErr_SetString(PyExc_AssertionError, "K and V have the same strides on either side");
    return NULL;
  }
  a.src_head_stride = s[0][1]; a.src_row_stride = s[0][2];
  a.dst_head_stride = s[2][1]; a.dst_row_stride = s[2][2];
  if (a.page_size > 0) {
    PyObject *ts = in.v[N_src_block_table], *td = in.v[N_dst_block_table];
    int32_t blocks = 0;
    if (!ts || !td) { PyErr_SetString(PyExc_TypeError, "paged caches need src_block_table and dst_block_table"); return NULL; }
    a.src_page_stride = s[0][0]; a.dst_page_stride = s[2][0];
    if (data(ts, &a.src_block_table) || data(td, &a.dst_block_table) || size_of(ts, 1, &a.max_blocks) || size_of(td, 1, &blocks)) return NULL;
    if (blocks != a.max_blocks) { PyErr_SetString(PyExc_AssertionError, "the block tables have the same width"); return NULL; }
  } else {
    a.src_batch_stride = s[0][0]; a.dst_batch_stride = s[2][0];
  }
  if (stream_handle(get(&in, N_stream), &a.stream)) return NULL;
  /* packed caches: sample b's first token; contiguous batch strides become 0 */
  if (get(&in, N_src_seq_start)) { if (data(get(&in, N_src_seq_start), &a.src_seq_start)) return NULL; a.src_batch_stride = 0; }
  if (get(&in, N_dst_seq_start)) { if (data(get(&in, N_dst_seq_start), &a.dst_seq_start)) return NULL; a.dst_batch_stride = 0; }
  int rc;
  Py_BEGIN_ALLOW_THREADS
  rc = g_kv(plan, &a);
  Py_END_ALLOW_THREADS
  return done(rc, "lightkv_compact_kv");
}

/* bind(address of lightkv_compress_layer, of lightkv_compress_layer_builtin_ws, of lightkv_compact_kv,
 *      fail(code, what) -> raises, fork_join(out) -> (event, event), raw_stream(device) -> handle, device() -> index) */
static PyObject* bind(PyObject* self, PyObject* args) {
  unsigned long long l, b, k;
  PyObject *fail, *fj, *rs, *dev;
  if (!PyArg_ParseTuple(args, "KKKOOOO", &l, &b, &k, &fail, &fj, &rs, &dev)) return NULL;
  g_layer = (layer_fn)(uintptr_t)l; g_layer_builtin = (layer_fn)(uintptr_t)b; g_kv = (kv_fn)(uintptr_t)k;
  Py_INCREF(fail); Py_INCREF(fj); Py_INCREF(rs); Py_INCREF(dev);
  Py_XSETREF(g_fail, fail); Py_XSETREF(g_fork_join, fj); Py_XSETREF(g_raw_stream, rs); Py_XSETREF(g_device, dev);
  Py_RETURN_NONE;
}

static PyMethodDef kMethods[] = {
    {"compress_layer", (PyCFunction)(void (*)(void))compress_layer, METH_FASTCALL | METH_KEYWORDS, NULL},
    {"compress_layer_builtin_ws", (PyCFunction)(void (*)(void))compress_layer_builtin_ws, METH_FASTCALL | METH_KEYWORDS, NULL},
    {"compact_kv", (PyCFunction)(void (*)(void))compact_kv, METH_FASTCALL | METH_KEYWORDS, NULL},
    {"bind", bind, METH_VARARGS, NULL},
    {NULL, NULL, 0, NULL}};
static struct PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "_binding", NULL, -1, kMethods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__binding(void) {
#define X(n) if (!(g_name[N_##n] = PyUnicode_InternFromString(#n))) return NULL;
  NAMES(X)
#undef X
  if (!(g_stride = PyUnicode_InternFromString("stride"))) return NULL;
  return PyModule_Create(&kModule);
}
