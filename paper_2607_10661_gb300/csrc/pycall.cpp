// Argument marshalling of the hot calls of the Python binding (module _ptdcall).
//
// A call through ctypes cost 7-10 us of host time beside the launch itself (Python-level checks
// of every tensor, torch.cuda.current_stream(), the conversion of a dozen arguments), more
// than many of the kernels take.  Each function here takes the same arguments as its
// counterpart in ptd.py, makes the same checks (a CUDA tensor, contiguous, of the right dtype) and
// calls the C ABI function.  It returns the number of kernels launched, or minus the status
// when the library refuses the call, or None when an argument is not of the plain form
// expected here: nothing has been enqueued then, and ptd.py's own path handles the call or
// raises its error.  Nothing is kept between calls.
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <dlfcn.h>

#include "../../include/ptd.h"

namespace {

PyObject *g_tensor, *g_i32, *g_f32, *g_bf16, *g_raw_stream, *g_get_device;
PyObject *s_is_cuda, *s_is_contiguous, *s_dtype, *s_data_ptr, *s_nbytes, *s_shape, *s_stride, *s_c;

#define PTD_FUNCTIONS(X)                                                                                            \
  X(ptd_tree_attention) X(ptd_topk_draft) X(ptd_verify_greedy) X(ptd_kv_compact) X(ptd_verify_sampling)             \
  X(ptd_verify_and_compact) X(ptd_draft_tree_update) X(ptd_pool_merge) X(ptd_pool_retrieve) X(ptd_tree_rope_append) \
  X(ptd_lm_head_topk) X(ptd_tree_verify_step) X(ptd_last_launch_count)
#define PTD_DECLARE(f) decltype(&f) p_##f;
PTD_FUNCTIONS(PTD_DECLARE)
#undef PTD_DECLARE

// Reads one call's arguments; the first that is not of the expected form clears `ok`.
struct Args {
  PyObject* const* a;
  Py_ssize_t n, i = 0;
  bool ok = true;
  PyObject* kept[3] = {};   // the structures read, held until the call has returned
  int n_kept = 0;
  Args(PyObject* const* args, Py_ssize_t count, Py_ssize_t want) : a(args), n(count) {
    ok = count == want && g_tensor != nullptr;
  }
  ~Args() {
    while (n_kept > 0) Py_DECREF(kept[--n_kept]);
  }
  Args(const Args&) = delete;
  Args& operator=(const Args&) = delete;
  void fail() {
    ok = false;
    PyErr_Clear();
  }
  PyObject* next() { return a[i++]; }
  bool attr_true(PyObject* o, PyObject* name, bool call) {
    PyObject* r = call ? PyObject_CallMethodNoArgs(o, name) : PyObject_GetAttr(o, name);
    Py_XDECREF(r);
    return r == Py_True;
  }
  // (dtype singletons and True outlive the references dropped here)
  PyObject* dtype_of(PyObject* o) {
    PyObject* d = PyObject_GetAttr(o, s_dtype);
    Py_XDECREF(d);
    return d;
  }
  void* pointer(PyObject* o) {
    PyObject* r = PyObject_CallMethodNoArgs(o, s_data_ptr);
    void* p = r != nullptr ? PyLong_AsVoidPtr(r) : nullptr;
    Py_XDECREF(r);
    if (PyErr_Occurred()) fail();
    return p;
  }
  // a contiguous CUDA tensor of `dtype` (NULL: any)
  void* tensor_of(PyObject* o, PyObject* dtype) {
    if (!ok) return nullptr;
    if ((PyObject*)Py_TYPE(o) != g_tensor || !attr_true(o, s_is_cuda, false) || !attr_true(o, s_is_contiguous, true) ||
        (dtype != nullptr && dtype_of(o) != dtype)) {
      fail();
      return nullptr;
    }
    return pointer(o);
  }
  void* tensor(PyObject* dtype = nullptr) {
    PyObject* o = next();
    return tensor_of(o, dtype);
  }
  int32_t* i32() { return static_cast<int32_t*>(tensor(g_i32)); }
  float* f32() { return static_cast<float*>(tensor(g_f32)); }
  // None, or a tensor and its size in bytes
  void* optional(size_t* bytes) {
    *bytes = 0;
    PyObject* o = next();
    if (o == Py_None) return nullptr;
    void* p = tensor_of(o, nullptr);
    if (!ok) return nullptr;
    PyObject* r = PyObject_GetAttr(o, s_nbytes);
    if (r != nullptr && PyLong_CheckExact(r)) *bytes = PyLong_AsSize_t(r); else ok = false;
    Py_XDECREF(r);
    if (PyErr_Occurred()) fail();
    return p;
  }
  // the dtype of a bf16 or fp32 tensor
  ptd_dtype kind(PyObject* o) {
    if (!ok) return PTD_F32;
    PyObject* d = (PyObject*)Py_TYPE(o) == g_tensor ? dtype_of(o) : nullptr;
    if (d != g_bf16 && d != g_f32) fail();
    return d == g_bf16 ? PTD_BF16 : PTD_F32;
  }
  // the sizes of a 2-D tensor
  void dims2(PyObject* o, int64_t* d0, int64_t* d1) {
    *d0 = *d1 = 0;
    if (!ok) return;
    PyObject* s = PyObject_GetAttr(o, s_shape);
    if (s != nullptr && PyTuple_Check(s) && PyTuple_GET_SIZE(s) == 2) {
      *d0 = PyLong_AsLongLong(PyTuple_GET_ITEM(s, 0));
      *d1 = PyLong_AsLongLong(PyTuple_GET_ITEM(s, 1));
    } else {
      ok = false;
    }
    Py_XDECREF(s);
    if (PyErr_Occurred()) fail();
  }
  // a 2-D tensor's rows: CUDA, unit column stride, rows at least a row apart
  void* rows2(PyObject* o, PyObject* dtype, int64_t* rows, int64_t* cols, int64_t* stride) {
    *stride = 0;
    dims2(o, rows, cols);
    if (!ok || (PyObject*)Py_TYPE(o) != g_tensor || !attr_true(o, s_is_cuda, false) || dtype_of(o) != dtype) {
      fail();
      return nullptr;
    }
    PyObject* s = PyObject_CallMethodNoArgs(o, s_stride);
    int64_t unit = 0;
    if (s != nullptr && PyTuple_Check(s) && PyTuple_GET_SIZE(s) == 2) {
      *stride = PyLong_AsLongLong(PyTuple_GET_ITEM(s, 0));
      unit = PyLong_AsLongLong(PyTuple_GET_ITEM(s, 1));
    }
    Py_XDECREF(s);
    if (PyErr_Occurred() || unit != 1 || *stride < *cols) {
      fail();
      return nullptr;
    }
    return pointer(o);
  }
  int64_t i64() {
    PyObject* o = next();
    if (!ok) return 0;
    if (!PyLong_CheckExact(o)) {
      ok = false;
      return 0;
    }
    const int64_t v = PyLong_AsLongLong(o);
    if (PyErr_Occurred()) fail();
    return v;
  }
  int32_t num() {
    const int64_t v = i64();
    if (v != (int32_t)v) ok = false;
    return (int32_t)v;
  }
  float real() {
    PyObject* o = next();
    if (!ok) return 0.f;
    if (!PyFloat_CheckExact(o) && !PyLong_CheckExact(o)) {
      ok = false;
      return 0.f;
    }
    const double v = PyFloat_AsDouble(o);
    if (PyErr_Occurred()) fail();
    return (float)v;
  }
  // the ctypes structure in the attribute `c` of a Tree, KVCache or StepBuffers (the attribute may be
  // a new object at each read, or be replaced by another thread while the call runs without the lock)
  template <typename S>
  S* structure() {
    PyObject* o = next();
    if (!ok) return nullptr;
    PyObject* c = PyObject_GetAttr(o, s_c);
    Py_buffer v;
    S* p = nullptr;
    if (c != nullptr && PyObject_GetBuffer(c, &v, PyBUF_SIMPLE) == 0) {
      if ((size_t)v.len == sizeof(S) && n_kept < 3) p = static_cast<S*>(v.buf);
      PyBuffer_Release(&v);
    }
    if (p == nullptr) {
      Py_XDECREF(c);
      fail();
      return nullptr;
    }
    kept[n_kept++] = c;
    return p;
  }
  // None (the current stream of the current device) or the stream's address
  void* stream() {
    PyObject* o = next();
    if (!ok) return nullptr;
    if (PyLong_CheckExact(o)) return PyLong_AsVoidPtr(o);
    if (o != Py_None) {
      ok = false;
      return nullptr;
    }
    PyObject* d = PyObject_CallNoArgs(g_get_device);
    PyObject* r = d != nullptr ? PyObject_CallOneArg(g_raw_stream, d) : nullptr;
    void* p = r != nullptr ? PyLong_AsVoidPtr(r) : nullptr;
    Py_XDECREF(d);
    Py_XDECREF(r);
    if (PyErr_Occurred()) fail();
    return p;
  }
};

// The call itself runs without the interpreter lock (a launch can wait for room in the stream).
#define PTD_CALL(expr)          \
  do {                          \
    ptd_status st_;             \
    Py_BEGIN_ALLOW_THREADS      \
    st_ = expr;                 \
    Py_END_ALLOW_THREADS        \
    return done(st_);           \
  } while (0)

PyObject* done(ptd_status st) { return PyLong_FromLong(st == PTD_OK ? (long)p_ptd_last_launch_count() : -(long)st); }

// (tree, cache, layer_begin, num_layers, q, num_q_heads, scale, out, workspace, dev_status, stream)
PyObject* tree_attention(PyObject*, PyObject* const* a, Py_ssize_t n) {
  Args g(a, n, 11);
  if (!g.ok) Py_RETURN_NONE;
  const ptd_tree* tree = g.structure<ptd_tree>();
  const ptd_kv_cache* cache = g.structure<ptd_kv_cache>();
  if (!g.ok) Py_RETURN_NONE;
  PyObject* dt = cache->dtype == PTD_BF16 ? g_bf16 : g_f32;
  const int32_t l0 = g.num(), nl = g.num();
  const void* q = g.tensor(dt);
  const int32_t hq = g.num();
  const float scale = g.real();
  void* out = g.tensor(dt);
  size_t wsb;
  void* ws = g.optional(&wsb);
  int32_t* status = g.i32();
  void* s = g.stream();
  if (!g.ok) Py_RETURN_NONE;
  PTD_CALL(p_ptd_tree_attention(tree, cache, l0, nl, q, hq, scale, out, ws, wsb, status, s));
}

// (logits, k, out_idx, out_val, vocab, stream)
PyObject* topk_draft(PyObject*, PyObject* const* a, Py_ssize_t n) {
  Args g(a, n, 6);
  if (!g.ok) Py_RETURN_NONE;
  const ptd_dtype dt = g.kind(a[0]);
  int64_t rows, stride;
  g.dims2(a[0], &rows, &stride);
  const void* logits = g.tensor();
  const int32_t k = g.num();
  int32_t* idx = g.i32();
  float* val = g.f32();
  const int64_t vocab = a[4] == Py_None ? (g.next(), stride) : g.i64();
  void* s = g.stream();
  if (!g.ok || vocab != (int32_t)vocab) Py_RETURN_NONE;
  PTD_CALL(p_ptd_topk_draft(logits, dt, rows, (int32_t)vocab, stride, k, idx, val, s));
}

// (tree, tokens, target, target_stride, accepted, accept_len, bonus, dev_status, stream)
PyObject* verify_greedy(PyObject*, PyObject* const* a, Py_ssize_t n) {
  Args g(a, n, 9);
  if (!g.ok) Py_RETURN_NONE;
  const ptd_tree* tree = g.structure<ptd_tree>();
  const int32_t* tokens = g.i32();
  const int32_t* target = g.i32();
  const int32_t stride = g.num();
  int32_t* acc = g.i32();
  int32_t* len = g.i32();
  int32_t* bonus = g.i32();
  int32_t* status = g.i32();
  void* s = g.stream();
  if (!g.ok) Py_RETURN_NONE;
  PTD_CALL(p_ptd_verify_greedy(tree, tokens, target, stride, acc, len, bonus, status, s));
}

// (tree, cache, accepted, accept_len, new_ctx, stream)
PyObject* kv_compact(PyObject*, PyObject* const* a, Py_ssize_t n) {
  Args g(a, n, 6);
  if (!g.ok) Py_RETURN_NONE;
  const ptd_tree* tree = g.structure<ptd_tree>();
  const ptd_kv_cache* cache = g.structure<ptd_kv_cache>();
  const int32_t* acc = g.i32();
  const int32_t* len = g.i32();
  int32_t* ctx = g.i32();
  void* s = g.stream();
  if (!g.ok) Py_RETURN_NONE;
  PTD_CALL(p_ptd_kv_compact(tree, cache, acc, len, ctx, s));
}

// (tree, tokens, logits, temperature, u_accept, u_bonus, accepted, accept_len, bonus, dev_status, stream)
PyObject* verify_sampling(PyObject*, PyObject* const* a, Py_ssize_t n) {
  Args g(a, n, 11);
  if (!g.ok) Py_RETURN_NONE;
  const ptd_tree* tree = g.structure<ptd_tree>();
  const int32_t* tokens = g.i32();
  PyObject* lg = g.next();
  const ptd_dtype dt = g.kind(lg);
  int64_t rows, vocab, stride;
  const void* logits = g.rows2(lg, dt == PTD_BF16 ? g_bf16 : g_f32, &rows, &vocab, &stride);
  const float temperature = g.real();
  const float* ua = g.f32();
  const float* ub = g.f32();
  int32_t* acc = g.i32();
  int32_t* len = g.i32();
  int32_t* bonus = g.i32();
  int32_t* status = g.i32();
  void* s = g.stream();
  if (!g.ok || vocab != (int32_t)vocab) Py_RETURN_NONE;
  PTD_CALL(p_ptd_verify_sampling(tree, tokens, logits, dt, (int32_t)vocab, stride, temperature, ua, ub, acc, len,
                                    bonus, status, s));
}

// (tree, cache, tokens, target, target_stride, accepted, accept_len, bonus, new_ctx, dev_status, stream)
PyObject* verify_and_compact(PyObject*, PyObject* const* a, Py_ssize_t n) {
  Args g(a, n, 11);
  if (!g.ok) Py_RETURN_NONE;
  const ptd_tree* tree = g.structure<ptd_tree>();
  const ptd_kv_cache* cache = g.structure<ptd_kv_cache>();
  const int32_t* tokens = g.i32();
  const int32_t* target = g.i32();
  const int32_t stride = g.num();
  int32_t* acc = g.i32();
  int32_t* len = g.i32();
  int32_t* bonus = g.i32();
  int32_t* ctx = g.i32();
  int32_t* status = g.i32();
  void* s = g.stream();
  if (!g.ok) Py_RETURN_NONE;
  PTD_CALL(p_ptd_verify_and_compact(tree, cache, tokens, target, stride, acc, len, bonus, ctx, status, s));
}

// (tree, cache, bufs, stream)
PyObject* tree_verify_step(PyObject*, PyObject* const* a, Py_ssize_t n) {
  Args g(a, n, 4);
  if (!g.ok) Py_RETURN_NONE;
  const ptd_tree* tree = g.structure<ptd_tree>();
  const ptd_kv_cache* cache = g.structure<ptd_kv_cache>();
  const ptd_step_args* args = g.structure<ptd_step_args>();
  void* s = g.stream();
  if (!g.ok) Py_RETURN_NONE;
  PTD_CALL(p_ptd_tree_verify_step(tree, cache, args, s));
}

// (in_count, in_parents, in_tokens, drafts, expand, width, max_depth, capacity, out_count, out_parents,
//  out_tokens, out_depths, old_to_new, dev_status, stream)
PyObject* draft_tree_update(PyObject*, PyObject* const* a, Py_ssize_t n) {
  Args g(a, n, 15);
  if (!g.ok) Py_RETURN_NONE;
  int64_t B, stride, d0, d1, rows, dstride;
  const int32_t* in_count = g.i32();
  g.dims2(a[1], &B, &stride);
  const int32_t* in_parents = g.i32();
  g.dims2(a[2], &d0, &d1);
  if (d0 != B || d1 != stride) g.ok = false;
  const int32_t* in_tokens = g.i32();
  g.dims2(a[3], &rows, &dstride);
  if (rows != B * stride) g.ok = false;
  const int32_t* drafts = g.i32();
  const int32_t expand = g.num(), width = g.num(), max_depth = g.num(), capacity = g.num();
  int32_t* out_count = g.i32();
  int32_t* out[3];
  for (int32_t*& o : out) {
    g.dims2(a[g.i], &d0, &d1);
    if (d0 != B || d1 != capacity) g.ok = false;
    o = g.i32();
  }
  g.dims2(a[12], &d0, &d1);
  if (d0 != B || d1 != stride) g.ok = false;
  int32_t* old_to_new = g.i32();
  int32_t* status = g.i32();
  void* s = g.stream();
  if (!g.ok || B != (int32_t)B || stride != (int32_t)stride || dstride != (int32_t)dstride) Py_RETURN_NONE;
  PTD_CALL(p_ptd_draft_tree_update((int32_t)B, (int32_t)stride, in_count, in_parents, in_tokens, drafts,
                                      (int32_t)dstride, expand, width, max_depth, capacity, out_count, out[0], out[1],
                                      out[2], old_to_new, status, s));
}

// (pool buffer, capacity, max_load, step, count, parents, tokens, dev_status, stream)
PyObject* pool_merge(PyObject*, PyObject* const* a, Py_ssize_t n) {
  Args g(a, n, 9);
  if (!g.ok) Py_RETURN_NONE;
  void* pool = g.tensor();
  const int32_t capacity = g.num(), max_load = g.num(), step = g.num();
  const int32_t* count = g.i32();
  const int32_t* parents = g.i32();
  const int32_t* tokens = g.i32();
  int32_t* status = g.i32();
  void* s = g.stream();
  if (!g.ok) Py_RETURN_NONE;
  PTD_CALL(p_ptd_pool_merge(pool, capacity, max_load, step, count, parents, tokens, status, s));
}

// (pool buffer, capacity, root_token, width, max_depth, max_nodes, out_count, out_parents, out_tokens, stream)
PyObject* pool_retrieve(PyObject*, PyObject* const* a, Py_ssize_t n) {
  Args g(a, n, 10);
  if (!g.ok) Py_RETURN_NONE;
  const void* pool = g.tensor();
  const int32_t capacity = g.num();
  const int32_t* root = g.i32();
  const int32_t width = g.num(), max_depth = g.num(), max_nodes = g.num();
  int32_t* count = g.i32();
  int32_t* out[2];
  for (int32_t*& o : out) {
    PyObject* t = a[g.i];
    o = g.i32();
    if (!g.ok) Py_RETURN_NONE;
    PyObject* r = PyObject_GetAttr(t, s_nbytes);
    if (r == nullptr || !PyLong_CheckExact(r) || PyLong_AsLongLong(r) < 4 * (int64_t)max_nodes) g.fail();
    Py_XDECREF(r);
  }
  void* s = g.stream();
  if (!g.ok) Py_RETURN_NONE;
  PTD_CALL(p_ptd_pool_retrieve(pool, capacity, root, width, max_depth, max_nodes, count, out[0], out[1], s));
}

// (tree, cache, layer_begin, num_layers, q, num_q_heads, k, v, rope_base, positions_out, dev_status, stream)
PyObject* tree_rope_append(PyObject*, PyObject* const* a, Py_ssize_t n) {
  Args g(a, n, 12);
  if (!g.ok) Py_RETURN_NONE;
  const ptd_tree* tree = g.structure<ptd_tree>();
  const ptd_kv_cache* cache = g.structure<ptd_kv_cache>();
  if (!g.ok) Py_RETURN_NONE;
  PyObject* dt = cache->dtype == PTD_BF16 ? g_bf16 : g_f32;
  const int32_t l0 = g.num(), nl = g.num();
  void* q = g.tensor(dt);
  const int32_t hq = g.num();
  const void* k = g.tensor(dt);
  const void* v = g.tensor(dt);
  const float base = g.real();
  int32_t* pos = a[9] == Py_None ? (g.next(), nullptr) : g.i32();
  int32_t* status = g.i32();
  void* s = g.stream();
  if (!g.ok) Py_RETURN_NONE;
  PTD_CALL(p_ptd_tree_rope_append(tree, cache, l0, nl, q, hq, k, v, base, pos, status, s));
}

// (hidden, weight, k, out_idx, out_val, workspace, dev_status, stream)
PyObject* lm_head_topk(PyObject*, PyObject* const* a, Py_ssize_t n) {
  Args g(a, n, 8);
  if (!g.ok) Py_RETURN_NONE;
  int64_t rows, d, hstride, vocab, wd, wstride;
  const void* hidden = g.rows2(g.next(), g_bf16, &rows, &d, &hstride);
  if (!g.ok) Py_RETURN_NONE;
  const void* weight = g.rows2(g.next(), g_bf16, &vocab, &wd, &wstride);
  const int32_t k = g.num();
  int32_t* idx = g.i32();
  float* val = g.f32();
  size_t wsb;
  if (a[g.i] == Py_None) Py_RETURN_NONE;
  void* ws = g.optional(&wsb);
  int32_t* status = g.i32();
  void* s = g.stream();
  if (!g.ok || d != wd || rows != (int32_t)rows || vocab != (int32_t)vocab || d != (int32_t)d) Py_RETURN_NONE;
  PTD_CALL(p_ptd_lm_head_topk(hidden, (int32_t)rows, hstride, weight, (int32_t)vocab, wstride, (int32_t)d, k, idx,
                                 val, ws, wsb, status, s));
}

// load(path of libptd.so, Tensor type, int32, float32, bfloat16, raw stream getter, device getter)
PyObject* load(PyObject*, PyObject* args) {
  const char* path;
  PyObject* o[6];
  if (!PyArg_ParseTuple(args, "sOOOOOO", &path, &o[0], &o[1], &o[2], &o[3], &o[4], &o[5])) return nullptr;
  void* h = dlopen(path, RTLD_NOW | RTLD_LOCAL);
  if (h == nullptr) {
    PyErr_SetString(PyExc_RuntimeError, dlerror());
    return nullptr;
  }
#define PTD_RESOLVE(f)                                                      \
  p_##f = reinterpret_cast<decltype(&f)>(dlsym(h, #f));                     \
  if (p_##f == nullptr) {                                                   \
    PyErr_SetString(PyExc_RuntimeError, "libptd.so has no symbol " #f);     \
    return nullptr;                                                         \
  }
  PTD_FUNCTIONS(PTD_RESOLVE)
#undef PTD_RESOLVE
  for (PyObject* x : o) Py_INCREF(x);
  g_tensor = o[0], g_i32 = o[1], g_f32 = o[2], g_bf16 = o[3], g_raw_stream = o[4], g_get_device = o[5];
  Py_RETURN_NONE;
}

#define PTD_METHOD(f) {#f, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(f)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {PTD_METHOD(tree_attention),
                         PTD_METHOD(topk_draft),
                         PTD_METHOD(verify_greedy),
                         PTD_METHOD(kv_compact),
                         PTD_METHOD(verify_sampling),
                         PTD_METHOD(verify_and_compact),
                         PTD_METHOD(tree_verify_step),
                         PTD_METHOD(draft_tree_update),
                         PTD_METHOD(pool_merge),
                         PTD_METHOD(pool_retrieve),
                         PTD_METHOD(tree_rope_append),
                         PTD_METHOD(lm_head_topk),
                         {"load", load, METH_VARARGS, nullptr},
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_ptdcall", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__ptdcall(void) {
  s_is_cuda = PyUnicode_InternFromString("is_cuda");
  s_is_contiguous = PyUnicode_InternFromString("is_contiguous");
  s_dtype = PyUnicode_InternFromString("dtype");
  s_data_ptr = PyUnicode_InternFromString("data_ptr");
  s_nbytes = PyUnicode_InternFromString("nbytes");
  s_shape = PyUnicode_InternFromString("shape");
  s_stride = PyUnicode_InternFromString("stride");
  s_c = PyUnicode_InternFromString("c");
  return PyModule_Create(&module);
}
