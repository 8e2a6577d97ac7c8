// Python entry points of the enqueueing calls (module _dlm_calls): argument marshalling only, as in _binding.py, for the
// calls a serving loop makes many times per step.  Through ctypes a call of ten tensors spent 6 - 10 us on marshalling,
// as long as the kernel it enqueues; here it is a few hundred nanoseconds (tensor fields and the current stream are read
// from their C++ objects).  Every function takes its arguments by position or by name and releases the GIL around the
// library call, as ctypes did.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "dlm.h"

namespace {

PyObject* g_error = nullptr;   // DlmError(code, where), set by the package
// The classes whose memory is read as a pointer and as a dlm_kv_cache (ctypes.c_void_p and the package's structure), set by
// the package.  Nothing else will do: the bytes of another object would be taken for device addresses.
PyTypeObject *g_handle_type = nullptr, *g_cache_type = nullptr;

struct Args;
typedef int (*CallFn)(Args&);

// One entry point: its name, its arguments' names and the call.
struct Entry {
  const char* name;
  int n_args;
  const char* const* arg_names;
  CallFn call;
};

// The arguments of one call.  Getters read argument i; the first failure sets a Python exception and `failed`.
struct Args {
  PyObject* const* v;
  bool failed = false;

  // pointer held by a ctypes.c_void_p, an int or None
  void* handle(int i) {
    PyObject* o = v[i];
    if (o == Py_None) return nullptr;
    if (PyLong_Check(o)) {
      void* const p = PyLong_AsVoidPtr(o);
      if (!p && PyErr_Occurred()) failed = true;
      return p;
    }
    return *static_cast<void**>(buffer(i, g_handle_type, sizeof(void*)));
  }
  // address of the memory behind a ctypes object of class `type` and at least `bytes` bytes (the argument stays alive during the call)
  void* buffer(int i, PyTypeObject* type, Py_ssize_t bytes) {
    static void* zero[16] = {};
    if (failed) return zero;
    if (!type || !PyObject_TypeCheck(v[i], type)) {
      PyErr_Format(PyExc_TypeError, "expected %s, got %s", type ? type->tp_name : "a ctypes object", Py_TYPE(v[i])->tp_name);
      failed = true;
      return zero;
    }
    Py_buffer b;
    if (PyObject_GetBuffer(v[i], &b, PyBUF_SIMPLE) != 0) { failed = true; return zero; }
    void* p = b.buf;
    const bool ok = b.len >= bytes;
    PyBuffer_Release(&b);
    if (!ok) {
      PyErr_SetString(PyExc_TypeError, "argument is too small");
      failed = true;
      return zero;
    }
    return p;
  }
  const dlm_kv_cache* cache(int i) { return static_cast<const dlm_kv_cache*>(buffer(i, g_cache_type, sizeof(dlm_kv_cache))); }
  int integer(int i) {
    if (failed) return 0;
    if (PyLong_Check(v[i])) return (int)PyLong_AsUnsignedLongMask(v[i]);
    PyObject* n = PyNumber_Long(v[i]);
    if (!n) { failed = true; return 0; }
    const int x = (int)PyLong_AsUnsignedLongMask(n);
    Py_DECREF(n);
    return x;
  }
  int truth(int i) {
    const int x = failed ? 0 : PyObject_IsTrue(v[i]);
    if (x < 0) failed = true;
    return x > 0;
  }
  float real(int i) {
    const double x = failed ? 0.0 : PyFloat_AsDouble(v[i]);
    if (x == -1.0 && PyErr_Occurred()) failed = true;
    return (float)x;
  }
  const at::Tensor* tensor(int i) {
    if (failed) return nullptr;
    if (THPVariable_Check(v[i])) {
      const at::Tensor& t = THPVariable_Unpack(v[i]);
      if (t.is_cuda() && t.is_contiguous()) return &t;
    }
    PyErr_SetString(PyExc_TypeError, "expected a contiguous CUDA tensor");
    failed = true;
    return nullptr;
  }
  // device pointer of a contiguous CUDA tensor of the given type, or of None
  void* ptr(int i, at::ScalarType type) {
    if (failed || v[i] == Py_None) return nullptr;
    const at::Tensor* t = tensor(i);
    if (!t) return nullptr;
    if (t->scalar_type() != type) {
      PyErr_Format(PyExc_TypeError, "expected dtype torch.%s", type == at::kBFloat16 ? "bfloat16" : type == at::kFloat ? "float32"
                                                               : type == at::kInt ? "int32" : "uint8");
      failed = true;
      return nullptr;
    }
    return t->data_ptr();
  }
  void* bf16(int i) { return ptr(i, at::kBFloat16); }
  float* f32(int i) { return static_cast<float*>(ptr(i, at::kFloat)); }
  int32_t* i32(int i) { return static_cast<int32_t*>(ptr(i, at::kInt)); }
  uint8_t* u8(int i) { return static_cast<uint8_t*>(ptr(i, at::kByte)); }
  void* scratch(int i, size_t& bytes) {
    bytes = 0;
    const at::Tensor* t = tensor(i);
    if (!t) return nullptr;
    bytes = t->nbytes();
    return t->data_ptr();
  }
};

#define RELEASED(expr)                                          \
  do {                                                          \
    if (a.failed) return 0;                                     \
    void* const s = c10::cuda::getCurrentCUDAStream().stream(); \
    int rc_;                                                    \
    Py_BEGIN_ALLOW_THREADS;                                     \
    rc_ = (expr);                                               \
    Py_END_ALLOW_THREADS;                                       \
    return rc_;                                                 \
  } while (0)

const char* const kCommitArgs[] = {"ctx", "cache", "k_new", "v_new", "src_len", "src_idx", "dst_pos", "dst_mode", "n_rows", "n_max",
                                   "advance_len", "layer_begin", "layer_end"};
int call_commit(Args& a) {
  dlm_ctx* ctx = static_cast<dlm_ctx*>(a.handle(0));
  const dlm_kv_cache* cache = a.cache(1);
  const void *k = a.bf16(2), *v = a.bf16(3);
  const int src_len = a.integer(4);
  const int32_t *src_idx = a.i32(5), *dst_pos = a.i32(6);
  const int dst_mode = a.integer(7);
  const int32_t* n_rows = a.i32(8);
  const int n_max = a.integer(9), advance = a.truth(10), lb = a.integer(11), le = a.integer(12);
  RELEASED(dlm_kv_cache_commit(ctx, cache, k, v, src_len, src_idx, dst_pos, dst_mode, n_rows, n_max, advance, lb, le, s));
}

const char* const kAttnArgs[] = {"ctx", "cache", "layer_begin", "layer_end", "q", "k_new", "v_new", "n_q_heads", "q_cap", "q_len",
                                 "softmax_scale", "cache_len_hint", "out", "lse", "workspace"};
int call_attn(Args& a) {
  dlm_ctx* ctx = static_cast<dlm_ctx*>(a.handle(0));
  const dlm_kv_cache* cache = a.cache(1);
  const int lb = a.integer(2), le = a.integer(3);
  const void *q = a.bf16(4), *k = a.bf16(5), *v = a.bf16(6);
  const int heads = a.integer(7), q_cap = a.integer(8);
  const int32_t* q_len = a.i32(9);
  const float scale = a.real(10);
  const int hint = a.integer(11);
  void* out = a.bf16(12);
  float* lse = a.f32(13);
  size_t bytes;
  void* ws = a.scratch(14, bytes);
  RELEASED(dlm_freecache_attn_step(ctx, cache, lb, le, q, k, v, heads, q_cap, q_len, scale, hint, out, lse, ws, bytes, s));
}

const char* const kUnmaskArgs[] = {"ctx", "logits", "batch", "block_len", "vocab", "masked", "tokens", "k", "tok", "conf", "sel_idx",
                                   "n_sel", "workspace"};
int call_unmask(Args& a) {
  dlm_ctx* ctx = static_cast<dlm_ctx*>(a.handle(0));
  const float* z = a.f32(1);
  const int batch = a.integer(2), block = a.integer(3), vocab = a.integer(4);
  uint8_t* masked = a.u8(5);
  int32_t* tokens = a.i32(6);
  const int k = a.integer(7);
  int32_t* tok = a.i32(8);
  float* conf = a.f32(9);
  int32_t *sel = a.i32(10), *n = a.i32(11);
  size_t bytes;
  void* ws = a.scratch(12, bytes);
  RELEASED(dlm_unmask_select(ctx, z, batch, block, vocab, masked, tokens, k, tok, conf, sel, n, ws, bytes, s));
}

const char* const kUnmaskStaticArgs[] = {"logits", "batch", "block_len", "vocab", "masked", "tokens", "k", "tok", "conf", "sel_idx", "n_sel"};
int call_unmask_static(Args& a) {
  const float* z = a.f32(0);
  const int batch = a.integer(1), block = a.integer(2), vocab = a.integer(3);
  uint8_t* masked = a.u8(4);
  int32_t* tokens = a.i32(5);
  const int k = a.integer(6);
  int32_t* tok = a.i32(7);
  float* conf = a.f32(8);
  int32_t *sel = a.i32(9), *n = a.i32(10);
  RELEASED(dlm_unmask_select_static(z, batch, block, vocab, masked, tokens, k, tok, conf, sel, n, s));
}

const char* const kScoredArgs[] = {"ctx", "logits", "batch", "block_len", "vocab", "masked", "tokens", "k", "score_kind", "noise", "tok",
                                   "conf", "score", "zmax", "sel_idx", "n_sel", "workspace"};
int call_scored(Args& a) {
  dlm_ctx* ctx = static_cast<dlm_ctx*>(a.handle(0));
  const float* z = a.f32(1);
  const int batch = a.integer(2), block = a.integer(3), vocab = a.integer(4);
  uint8_t* masked = a.u8(5);
  int32_t* tokens = a.i32(6);
  const int k = a.integer(7), kind = a.integer(8);
  const float* noise = a.f32(9);
  int32_t* tok = a.i32(10);
  float *conf = a.f32(11), *score = a.f32(12), *zmax = a.f32(13);
  int32_t *sel = a.i32(14), *n = a.i32(15);
  size_t bytes;
  void* ws = a.scratch(16, bytes);
  RELEASED(dlm_unmask_select_scored(ctx, z, batch, block, vocab, masked, tokens, k, kind, noise, tok, conf, score, zmax, sel, n, ws, bytes, s));
}

const char* const kAcceptArgs[] = {"ctx", "tok_dlm", "tok_ar", "batch", "block_len", "masked", "tokens", "fallback_source", "accept",
                                   "acc_idx", "n_acc"};
int call_accept(Args& a) {
  dlm_ctx* ctx = static_cast<dlm_ctx*>(a.handle(0));
  const int32_t *dlm_t = a.i32(1), *ar = a.i32(2);
  const int batch = a.integer(3), block = a.integer(4);
  uint8_t* masked = a.u8(5);
  int32_t* tokens = a.i32(6);
  const int fallback = a.integer(7);
  uint8_t* accept = a.u8(8);
  int32_t *idx = a.i32(9), *n = a.i32(10);
  RELEASED(dlm_guided_accept(ctx, dlm_t, ar, batch, block, masked, tokens, fallback, accept, idx, n, s));
}

const char* const kAcceptTopkArgs[] = {"ctx", "tok_dlm", "tok_ar_topk", "top_k", "batch", "block_len", "masked", "tokens",
                                       "fallback_source", "accept", "acc_idx", "n_acc"};
int call_accept_topk(Args& a) {
  dlm_ctx* ctx = static_cast<dlm_ctx*>(a.handle(0));
  const int32_t *dlm_t = a.i32(1), *ar = a.i32(2);
  const int top_k = a.integer(3), batch = a.integer(4), block = a.integer(5);
  uint8_t* masked = a.u8(6);
  int32_t* tokens = a.i32(7);
  const int fallback = a.integer(8);
  uint8_t* accept = a.u8(9);
  int32_t *idx = a.i32(10), *n = a.i32(11);
  RELEASED(dlm_guided_accept_topk(ctx, dlm_t, ar, top_k, batch, block, masked, tokens, fallback, accept, idx, n, s));
}

const char* const kAcceptThresholdArgs[] = {"ctx", "tok_dlm", "zmax_dlm", "tok_ar_topk", "logit_ar_topk", "top_k", "tau", "batch",
                                            "block_len", "masked", "tokens", "fallback_source", "accept", "acc_idx", "n_acc"};
int call_accept_threshold(Args& a) {
  dlm_ctx* ctx = static_cast<dlm_ctx*>(a.handle(0));
  const int32_t* dlm_t = a.i32(1);
  const float* zmax = a.f32(2);
  const int32_t* ar = a.i32(3);
  const float* lg = a.f32(4);
  const int top_k = a.integer(5);
  const float tau = a.real(6);
  const int batch = a.integer(7), block = a.integer(8);
  uint8_t* masked = a.u8(9);
  int32_t* tokens = a.i32(10);
  const int fallback = a.integer(11);
  uint8_t* accept = a.u8(12);
  int32_t *idx = a.i32(13), *n = a.i32(14);
  RELEASED(dlm_guided_accept_threshold(ctx, dlm_t, zmax, ar, lg, top_k, tau, batch, block, masked, tokens, fallback, accept, idx, n, s));
}

const char* const kQkvArgs[] = {"ctx", "x", "w", "bias", "batch", "q_cap", "d_model", "n_q_heads", "n_kv_heads", "head_dim", "q_out",
                                "k_out", "v_out", "workspace"};
int call_qkv(Args& a) {
  dlm_ctx* ctx = static_cast<dlm_ctx*>(a.handle(0));
  const void *x = a.bf16(1), *w = a.bf16(2), *bias = a.bf16(3);
  const int batch = a.integer(4), q_cap = a.integer(5), dm = a.integer(6), hq = a.integer(7), hkv = a.integer(8), d = a.integer(9);
  void *q = a.bf16(10), *k = a.bf16(11), *v = a.bf16(12);
  size_t bytes;
  void* ws = a.scratch(13, bytes);
  RELEASED(dlm_window_qkv_project(ctx, x, w, bias, batch, q_cap, dm, hq, hkv, d, q, k, v, ws, bytes, s));
}

const char* const kRopeArgs[] = {"ctx", "x", "w", "bias", "rope_cos", "rope_sin", "batch", "q_cap", "d_model", "n_q_heads", "n_kv_heads",
                                 "head_dim", "q_out", "k_out", "v_out", "workspace"};
int call_rope(Args& a) {
  dlm_ctx* ctx = static_cast<dlm_ctx*>(a.handle(0));
  const void *x = a.bf16(1), *w = a.bf16(2), *bias = a.bf16(3);
  const float *cs = a.f32(4), *sn = a.f32(5);
  const int batch = a.integer(6), q_cap = a.integer(7), dm = a.integer(8), hq = a.integer(9), hkv = a.integer(10), d = a.integer(11);
  void *q = a.bf16(12), *k = a.bf16(13), *v = a.bf16(14);
  size_t bytes;
  void* ws = a.scratch(15, bytes);
  RELEASED(dlm_window_qkv_project_rope(ctx, x, w, bias, cs, sn, batch, q_cap, dm, hq, hkv, d, q, k, v, ws, bytes, s));
}

const char* const kStageArgs[] = {"ctx", "x", "w", "bias", "rope_cos", "rope_sin", "batch", "q_cap", "d_model", "n_q_heads", "n_kv_heads",
                                  "head_dim", "q_len", "q_out", "k_out", "v_out", "cache", "layer", "workspace"};
int call_stage(Args& a) {
  dlm_ctx* ctx = static_cast<dlm_ctx*>(a.handle(0));
  const void *x = a.bf16(1), *w = a.bf16(2), *bias = a.bf16(3);
  const float *cs = a.f32(4), *sn = a.f32(5);
  const int batch = a.integer(6), q_cap = a.integer(7), dm = a.integer(8), hq = a.integer(9), hkv = a.integer(10), d = a.integer(11);
  const int32_t* q_len = a.i32(12);
  void *q = a.bf16(13), *k = a.bf16(14), *v = a.bf16(15);
  const dlm_kv_cache* cache = a.cache(16);
  const int layer = a.integer(17);
  size_t bytes;
  void* ws = a.scratch(18, bytes);
  RELEASED(dlm_window_qkv_project_stage(ctx, x, w, bias, cs, sn, batch, q_cap, dm, hq, hkv, d, q_len, q, k, v, cache, layer, ws, bytes, s));
}

const char* const kOutArgs[] = {"ctx", "o", "wo", "bias", "batch", "q_cap", "d_model", "n_q_heads", "head_dim", "y", "workspace"};
int call_out(Args& a) {
  dlm_ctx* ctx = static_cast<dlm_ctx*>(a.handle(0));
  const void *o = a.bf16(1), *wo = a.bf16(2), *bias = a.bf16(3);
  const int batch = a.integer(4), q_cap = a.integer(5), dm = a.integer(6), hq = a.integer(7), d = a.integer(8);
  void* y = a.bf16(9);
  size_t bytes;
  void* ws = a.scratch(10, bytes);
  RELEASED(dlm_window_out_project(ctx, o, wo, bias, batch, q_cap, dm, hq, d, y, ws, bytes, s));
}

#define ENTRY(name, names, fn) {name, (int)(sizeof(names) / sizeof(names[0])), names, fn}
const Entry kEntries[] = {
    ENTRY("dlm_kv_cache_commit", kCommitArgs, call_commit),
    ENTRY("dlm_freecache_attn_step", kAttnArgs, call_attn),
    ENTRY("dlm_unmask_select", kUnmaskArgs, call_unmask),
    ENTRY("dlm_unmask_select_static", kUnmaskStaticArgs, call_unmask_static),
    ENTRY("dlm_unmask_select_scored", kScoredArgs, call_scored),
    ENTRY("dlm_guided_accept", kAcceptArgs, call_accept),
    ENTRY("dlm_guided_accept_topk", kAcceptTopkArgs, call_accept_topk),
    ENTRY("dlm_guided_accept_threshold", kAcceptThresholdArgs, call_accept_threshold),
    ENTRY("dlm_window_qkv_project", kQkvArgs, call_qkv),
    ENTRY("dlm_window_qkv_project_rope", kRopeArgs, call_rope),
    ENTRY("dlm_window_qkv_project_stage", kStageArgs, call_stage),
    ENTRY("dlm_window_out_project", kOutArgs, call_out),
};
constexpr int kNumEntries = sizeof(kEntries) / sizeof(kEntries[0]);
constexpr int kMaxArgs = 24;

PyObject* run(const Entry& e, PyObject* const* args, Py_ssize_t n, PyObject* kwnames) {
  PyObject* ordered[kMaxArgs];
  if (n != e.n_args || (kwnames && PyTuple_GET_SIZE(kwnames) > 0)) {   // by name: put them in order
    const Py_ssize_t n_kw = kwnames ? PyTuple_GET_SIZE(kwnames) : 0;
    if (n + n_kw != e.n_args) {
      PyErr_Format(PyExc_TypeError, "%s() takes %d arguments (%zd given)", e.name, e.n_args, n + n_kw);
      return nullptr;
    }
    for (int i = 0; i < e.n_args; ++i) ordered[i] = i < n ? args[i] : nullptr;
    for (Py_ssize_t k = 0; k < n_kw; ++k) {
      PyObject* key = PyTuple_GET_ITEM(kwnames, k);
      int at = -1;
      for (int i = 0; i < e.n_args; ++i)
        if (PyUnicode_CompareWithASCIIString(key, e.arg_names[i]) == 0) at = i;
      if (at < 0 || ordered[at]) {
        PyErr_Format(PyExc_TypeError, "%s() got an unexpected or repeated argument '%U'", e.name, key);
        return nullptr;
      }
      ordered[at] = args[n + k];
    }
    args = ordered;
  }
  Args a{args};
  const int rc = e.call(a);
  if (a.failed) return nullptr;
  if (rc != DLM_OK) {
    PyObject* err = g_error ? PyObject_CallFunction(g_error, "is", rc, e.name) : nullptr;
    if (err) {
      PyErr_SetObject(g_error, err);
      Py_DECREF(err);
    } else if (!PyErr_Occurred()) {
      PyErr_Format(PyExc_RuntimeError, "%s: %s (%d)", e.name, dlm_strerror(rc), rc);
    }
    return nullptr;
  }
  Py_RETURN_NONE;
}

template <int I>
PyObject* trampoline(PyObject*, PyObject* const* args, Py_ssize_t n, PyObject* kwnames) {
  try {
    return run(kEntries[I], args, n, kwnames);
  } catch (const std::exception& e) {
    PyErr_SetString(PyExc_RuntimeError, e.what());
    return nullptr;
  }
}

PyObject* set_error(PyObject*, PyObject* cls) {
  Py_XINCREF(cls);
  Py_XSETREF(g_error, cls);
  Py_RETURN_NONE;
}

PyObject* set_types(PyObject*, PyObject* args) {
  PyObject *handle, *cache;
  if (!PyArg_ParseTuple(args, "O!O!", &PyType_Type, &handle, &PyType_Type, &cache)) return nullptr;
  Py_INCREF(handle);
  Py_INCREF(cache);
  Py_XSETREF(g_handle_type, reinterpret_cast<PyTypeObject*>(handle));
  Py_XSETREF(g_cache_type, reinterpret_cast<PyTypeObject*>(cache));
  Py_RETURN_NONE;
}

PyMethodDef g_methods[kNumEntries + 3];

template <int... I>
void fill_methods(std::integer_sequence<int, I...>) {
  ((g_methods[I] = {kEntries[I].name, (PyCFunction)(void*)trampoline<I>, METH_FASTCALL | METH_KEYWORDS, nullptr}), ...);
}

PyModuleDef g_module = {PyModuleDef_HEAD_INIT, "_dlm_calls", nullptr, -1, g_methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

#ifndef DLM_CALLS_BUILT_FOR   // the torch, the Python and the sources of this build (build.py)
#define DLM_CALLS_BUILT_FOR "unknown"
#endif

PyMODINIT_FUNC PyInit__dlm_calls() {
  fill_methods(std::make_integer_sequence<int, kNumEntries>());
  g_methods[kNumEntries] = {"set_error", set_error, METH_O, nullptr};
  g_methods[kNumEntries + 1] = {"set_types", set_types, METH_VARARGS, nullptr};
  PyObject* m = PyModule_Create(&g_module);
  if (m && PyModule_AddStringConstant(m, "built_for", DLM_CALLS_BUILT_FOR) != 0) Py_CLEAR(m);
  return m;
}
