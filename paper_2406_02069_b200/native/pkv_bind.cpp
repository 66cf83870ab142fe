// Native half of the Python binding: checks the tensors of a call and hands it to the C boundary
// (include/pyramidkv.h) without going through ctypes.
//
// A per-layer call on a short context takes the GPU some 20 us, and one decode step makes a call per layer, so what the
// host spends per call is what such programs wait for.  Checks through tensor attributes and ctypes marshalling took 25
// of the 32 us that the host needed for a compress_layer call and 6.5 of the 9.3 us of a decode_attention call; with
// this file those calls take 7 and 2.8 us, launches included.
//
// Every function returns the C status (PKV_OK = 0, an error code otherwise), or kNotTaken when an argument is not what
// the quick checks accept: another kind of object, memory that is not on a CUDA device, a tensor that is too small.
// Nothing has been enqueued then; the caller goes through binding.py's own checks, which accept the rarer forms
// (pinned host memory) and raise the error with its reason for the rest.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <algorithm>
#include <cstring>
#include <vector>

#include <ATen/core/Tensor.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "pyramidkv.h"

namespace {

constexpr int kNotTaken = -1;
PyObject* g_config_type = nullptr;       // PkvConfig: other objects that expose a buffer of its size are not configurations

// A tensor argument as the checks need it (borrowed: the arguments outlive the call).
struct View {
  const at::Tensor* t = nullptr;
  explicit operator bool() const { return t != nullptr; }
  void* ptr() const { return t->data_ptr(); }
  int64_t size(int i) const { return t->sizes()[i]; }
  int64_t stride(int i) const { return t->strides()[i]; }
  pkv_tensor strided() const { return pkv_tensor{t->data_ptr(), stride(0), stride(1), stride(2)}; }
};

bool get(PyObject* o, View* v) {
  if (!THPVariable_Check(o)) return false;
  const at::Tensor& t = THPVariable_Unpack(o);
  if (!t.defined() || t.layout() != c10::kStrided || !t.is_cuda() || !t.has_storage()) return false;
  v->t = &t;
  return true;
}

c10::ScalarType scalar_type(const pkv_config* c) {
  return c->dtype == PKV_DTYPE_FP32 ? c10::kFloat : (c->dtype == PKV_DTYPE_BF16 ? c10::kBFloat16 : c10::kHalf);
}

// What every call starts with: the configuration, the lengths and the stream.
struct Call {
  Py_buffer buf{};
  const pkv_config* cfg = nullptr;
  int32_t lens[PKV_MAX_BATCH];
  int32_t batch = 0;
  int32_t longest = 0;
  void* stream = nullptr;

  ~Call() { if (cfg) PyBuffer_Release(&buf); }

  bool open(PyObject* config, PyObject* seq_lens) {
    if (!g_config_type || PyObject_IsInstance(config, g_config_type) != 1) { PyErr_Clear(); return false; }
    if (PyObject_GetBuffer(config, &buf, PyBUF_SIMPLE) != 0) { PyErr_Clear(); return false; }
    cfg = static_cast<const pkv_config*>(buf.buf);               // released by the destructor from here on
    if (buf.len != static_cast<Py_ssize_t>(sizeof(pkv_config))) return false;
    if (cfg->num_kv_heads < 1 || cfg->dtype < PKV_DTYPE_FP32 || cfg->dtype > PKV_DTYPE_FP16) return false;
    const bool list = PyList_Check(seq_lens);
    if (!list && !PyTuple_Check(seq_lens)) return false;
    const Py_ssize_t n = list ? PyList_GET_SIZE(seq_lens) : PyTuple_GET_SIZE(seq_lens);
    if (n < 1 || n > PKV_MAX_BATCH) return false;
    for (Py_ssize_t i = 0; i < n; ++i) {
      PyObject* o = list ? PyList_GET_ITEM(seq_lens, i) : PyTuple_GET_ITEM(seq_lens, i);
      if (!PyLong_CheckExact(o)) return false;
      const long v = PyLong_AsLong(o);
      if ((v == -1 && PyErr_Occurred()) || v < cfg->window + 1l || v > INT32_MAX) { PyErr_Clear(); return false; }
      lens[i] = static_cast<int32_t>(v);
      longest = std::max(longest, lens[i]);
    }
    batch = static_cast<int32_t>(n);
    return true;
  }

  // Last of the checks: the current stream is only asked for once the tensors are known to live on a device.
  bool on_stream(PyObject* stream_or_none) {
    if (stream_or_none == Py_None) {
      stream = c10::cuda::getCurrentCUDAStream().stream();
    } else {
      PyObject* s = PyObject_GetAttrString(stream_or_none, "cuda_stream");
      if (!s) { PyErr_Clear(); return false; }
      stream = PyLong_AsVoidPtr(s);
      Py_DECREF(s);
      if (PyErr_Occurred()) { PyErr_Clear(); return false; }
    }
    return true;
  }

  // A K or V tensor as large as the call will read.
  bool kv(PyObject* o, View* v) const {
    return get(o, v) && v->t->dim() == 4 && v->stride(3) == 1 && v->t->scalar_type() == scalar_type(cfg) && v->size(0) >= batch &&
           v->size(1) == cfg->num_kv_heads && v->size(3) == cfg->head_dim && v->size(2) >= longest &&
           (batch == 1 || v->stride(0) > 0) && (cfg->num_kv_heads == 1 || v->stride(1) > 0) && v->stride(2) >= cfg->head_dim;
  }
  bool q(PyObject* o, View* v) const {
    return get(o, v) && v->t->dim() == 4 && v->stride(3) == 1 && v->t->scalar_type() == scalar_type(cfg) && v->size(0) >= batch &&
           v->size(1) == cfg->num_q_heads && v->size(2) == cfg->window && v->size(3) == cfg->head_dim;
  }
  bool scores(PyObject* o, View* v) const {
    const int64_t columns = longest - cfg->window;
    return get(o, v) && v->t->dim() == 3 && v->t->scalar_type() == c10::kFloat && v->size(0) >= batch &&
           v->size(1) == cfg->num_kv_heads && v->size(2) >= columns && v->stride(2) == 1 && v->stride(1) >= columns &&
           (batch == 1 || v->stride(0) == cfg->num_kv_heads * v->stride(1));
  }
  // A contiguous tensor of a type with at least so many elements.
  static bool flat(PyObject* o, View* v, c10::ScalarType type, int64_t least) {
    return get(o, v) && v->t->scalar_type() == type && v->t->is_contiguous() && v->t->numel() >= least;
  }
  bool lse(PyObject* o, View* v) const {
    return flat(o, v, c10::kFloat, static_cast<int64_t>(batch) * cfg->num_q_heads * cfg->window);
  }
  bool rows_out(PyObject* k, PyObject* v, PyObject* idx, int64_t rows, View* kv_, View* vv, View* iv) const {
    return flat(k, kv_, scalar_type(cfg), rows * cfg->head_dim) && flat(v, vv, scalar_type(cfg), rows * cfg->head_dim) &&
           flat(idx, iv, c10::kInt, rows);
  }
  static bool workspace(PyObject* o, View* v) { return flat(o, v, c10::kByte, 1); }
  bool attn_out(PyObject* o, View* v) const {
    return flat(o, v, c10::kFloat, 0) && v->t->dim() == 4 && v->size(0) == batch && v->size(1) == cfg->num_q_heads &&
           v->size(2) == cfg->window && v->size(3) == cfg->head_dim;
  }
  // Packed rows of a layer with budget k_layer, or a negative number for a configuration the library refuses.
  int64_t packed_rows(int32_t k_layer) const {
    int64_t rows = 0;
    for (int b = 0; b < batch; ++b) {
      const int c = pyramidkv_kept_count(cfg, k_layer, lens[b]);
      if (c < 0) return -1;
      rows += c;
    }
    return rows * cfg->num_kv_heads;
  }
  // ... of layer `layer`; the schedule of the last configuration is remembered per thread.
  int64_t layer_rows(int64_t layer) const {
    thread_local pkv_config last{};
    thread_local std::vector<int32_t> budgets;
    if (layer < 0 || layer >= cfg->num_layers) return -1;
    if (budgets.empty() || std::memcmp(&last, cfg, sizeof last) != 0) {
      budgets.assign(static_cast<size_t>(cfg->num_layers), 0);
      if (pyramidkv_layer_budgets(cfg, budgets.data()) != PKV_OK) { budgets.clear(); return -1; }
      last = *cfg;
    }
    return packed_rows(budgets[static_cast<size_t>(layer)]);
  }
};

bool as_int32(PyObject* o, int32_t* out) {
  if (!PyLong_Check(o)) return false;
  const long v = PyLong_AsLong(o);
  if (v < INT32_MIN || v > INT32_MAX || (v == -1 && PyErr_Occurred())) { PyErr_Clear(); return false; }
  *out = static_cast<int32_t>(v);
  return true;
}

PyObject* status(int rc) { return PyLong_FromLong(rc); }
PyObject* not_taken() { return PyLong_FromLong(kNotTaken); }

// Runs the C call with the interpreter's lock released, as ctypes does; the lock is taken again also when it throws.
template <typename F>
PyObject* without_gil(F&& f) {
  struct Release {
    PyThreadState* state = PyEval_SaveThread();
    ~Release() { PyEval_RestoreThread(state); }
  };
  int rc;
  {
    Release unlocked;
    rc = f();
  }
  return status(rc);
}

// (cfg, layer, q_win, k, v, seq_lens, k_out, v_out, indices, workspace, scores, stream, window_lse)
PyObject* compress_layer(PyObject*, PyObject* const* a, Py_ssize_t n) {
  Call c;
  View q, k, v, ko, vo, idx, ws, sc, lse;
  int32_t layer;
  if (n != 13 || !as_int32(a[1], &layer) || !c.open(a[0], a[5])) return not_taken();
  const int64_t rows = c.layer_rows(layer);
  if (rows < 0 || !c.q(a[2], &q) || !c.kv(a[3], &k) || !c.kv(a[4], &v) || !c.rows_out(a[6], a[7], a[8], rows, &ko, &vo, &idx) ||
      !Call::workspace(a[9], &ws) || (a[10] != Py_None && !c.scores(a[10], &sc)) || (a[12] != Py_None && !c.lse(a[12], &lse)) ||
      !c.on_stream(a[11]))
    return not_taken();
  float* s = sc ? static_cast<float*>(sc.ptr()) : nullptr;
  const int64_t ld = sc ? sc.stride(1) : 0;
  return without_gil([&] {
    return lse ? pyramidkv_compress_layer_lse(c.cfg, layer, q.strided(), k.strided(), v.strided(), static_cast<const float*>(lse.ptr()),
                                              c.lens, c.batch, ko.ptr(), vo.ptr(), static_cast<int32_t*>(idx.ptr()), s, ld, ws.ptr(),
                                              static_cast<size_t>(ws.t->numel()), c.stream)
               : pyramidkv_compress_layer(c.cfg, layer, q.strided(), k.strided(), v.strided(), c.lens, c.batch, ko.ptr(), vo.ptr(),
                                          static_cast<int32_t*>(idx.ptr()), s, ld, ws.ptr(), static_cast<size_t>(ws.t->numel()),
                                          c.stream);
  });
}

// (cfg, layer, q_win, k, v, seq_lens, attn_out, k_out, v_out, indices, workspace, scores, stream)
PyObject* attend_compress_layer(PyObject*, PyObject* const* a, Py_ssize_t n) {
  Call c;
  View q, k, v, at, ko, vo, idx, ws, sc;
  int32_t layer;
  if (n != 13 || !as_int32(a[1], &layer) || !c.open(a[0], a[5])) return not_taken();
  const int64_t rows = c.layer_rows(layer);
  if (rows < 0 || !c.q(a[2], &q) || !c.kv(a[3], &k) || !c.kv(a[4], &v) || !c.attn_out(a[6], &at) ||
      !c.rows_out(a[7], a[8], a[9], rows, &ko, &vo, &idx) || !Call::workspace(a[10], &ws) ||
      (a[11] != Py_None && !c.scores(a[11], &sc)) || !c.on_stream(a[12]))
    return not_taken();
  return without_gil([&] {
    return pyramidkv_attend_compress_layer(c.cfg, layer, q.strided(), k.strided(), v.strided(), c.lens, c.batch,
                                           static_cast<float*>(at.ptr()), ko.ptr(), vo.ptr(), static_cast<int32_t*>(idx.ptr()),
                                           sc ? static_cast<float*>(sc.ptr()) : nullptr, sc ? sc.stride(1) : 0, ws.ptr(),
                                           static_cast<size_t>(ws.t->numel()), c.stream);
  });
}

// Block table and pools of a paged call: [num_pages][page_size][d] pools of one shape.
bool paged(const Call& c, PyObject* table, PyObject* k, PyObject* v, View* tab, View* kp, View* vp) {
  return Call::flat(table, tab, c10::kInt, 0) && Call::flat(k, kp, scalar_type(c.cfg), 1) && Call::flat(v, vp, scalar_type(c.cfg), 1) &&
         kp->t->dim() == 3 && kp->t->sizes() == vp->t->sizes() && kp->size(2) == c.cfg->head_dim && kp->size(0) <= INT32_MAX &&
         kp->size(1) <= INT32_MAX;
}

// (cfg, layer, q_win, k, v, seq_lens, block_table, k_pool, v_pool, indices, workspace, scores, stream, window_lse)
PyObject* compress_layer_paged(PyObject*, PyObject* const* a, Py_ssize_t n) {
  Call c;
  View q, k, v, tab, kp, vp, idx, ws, sc, lse;
  int32_t layer;
  if (n != 14 || !as_int32(a[1], &layer) || !c.open(a[0], a[5])) return not_taken();
  const int64_t rows = c.layer_rows(layer);
  if (rows < 0 || !c.q(a[2], &q) || !c.kv(a[3], &k) || !c.kv(a[4], &v) || !paged(c, a[6], a[7], a[8], &tab, &kp, &vp) ||
      !Call::flat(a[9], &idx, c10::kInt, rows) || !Call::workspace(a[10], &ws) || (a[11] != Py_None && !c.scores(a[11], &sc)) ||
      (a[13] != Py_None && !c.lse(a[13], &lse)) || !c.on_stream(a[12]))
    return not_taken();
  return without_gil([&] {
    return pyramidkv_compress_layer_paged(
        c.cfg, layer, q.strided(), k.strided(), v.strided(), lse ? static_cast<const float*>(lse.ptr()) : nullptr, c.lens, c.batch,
        static_cast<const int32_t*>(tab.ptr()), static_cast<int32_t>(kp.size(1)), static_cast<int32_t>(kp.size(0)), kp.ptr(), vp.ptr(),
        static_cast<int32_t*>(idx.ptr()), sc ? static_cast<float*>(sc.ptr()) : nullptr, sc ? sc.stride(1) : 0, ws.ptr(),
        static_cast<size_t>(ws.t->numel()), c.stream);
  });
}

// (cfg, q_win, k, seq_lens, scores, workspace, stream, window_lse)
PyObject* score_window(PyObject*, PyObject* const* a, Py_ssize_t n) {
  Call c;
  View q, k, sc, ws, lse;
  if (n != 8 || !c.open(a[0], a[3]) || !c.q(a[1], &q) || !c.kv(a[2], &k) || !c.scores(a[4], &sc) || !Call::workspace(a[5], &ws) ||
      (a[7] != Py_None && !c.lse(a[7], &lse)) || !c.on_stream(a[6]))
    return not_taken();
  float* s = static_cast<float*>(sc.ptr());
  return without_gil([&] {
    return lse ? pyramidkv_score_window_lse(c.cfg, q.strided(), k.strided(), static_cast<const float*>(lse.ptr()), c.lens, c.batch, s,
                                            sc.stride(1), ws.ptr(), static_cast<size_t>(ws.t->numel()), c.stream)
               : pyramidkv_score_window(c.cfg, q.strided(), k.strided(), c.lens, c.batch, s, sc.stride(1), ws.ptr(),
                                        static_cast<size_t>(ws.t->numel()), c.stream);
  });
}

// (cfg, scores, seq_lens, k_layer, indices, workspace, stream)
PyObject* select_topk(PyObject*, PyObject* const* a, Py_ssize_t n) {
  Call c;
  View sc, idx, ws;
  int32_t kl;
  if (n != 7 || !as_int32(a[3], &kl) || !c.open(a[0], a[2]) || !c.scores(a[1], &sc)) return not_taken();
  const int64_t rows = c.packed_rows(kl);
  if (rows < 0 || !Call::flat(a[4], &idx, c10::kInt, rows) || !Call::workspace(a[5], &ws) || !c.on_stream(a[6])) return not_taken();
  return without_gil([&] {
    return pyramidkv_select_topk(c.cfg, static_cast<const float*>(sc.ptr()), sc.stride(1), c.lens, c.batch, kl,
                                 static_cast<int32_t*>(idx.ptr()), ws.ptr(), static_cast<size_t>(ws.t->numel()), c.stream);
  });
}

// (cfg, k, v, indices, seq_lens, k_layer, k_out, v_out, stream)
PyObject* gather_compact(PyObject*, PyObject* const* a, Py_ssize_t n) {
  Call c;
  View k, v, idx, ko, vo;
  int32_t kl;
  if (n != 9 || !as_int32(a[5], &kl) || !c.open(a[0], a[4]) || !c.kv(a[1], &k) || !c.kv(a[2], &v)) return not_taken();
  const int64_t rows = c.packed_rows(kl);
  if (rows < 0 || !c.rows_out(a[6], a[7], a[3], rows, &ko, &vo, &idx) || !c.on_stream(a[8])) return not_taken();
  return without_gil([&] {
    return pyramidkv_gather_compact(c.cfg, k.strided(), v.strided(), static_cast<const int32_t*>(idx.ptr()), c.lens, c.batch, kl,
                                    ko.ptr(), vo.ptr(), c.stream);
  });
}

// (cfg, q, k_cache, v_cache, seq_lens, k_layer, out, stream)
PyObject* decode_attention(PyObject*, PyObject* const* a, Py_ssize_t n) {
  Call c;
  View q, k, v, out;
  int32_t kl;
  if (n != 8 || !as_int32(a[5], &kl) || !c.open(a[0], a[4])) return not_taken();
  const int64_t rows = c.packed_rows(kl), elems = static_cast<int64_t>(c.batch) * c.cfg->num_q_heads * c.cfg->head_dim;
  const c10::ScalarType type = scalar_type(c.cfg);
  if (rows < 0 || !Call::flat(a[1], &q, type, elems) || !Call::flat(a[2], &k, type, rows * c.cfg->head_dim) ||
      !Call::flat(a[3], &v, type, rows * c.cfg->head_dim) || !Call::flat(a[6], &out, c10::kFloat, elems) || !c.on_stream(a[7]))
    return not_taken();
  return without_gil([&] {
    return pyramidkv_decode_attention(c.cfg, q.ptr(), k.ptr(), v.ptr(), c.lens, c.batch, kl, static_cast<float*>(out.ptr()), c.stream);
  });
}

// (cfg, q, block_table, k_pool, v_pool, seq_lens, k_layer, out, workspace, stream)
PyObject* decode_attention_paged(PyObject*, PyObject* const* a, Py_ssize_t n) {
  Call c;
  View q, tab, kp, vp, out, ws;
  int32_t kl;
  if (n != 10 || !as_int32(a[6], &kl) || !c.open(a[0], a[5])) return not_taken();
  const int64_t elems = static_cast<int64_t>(c.batch) * c.cfg->num_q_heads * c.cfg->head_dim;
  if (!Call::flat(a[1], &q, scalar_type(c.cfg), elems) || !paged(c, a[2], a[3], a[4], &tab, &kp, &vp) ||
      !Call::flat(a[7], &out, c10::kFloat, elems) || !Call::workspace(a[8], &ws) || !c.on_stream(a[9]))
    return not_taken();
  return without_gil([&] {
    return pyramidkv_decode_attention_paged(c.cfg, q.ptr(), kp.ptr(), vp.ptr(), static_cast<const int32_t*>(tab.ptr()),
                                            static_cast<int32_t>(kp.size(1)), static_cast<int32_t>(kp.size(0)), c.lens, c.batch, kl,
                                            static_cast<float*>(out.ptr()), ws.ptr(), static_cast<size_t>(ws.t->numel()), c.stream);
  });
}

// A tensor that cannot be asked for its data (a fake one, say) or a CUDA runtime that does not answer throws: left to the
// other path too.
template <PyObject* (*F)(PyObject*, PyObject* const*, Py_ssize_t)>
PyObject* guarded(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  try {
    return F(self, a, n);
  } catch (...) {
    PyErr_Clear();
    return not_taken();
  }
}

// (type): the class of the configurations.
PyObject* set_config_type(PyObject*, PyObject* type) {
  Py_INCREF(type);
  Py_XDECREF(g_config_type);
  g_config_type = type;
  Py_RETURN_NONE;
}

#define PKV_METHOD(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)(void)>(guarded<name>)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {PKV_METHOD(compress_layer), PKV_METHOD(attend_compress_layer), PKV_METHOD(compress_layer_paged),
                         PKV_METHOD(score_window), PKV_METHOD(select_topk), PKV_METHOD(gather_compact), PKV_METHOD(decode_attention),
                         PKV_METHOD(decode_attention_paged), {"set_config_type", set_config_type, METH_O, nullptr}, {nullptr, nullptr, 0, nullptr}};
PyModuleDef module_def = {PyModuleDef_HEAD_INIT, "_pkv_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__pkv_native() { return PyModule_Create(&module_def); }
