// _jetcall: the Python side of the C ABI's call path, in C++.
//
// An entry point takes up to thirty arguments, ten of them tensors.  Marshalled by ctypes from Python a call cost
// 11 - 20 us of host time (data_ptr() of every tensor, the current stream, one conversion object per argument), more
// than the kernels of a small call take; here it is one pass over the argument vector, 0.5 us for the twenty-nine
// arguments of an attention call.  (A commit of one launch as a whole: 11.3 -> 3.0 us, a step of four: 64 -> 14 - 22 us, by host.)
// Only argument marshalling lives here: every function calls the C function of the same name in libjet.so with the GIL
// released and returns its status.
//
// A device pointer is None, an int, a torch tensor, or anything with a data_ptr() method.  Plain tensors (and Parameters) are
// read natively; a subclass is asked through its own Python methods, which it may override.  A tensor without an address
// (sparse, wrapped by a transform) makes at::Tensor throw: the entry points below turn that into the Python exception
// that the tensor's own method raises (see guarded).
#include <Python.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include "jet.h"

extern "C" jet_status jet_internal_tree_build_step(
    const float* rows, int64_t batch_stride, int64_t depth_stride, const int32_t* root_token, int batch, int N, int V, int W, int B,
    const int32_t* node_budget, int score_mode, float alpha, int32_t* parent, int32_t* depth, int32_t* token, float* score,
    uint32_t* anc_mask, int32_t* n_nodes, float* depth_entropy, float* depth_lse, int from_logits, const int32_t* len_src,
    int32_t* len_dst, void* workspace, size_t workspace_bytes, void* stream);
extern "C" jet_status jet_internal_kv_compact_step(
    const void* tree_k, const void* tree_v, void* k_cache, void* v_cache, int64_t cache_layer_stride, int64_t kv_batch_stride,
    const int32_t* page_table, int max_pages_per_seq, int page_size, const int32_t* path, const int32_t* accept_len, int32_t* seq_len,
    int layers, int batch, int B, int Hkv, int D, int N, int tail, int32_t* arrived, void* stream);
extern "C" jet_status jet_internal_accept_commit(
    const void* rows, int64_t row_stride, const void* lm_head_weight, int d, const int32_t* token, const int32_t* parent,
    const int32_t* depth, const uint32_t* anc_mask, const int32_t* n_nodes, int batch, int B, int V, int N, int32_t* tgt_argmax,
    int32_t* accept_len, int32_t* path, int32_t* out_tokens, int32_t* device_status, void* workspace, size_t workspace_bytes,
    const void* tree_k, const void* tree_v, void* k_cache, void* v_cache, int64_t cache_layer_stride, int64_t kv_batch_stride,
    const int32_t* page_table, int max_pages_per_seq, int page_size, int32_t* seq_len, int layers, int Hkv, int D, int tail,
    int32_t* arrived, void* stream);
extern "C" int jet_internal_accept_commit_launches(int hidden, int layers, int batch, int B, int V, int Hkv, int D, int N, int tail);

namespace {

// Walks the positional arguments of one call; after the first conversion error every further read returns 0.
class Args {
 public:
  Args(PyObject* const* argv, Py_ssize_t argc, Py_ssize_t want) : argv_(argv) {
    if (argc != want) {
      PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, argc);
      bad_ = true;
    }
  }
  bool bad() const { return bad_; }

  void* ptr() {
    PyObject* o = next();
    return o ? address(o) : nullptr;
  }
  // Element `layer` of the leading dimension of a stacked tensor (None and plain addresses as in ptr()).
  void* layer_ptr(int64_t layer) {
    PyObject* o = next();
    if (!o) return nullptr;
    if (!THPVariable_Check(o)) return address(o);
    if (!THPVariable_CheckExact(o)) {
      PyObject* index = PyLong_FromLongLong(layer);
      PyObject* slice = index ? PyObject_GetItem(o, index) : nullptr;
      if (!slice) bad_ = true;
      void* p = slice ? address(slice) : nullptr;
      Py_XDECREF(slice);
      Py_XDECREF(index);
      return p;
    }
    const at::Tensor& t = THPVariable_Unpack(o);
    const int64_t n = t.dim() > 0 ? t.size(0) : 0;
    if (layer < -n || layer >= n) {
      PyErr_Format(PyExc_IndexError, "layer %lld is out of range for %lld layers", static_cast<long long>(layer),
                   static_cast<long long>(n));
      bad_ = true;
      return nullptr;
    }
    if (layer < 0) layer += n;
    return static_cast<char*>(t.data_ptr()) + layer * t.stride(0) * static_cast<int64_t>(t.element_size());
  }
  // Workspace pointer and its size in bytes; the size argument that follows may be None (= the tensor's own).
  void* workspace(size_t* bytes) {
    PyObject* o = next();
    PyObject* n = next();
    if (!o || !n) return nullptr;
    void* p = address(o);
    *bytes = 0;
    if (n != Py_None) {
      *bytes = static_cast<size_t>(as_int(n));
    } else if (THPVariable_Check(o)) {
      const at::Tensor& t = THPVariable_Unpack(o);
      *bytes = static_cast<size_t>(t.numel()) * t.element_size();
    } else if (o != Py_None) {
      PyErr_SetString(PyExc_TypeError, "a workspace given by address needs workspace_bytes");
      bad_ = true;
    }
    return p;
  }
  int64_t i64() {
    PyObject* o = next();
    return o ? as_int(o) : 0;
  }
  int i32() {
    const int64_t v = i64();
    if (v < INT32_MIN || v > INT32_MAX) {
      if (!bad_) PyErr_SetString(PyExc_OverflowError, "argument does not fit in 32 bits");
      bad_ = true;
    }
    return static_cast<int>(v);
  }
  float f32() {
    PyObject* o = next();
    if (!o) return 0.0f;
    const double v = PyFloat_AsDouble(o);
    if (v == -1.0 && PyErr_Occurred()) bad_ = true;
    return static_cast<float>(v);
  }
  // None = torch's current stream of the current device, an int, or an object with a cuda_stream attribute.
  void* stream() {
    PyObject* o = next();
    if (!o) return nullptr;
    if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
    if (PyLong_Check(o)) return PyLong_AsVoidPtr(o);
    PyObject* s = PyObject_GetAttrString(o, "cuda_stream");
    void* p = s ? PyLong_AsVoidPtr(s) : nullptr;
    Py_XDECREF(s);
    if (PyErr_Occurred()) bad_ = true;
    return p;
  }

 private:
  PyObject* next() { return bad_ ? nullptr : argv_[i_++]; }
  int64_t as_int(PyObject* o) {
    const int64_t v = PyLong_AsLongLong(o);
    if (v == -1 && PyErr_Occurred()) bad_ = true;
    return v;
  }
  void* address(PyObject* o) {
    if (o == Py_None) return nullptr;
    if (THPVariable_CheckExact(o)) return THPVariable_Unpack(o).data_ptr();
    PyObject* v = PyLong_Check(o) ? Py_NewRef(o) : PyObject_CallMethod(o, "data_ptr", nullptr);
    void* p = v ? PyLong_AsVoidPtr(v) : nullptr;
    Py_XDECREF(v);
    if (PyErr_Occurred()) bad_ = true;
    return p;
  }
  PyObject* const* argv_;
  Py_ssize_t i_ = 0;
  bool bad_ = false;
};

template <typename T>
const T* in(void* p) { return static_cast<const T*>(p); }
template <typename T>
T* out(void* p) { return static_cast<T*>(p); }

class WithoutGil {
 public:
  WithoutGil() : state_(PyEval_SaveThread()) {}
  ~WithoutGil() { PyEval_RestoreThread(state_); }

 private:
  PyThreadState* state_;
};

#define JET_CALL(expr)                       \
  do {                                       \
    if (a.bad()) return nullptr;             \
    jet_status status;                       \
    {                                        \
      WithoutGil no_gil;                     \
      status = (expr);                       \
    }                                        \
    return PyLong_FromLong(status);          \
  } while (0)

using Entry = PyObject* (*)(PyObject*, PyObject* const*, Py_ssize_t);

// An exception that leaves a function the interpreter calls ends the process; here it becomes a Python exception.
template <Entry kEntry>
PyObject* guarded(PyObject* self, PyObject* const* argv, Py_ssize_t argc) {
  HANDLE_TH_ERRORS
  return kEntry(self, argv, argc);
  END_HANDLE_TH_ERRORS
}

// Strides of [batch, N, V] rows: given, or None = those of the tensor itself.
void row_strides(PyObject* rows, PyObject* const* given, int64_t (&s)[2], bool* bad) {
  for (int d = 0; d < 2; ++d) {
    if (given[d] == Py_None && THPVariable_CheckExact(rows) && THPVariable_Unpack(rows).dim() > d) {
      s[d] = THPVariable_Unpack(rows).stride(d);
    } else if (given[d] == Py_None && THPVariable_Check(rows)) {
      PyObject* v = PyObject_CallMethod(rows, "stride", "i", d);
      s[d] = v ? PyLong_AsLongLong(v) : -1;
      Py_XDECREF(v);
      if (s[d] == -1 && PyErr_Occurred()) { *bad = true; return; }
    } else {
      s[d] = PyLong_AsLongLong(given[d]);
      if (s[d] == -1 && PyErr_Occurred()) { *bad = true; return; }
    }
  }
}

// (rows, batch_stride, depth_stride, root_token, batch, N, V, W, B, parent, depth, token, score, anc_mask, n_nodes,
//  workspace, workspace_bytes, stream)
PyObject* tree_build(PyObject*, PyObject* const* argv, Py_ssize_t argc) {
  Args a(argv, argc, 18);
  if (a.bad()) return nullptr;
  int64_t s[2];
  bool bad = false;
  row_strides(argv[0], argv + 1, s, &bad);
  if (bad) return nullptr;
  const float* rows = in<float>(a.ptr());
  Args b(argv + 3, argc - 3, 15);
  const int32_t* root = in<int32_t>(b.ptr());
  const int batch = b.i32(), N = b.i32(), V = b.i32(), W = b.i32(), B = b.i32();
  int32_t* parent = out<int32_t>(b.ptr());
  int32_t* depth = out<int32_t>(b.ptr());
  int32_t* token = out<int32_t>(b.ptr());
  float* score = out<float>(b.ptr());
  uint32_t* anc = out<uint32_t>(b.ptr());
  int32_t* n_nodes = out<int32_t>(b.ptr());
  size_t wb = 0;
  void* ws = b.workspace(&wb);
  void* st = b.stream();
  if (b.bad()) return nullptr;
  JET_CALL(jet_tree_build(rows, s[0], s[1], root, batch, N, V, W, B, parent, depth, token, score, anc, n_nodes, ws, wb, st));
}

// (rows, batch_stride, depth_stride, root_token, batch, N, V, W, B, node_budget, score_mode, alpha, parent, depth, token,
//  score, anc_mask, n_nodes, depth_entropy, depth_lse, from_logits, workspace, workspace_bytes, stream, len_src, len_dst);
// len_dst not None: the same call also sets len_dst = len_src.
PyObject* tree_build_scored(PyObject*, PyObject* const* argv, Py_ssize_t argc) {
  Args a(argv, argc, 26);
  if (a.bad()) return nullptr;
  int64_t s[2];
  bool bad = false;
  row_strides(argv[0], argv + 1, s, &bad);
  if (bad) return nullptr;
  const float* rows = in<float>(a.ptr());
  Args b(argv + 3, argc - 3, 23);
  const int32_t* root = in<int32_t>(b.ptr());
  const int batch = b.i32(), N = b.i32(), V = b.i32(), W = b.i32(), B = b.i32();
  const int32_t* budget = in<int32_t>(b.ptr());
  const int mode = b.i32();
  const float alpha = b.f32();
  int32_t* parent = out<int32_t>(b.ptr());
  int32_t* depth = out<int32_t>(b.ptr());
  int32_t* token = out<int32_t>(b.ptr());
  float* score = out<float>(b.ptr());
  uint32_t* anc = out<uint32_t>(b.ptr());
  int32_t* n_nodes = out<int32_t>(b.ptr());
  float* entropy = out<float>(b.ptr());
  float* lse = out<float>(b.ptr());
  const bool from_logits = b.i32() != 0;
  size_t wb = 0;
  void* ws = b.workspace(&wb);
  void* st = b.stream();
  const int32_t* len_src = in<int32_t>(b.ptr());
  int32_t* len_dst = out<int32_t>(b.ptr());
  if (b.bad()) return nullptr;
  if (len_dst)
    JET_CALL(jet_internal_tree_build_step(rows, s[0], s[1], root, batch, N, V, W, B, budget, mode, alpha, parent, depth, token,
                                          score, anc, n_nodes, entropy, lse, from_logits ? 1 : 0, len_src, len_dst, ws, wb, st));
  JET_CALL(from_logits ? jet_tree_build_logits(rows, s[0], s[1], root, batch, N, V, W, B, budget, mode, alpha, parent, depth,
                                               token, score, anc, n_nodes, entropy, lse, ws, wb, st)
                       : jet_tree_build_scored(rows, s[0], s[1], root, batch, N, V, W, B, budget, mode, alpha, parent, depth,
                                               token, score, anc, n_nodes, entropy, ws, wb, st));
}

// (layer, q, k_cache, v_cache, page_table, max_pages, page_size, num_pages, seq_len, max_seq_len, tree_k, tree_v, anc_mask,
//  n_nodes, batch, B, Hq, Hkv, D, kv_batch_stride, scale, out, lse, device_status, workspace, workspace_bytes, stream, flags,
//  tail).  layer None: the tensors are those of one layer; else q, the caches, tree_k / tree_v and out are stacked.
PyObject* tree_verify_attn(PyObject*, PyObject* const* argv, Py_ssize_t argc) {
  Args a(argv + 1, argc - 1, 28);
  if (a.bad()) return nullptr;
  const bool stacked = argv[0] != Py_None;
  const int64_t layer = stacked ? PyLong_AsLongLong(argv[0]) : 0;
  if (layer == -1 && PyErr_Occurred()) return nullptr;
  auto per_layer = [&] { return stacked ? a.layer_ptr(layer) : a.ptr(); };
  const void* q = per_layer();
  const void* k = per_layer();
  const void* v = per_layer();
  const int32_t* table = in<int32_t>(a.ptr());
  const int max_pages = a.i32(), page_size = a.i32();
  const int64_t num_pages = a.i64();
  const int32_t* seq_len = in<int32_t>(a.ptr());
  const int max_seq_len = a.i32();
  const void* tk = per_layer();
  const void* tv = per_layer();
  const uint32_t* anc = in<uint32_t>(a.ptr());
  const int32_t* n_nodes = in<int32_t>(a.ptr());
  const int batch = a.i32(), B = a.i32(), Hq = a.i32(), Hkv = a.i32(), D = a.i32();
  const int64_t stride = a.i64();
  const float scale = a.f32();
  void* o = per_layer();
  float* lse = out<float>(a.ptr());
  int32_t* dev_status = out<int32_t>(a.ptr());
  size_t wb = 0;
  void* ws = a.workspace(&wb);
  void* st = a.stream();
  const uint32_t flags = static_cast<uint32_t>(a.i64());
  const bool tail = a.i32() != 0;
  JET_CALL(tail ? jet_tree_verify_attn_tail_ex(q, k, v, table, max_pages, page_size, num_pages, seq_len, max_seq_len, anc,
                                               n_nodes, batch, B, Hq, Hkv, D, stride, scale, o, lse, dev_status, ws, wb, st,
                                               flags)
                : jet_tree_verify_attn_ex(q, k, v, table, max_pages, page_size, num_pages, seq_len, max_seq_len, tk, tv, anc,
                                          n_nodes, batch, B, Hq, Hkv, D, stride, scale, o, lse, dev_status, ws, wb, st, flags));
}

// (logits, row_stride, token, parent, depth, anc_mask, n_nodes, batch, B, V, N, tgt_argmax, accept_len, path, out_tokens,
//  workspace, workspace_bytes, stream, static)
PyObject* tree_accept(PyObject*, PyObject* const* argv, Py_ssize_t argc) {
  Args a(argv, argc, 19);
  const float* logits = in<float>(a.ptr());
  const int64_t stride = a.i64();
  const int32_t* token = in<int32_t>(a.ptr());
  const int32_t* parent = in<int32_t>(a.ptr());
  const int32_t* depth = in<int32_t>(a.ptr());
  const uint32_t* anc = in<uint32_t>(a.ptr());
  const int32_t* n_nodes = in<int32_t>(a.ptr());
  const int batch = a.i32(), B = a.i32(), V = a.i32(), N = a.i32();
  int32_t* tgt = out<int32_t>(a.ptr());
  int32_t* len = out<int32_t>(a.ptr());
  int32_t* path = out<int32_t>(a.ptr());
  int32_t* toks = out<int32_t>(a.ptr());
  size_t wb = 0;
  void* ws = a.workspace(&wb);
  void* st = a.stream();
  const bool built_in = a.i32() != 0;
  JET_CALL(built_in ? jet_tree_accept_static(logits, stride, token, parent, depth, anc, n_nodes, batch, B, V, N, tgt, len, path,
                                             toks, st)
                    : jet_tree_accept(logits, stride, token, parent, depth, anc, n_nodes, batch, B, V, N, tgt, len, path, toks,
                                      ws, wb, st));
}

// (hidden, lm_head_weight, d, token, parent, depth, anc_mask, n_nodes, batch, B, V, N, tgt_argmax, accept_len, path,
//  out_tokens, device_status, workspace, workspace_bytes, stream)
PyObject* tree_accept_hidden(PyObject*, PyObject* const* argv, Py_ssize_t argc) {
  Args a(argv, argc, 20);
  const void* hidden = a.ptr();
  const void* weight = a.ptr();
  const int d = a.i32();
  const int32_t* token = in<int32_t>(a.ptr());
  const int32_t* parent = in<int32_t>(a.ptr());
  const int32_t* depth = in<int32_t>(a.ptr());
  const uint32_t* anc = in<uint32_t>(a.ptr());
  const int32_t* n_nodes = in<int32_t>(a.ptr());
  const int batch = a.i32(), B = a.i32(), V = a.i32(), N = a.i32();
  int32_t* tgt = out<int32_t>(a.ptr());
  int32_t* len = out<int32_t>(a.ptr());
  int32_t* path = out<int32_t>(a.ptr());
  int32_t* toks = out<int32_t>(a.ptr());
  int32_t* dev_status = out<int32_t>(a.ptr());
  size_t wb = 0;
  void* ws = a.workspace(&wb);
  void* st = a.stream();
  JET_CALL(jet_tree_accept_hidden(hidden, weight, d, token, parent, depth, anc, n_nodes, batch, B, V, N, tgt, len, path, toks,
                                  dev_status, ws, wb, st));
}

// (logits, row_stride, temperature, draft_logp, logp_batch_stride, logp_depth_stride, token, parent, depth, anc_mask,
//  n_nodes, u_accept, u_sample, batch, B, V, N, alpha, accept_len, path, out_tokens, workspace, workspace_bytes, stream)
PyObject* tree_accept_sample(PyObject*, PyObject* const* argv, Py_ssize_t argc) {
  Args a(argv, argc, 24);
  const float* logits = in<float>(a.ptr());
  const int64_t stride = a.i64();
  const float temperature = a.f32();
  const float* logp = in<float>(a.ptr());
  const int64_t bs = a.i64(), ds = a.i64();
  const int32_t* token = in<int32_t>(a.ptr());
  const int32_t* parent = in<int32_t>(a.ptr());
  const int32_t* depth = in<int32_t>(a.ptr());
  const uint32_t* anc = in<uint32_t>(a.ptr());
  const int32_t* n_nodes = in<int32_t>(a.ptr());
  const float* ua = in<float>(a.ptr());
  const float* us = in<float>(a.ptr());
  const int batch = a.i32(), B = a.i32(), V = a.i32(), N = a.i32();
  float* alpha = out<float>(a.ptr());
  int32_t* len = out<int32_t>(a.ptr());
  int32_t* path = out<int32_t>(a.ptr());
  int32_t* toks = out<int32_t>(a.ptr());
  size_t wb = 0;
  void* ws = a.workspace(&wb);
  void* st = a.stream();
  JET_CALL(jet_tree_accept_sample(logits, stride, temperature, logp, bs, ds, token, parent, depth, anc, n_nodes, ua, us, batch,
                                  B, V, N, alpha, len, path, toks, ws, wb, st));
}

// (tree_k, tree_v, k_cache, v_cache, cache_layer_stride, kv_batch_stride, page_table, max_pages, page_size, path, accept_len,
//  seq_len, layers, batch, B, Hkv, D, N, stream, tail)
PyObject* kv_compact(PyObject*, PyObject* const* argv, Py_ssize_t argc) {
  Args a(argv, argc, 20);
  const void* tk = a.ptr();
  const void* tv = a.ptr();
  void* k = a.ptr();
  void* v = a.ptr();
  const int64_t ls = a.i64(), bs = a.i64();
  const int32_t* table = in<int32_t>(a.ptr());
  const int max_pages = a.i32(), page_size = a.i32();
  const int32_t* path = in<int32_t>(a.ptr());
  const int32_t* len = in<int32_t>(a.ptr());
  int32_t* seq_len = out<int32_t>(a.ptr());
  const int layers = a.i32(), batch = a.i32(), B = a.i32(), Hkv = a.i32(), D = a.i32(), N = a.i32();
  void* st = a.stream();
  const bool tail = a.i32() != 0;
  JET_CALL(tail ? jet_kv_compact_tail(k, v, ls, bs, table, max_pages, page_size, path, len, seq_len, layers, batch, B, Hkv, D,
                                      N, st)
                : jet_kv_compact(tk, tv, k, v, ls, bs, table, max_pages, page_size, path, len, seq_len, layers, batch, B, Hkv,
                                 D, N, st));
}

// (tree_k, tree_v, k_cache, v_cache, cache_layer_stride, kv_batch_stride, page_table, max_pages, page_size, path, accept_len,
//  seq_len, layers, batch, B, Hkv, D, N, tail, arrived, stream)
PyObject* kv_compact_step(PyObject*, PyObject* const* argv, Py_ssize_t argc) {
  Args a(argv, argc, 21);
  const void* tk = a.ptr();
  const void* tv = a.ptr();
  void* k = a.ptr();
  void* v = a.ptr();
  const int64_t ls = a.i64(), bs = a.i64();
  const int32_t* table = in<int32_t>(a.ptr());
  const int max_pages = a.i32(), page_size = a.i32();
  const int32_t* path = in<int32_t>(a.ptr());
  const int32_t* len = in<int32_t>(a.ptr());
  int32_t* seq_len = out<int32_t>(a.ptr());
  const int layers = a.i32(), batch = a.i32(), B = a.i32(), Hkv = a.i32(), D = a.i32(), N = a.i32(), tail = a.i32();
  int32_t* arrived = out<int32_t>(a.ptr());
  void* st = a.stream();
  JET_CALL(jet_internal_kv_compact_step(tk, tv, k, v, ls, bs, table, max_pages, page_size, path, len, seq_len, layers, batch, B, Hkv,
                                        D, N, tail, arrived, st));
}

// (rows, row_stride, lm_head_weight, d, token, parent, depth, anc_mask, n_nodes, batch, B, V, N, tgt_argmax, accept_len, path,
//  out_tokens, device_status, workspace, workspace_bytes, tree_k, tree_v, k_cache, v_cache, cache_layer_stride, kv_batch_stride,
//  page_table, max_pages, page_size, seq_len, layers, Hkv, D, tail, arrived, stream).  lm_head_weight None: rows are logits.
PyObject* accept_commit(PyObject*, PyObject* const* argv, Py_ssize_t argc) {
  Args a(argv, argc, 36);
  const void* rows = a.ptr();
  const int64_t stride = a.i64();
  const void* weight = a.ptr();
  const int d = a.i32();
  const int32_t* token = in<int32_t>(a.ptr());
  const int32_t* parent = in<int32_t>(a.ptr());
  const int32_t* depth = in<int32_t>(a.ptr());
  const uint32_t* anc = in<uint32_t>(a.ptr());
  const int32_t* n_nodes = in<int32_t>(a.ptr());
  const int batch = a.i32(), B = a.i32(), V = a.i32(), N = a.i32();
  int32_t* tgt = out<int32_t>(a.ptr());
  int32_t* len = out<int32_t>(a.ptr());
  int32_t* path = out<int32_t>(a.ptr());
  int32_t* toks = out<int32_t>(a.ptr());
  int32_t* dev_status = out<int32_t>(a.ptr());
  size_t wb = 0;
  void* ws = a.workspace(&wb);
  const void* tk = a.ptr();
  const void* tv = a.ptr();
  void* k = a.ptr();
  void* v = a.ptr();
  const int64_t ls = a.i64(), bs = a.i64();
  const int32_t* table = in<int32_t>(a.ptr());
  const int max_pages = a.i32(), page_size = a.i32();
  int32_t* seq_len = out<int32_t>(a.ptr());
  const int layers = a.i32(), Hkv = a.i32(), D = a.i32(), tail = a.i32();
  int32_t* arrived = out<int32_t>(a.ptr());
  void* st = a.stream();
  JET_CALL(jet_internal_accept_commit(rows, stride, weight, d, token, parent, depth, anc, n_nodes, batch, B, V, N, tgt, len, path, toks,
                                      dev_status, ws, wb, tk, tv, k, v, ls, bs, table, max_pages, page_size, seq_len, layers, Hkv, D,
                                      tail, arrived, st));
}

// (hidden, layers, batch, B, V, Hkv, D, N, tail)
PyObject* accept_commit_launches(PyObject*, PyObject* const* argv, Py_ssize_t argc) {
  Args a(argv, argc, 9);
  const int hidden = a.i32(), layers = a.i32(), batch = a.i32(), B = a.i32(), V = a.i32(), Hkv = a.i32(), D = a.i32(), N = a.i32(),
            tail = a.i32();
  if (a.bad()) return nullptr;
  return PyLong_FromLong(jet_internal_accept_commit_launches(hidden, layers, batch, B, V, Hkv, D, N, tail));
}

#define JET_METHOD(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(guarded<name>)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {JET_METHOD(tree_build),         JET_METHOD(tree_build_scored),  JET_METHOD(tree_verify_attn),
                         JET_METHOD(tree_accept),        JET_METHOD(tree_accept_hidden), JET_METHOD(tree_accept_sample),
                         JET_METHOD(kv_compact),         JET_METHOD(kv_compact_step),    JET_METHOD(accept_commit),
                         JET_METHOD(accept_commit_launches), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module_def = {PyModuleDef_HEAD_INIT, "_jetcall", "argument marshalling of libjet.so", -1, methods,
                          nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__jetcall() {
  PyObject* m = PyModule_Create(&module_def);
  if (m && PyModule_AddStringConstant(m, "torch_version", JET_TORCH_VERSION) != 0) Py_CLEAR(m);
  return m;
}
