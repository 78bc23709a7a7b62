// _calls: the step's entry points for Python, taking torch tensors.  Argument marshalling only, in native code because
// a step is many small calls: through ctypes the four calls of a one-layer step kept the host busy for 61 us, now for
// 17 us (an attention call 24 -> 5.6 us); turning tensors into pointers and finding the current stream was most of it.
// Each function returns the library's status code.
//
// The checks are those a C caller makes itself: tensors are dense (for the *_layers calls within a layer), of the
// expected rank, and layer strides of K and V agree.  A violation raises AssertionError or ValueError.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "treeverify.h"

namespace {

struct Failed {};      // a Python error is set

[[noreturn]] void raise(PyObject* type, const char* what) {
  PyErr_SetString(type, what);
  throw Failed();
}

struct Args {
  PyObject* const* a;
  Py_ssize_t n;
  Args(PyObject* const* a_, Py_ssize_t n_, Py_ssize_t want) : a(a_), n(n_) {
    if (n != want) raise(PyExc_TypeError, "treeverify: wrong number of arguments");
  }
  bool none(int i) const { return a[i] == Py_None; }
  const at::Tensor& tensor(int i) const {
    if (!THPVariable_Check(a[i])) raise(PyExc_TypeError, "treeverify takes torch tensors");
    return THPVariable_Unpack(a[i]);
  }
  const at::Tensor& tensor(int i, int rank) const {
    const at::Tensor& t = tensor(i);
    if (t.dim() != rank) raise(PyExc_ValueError, "treeverify: a tensor has the wrong number of dimensions");
    return t;
  }
  // Device (or host) address of a dense tensor, of a plain integer, or NULL for None.
  template <typename T = void>
  T* ptr(int i) const {
    if (none(i)) return nullptr;
    if (PyLong_Check(a[i])) {
      void* p = PyLong_AsVoidPtr(a[i]);
      if (!p && PyErr_Occurred()) throw Failed();
      return static_cast<T*>(p);
    }
    const at::Tensor& t = tensor(i);
    if (!t.is_contiguous()) raise(PyExc_AssertionError, "treeverify takes dense tensors");
    return static_cast<T*>(t.data_ptr());
  }
  // ... of a tensor [L, ...] whose layers are dense, L of them or (more) at least L.
  template <typename T = void>
  T* layers(int i, int64_t L, bool more = false) const {
    if (none(i)) return nullptr;
    const at::Tensor& t = tensor(i);
    bool dense = t.dim() >= 1 && (more ? t.size(0) >= L : t.size(0) == L);
    int64_t want = 1;
    for (int64_t d = t.dim() - 1; d >= 1 && dense; --d) {
      dense = t.size(d) == 1 || t.stride(d) == want;
      want *= t.size(d);
    }
    if (!dense) raise(PyExc_AssertionError, "treeverify takes dense layers");
    return static_cast<T*>(t.data_ptr());
  }
  int64_t layer_stride(int i) const { return none(i) ? 0 : tensor(i).stride(0); }
  size_t bytes(int i) const { return tensor(i).nbytes(); }
  float number(int i) const {
    const double v = PyFloat_AsDouble(a[i]);
    if (v == -1.0 && PyErr_Occurred()) throw Failed();
    return (float)v;
  }
  int integer(int i) const {
    const long v = PyLong_AsLong(a[i]);
    if (v == -1 && PyErr_Occurred()) throw Failed();
    return (int)v;
  }
  // None: torch's current stream; otherwise an object with a cuda_stream, or the handle itself.
  tv_stream stream(int i) const {
    if (none(i)) return c10::cuda::getCurrentCUDAStream().stream();
    PyObject* h = PyObject_GetAttrString(a[i], "cuda_stream");
    if (!h) {
      PyErr_Clear();
      h = PyNumber_Long(a[i]);
      if (!h) throw Failed();
    }
    void* p = PyLong_AsVoidPtr(h);
    Py_DECREF(h);
    if (!p && PyErr_Occurred()) throw Failed();
    return p;
  }
};

// Runs a library call without the interpreter lock, as a foreign function would.
template <typename F>
PyObject* call(F&& f) {
  int rc;
  Py_BEGIN_ALLOW_THREADS
  rc = f();
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(rc);
}

template <PyObject* (*BODY)(PyObject* const*, Py_ssize_t)>
PyObject* guarded(PyObject*, PyObject* const* a, Py_ssize_t n) {
  try {
    return BODY(a, n);
  } catch (const Failed&) {
    return nullptr;
  } catch (const std::exception& e) {
    PyErr_SetString(PyExc_RuntimeError, e.what());
    return nullptr;
  }
}

// parent, n_nodes, Dcap, Pcap, anc_bits, dense_mask, depth, anc_table, retrieve_indices, n_paths, status, stream
PyObject* build_mask(PyObject* const* a, Py_ssize_t n) {
  Args x(a, n, 12);
  const at::Tensor& parent = x.tensor(0, 2);
  const int B = parent.size(0), N = parent.size(1);
  const auto *p = x.ptr<int32_t>(0), *nn = x.ptr<int32_t>(1);
  const int Dcap = x.integer(2), Pcap = x.integer(3);
  auto* bits = x.ptr<uint32_t>(4);
  auto* dense = x.ptr<uint8_t>(5);
  auto *depth = x.ptr<int32_t>(6), *table = x.ptr<int32_t>(7), *rows = x.ptr<int32_t>(8), *paths = x.ptr<int32_t>(9),
       *st = x.ptr<int32_t>(10);
  const tv_stream s = x.stream(11);
  return call([&] { return tree_build_mask(p, nn, B, N, Dcap, Pcap, bits, dense, depth, table, rows, paths, st, s); });
}

// q, k_cache, v_cache, k_tree, v_tree, prefix_len, n_nodes, anc_bits, scale, out, workspace, status, lse, stream
PyObject* verify_attn(PyObject* const* a, Py_ssize_t n) {
  Args x(a, n, 14);
  const at::Tensor &q = x.tensor(0, 4), &kc = x.tensor(1, 4);
  const int B = q.size(0), N = q.size(1), Hq = q.size(2), d = q.size(3), Hkv = kc.size(1), Scap = kc.size(2);
  const auto *pq = x.ptr<tv_bf16>(0), *pk = x.ptr<tv_bf16>(1), *pv = x.ptr<tv_bf16>(2), *kt = x.ptr<tv_bf16>(3),
             *vt = x.ptr<tv_bf16>(4);
  const auto *S = x.ptr<int32_t>(5), *nn = x.ptr<int32_t>(6);
  const auto* bits = x.ptr<uint32_t>(7);
  const float scale = x.number(8);
  auto* out = x.ptr<tv_bf16>(9);
  void* ws = x.ptr(10);
  const size_t wsb = x.bytes(10);
  auto* st = x.ptr<int32_t>(11);
  auto* lse = x.ptr<float>(12);
  const tv_stream s = x.stream(13);
  return call([&] {
    return tree_verify_attn(pq, pk, pv, kt, vt, S, nn, bits, B, N, Hq, Hkv, d, Scap, scale, out, lse, ws, wsb, st, s);
  });
}

// ... with flags in front of the stream
PyObject* verify_attn_layers(PyObject* const* a, Py_ssize_t n) {
  Args x(a, n, 15);
  const at::Tensor &q = x.tensor(0, 5), &kc = x.tensor(1, 5);
  const int L = q.size(0), B = q.size(1), N = q.size(2), Hq = q.size(3), d = q.size(4), Hkv = kc.size(2), Scap = kc.size(3);
  const auto *pq = x.layers<tv_bf16>(0, L), *pk = x.layers<tv_bf16>(1, L), *pv = x.layers<tv_bf16>(2, L),
             *kt = x.layers<tv_bf16>(3, L), *vt = x.layers<tv_bf16>(4, L);
  if (x.layer_stride(1) != x.layer_stride(2) || (kt && vt && x.layer_stride(3) != x.layer_stride(4)))
    raise(PyExc_AssertionError, "treeverify: K and V need the same layer stride");
  const auto *S = x.ptr<int32_t>(5), *nn = x.ptr<int32_t>(6);
  const auto* bits = x.ptr<uint32_t>(7);
  const float scale = x.number(8);
  auto* out = x.layers<tv_bf16>(9, L);
  void* ws = x.ptr(10);
  const size_t wsb = x.bytes(10);
  auto* st = x.ptr<int32_t>(11);
  x.layers(12, L);
  auto* lse = x.ptr<float>(12);
  const unsigned flags = (unsigned)x.integer(13);
  const tv_stream s = x.stream(14);
  const int64_t ql = x.layer_stride(0), cl = x.layer_stride(1), tl = x.layer_stride(3), ol = x.layer_stride(9);
  return call([&] {
    return tree_verify_attn_layers(pq, pk, pv, kt, vt, S, nn, bits, L, B, N, Hq, Hkv, d, Scap, scale, ql, cl, tl, out, ol, lse,
                                   ws, wsb, st, flags, s);
  });
}

// q, k_pages, v_pages, block_table, k_tree, v_tree, prefix_len, n_nodes, anc_bits, scale, out, workspace, status, lse, stream
PyObject* verify_attn_paged(PyObject* const* a, Py_ssize_t n) {
  Args x(a, n, 15);
  const at::Tensor &q = x.tensor(0, 4), &kp = x.tensor(1, 4), &table = x.tensor(3, 2);
  const int B = q.size(0), N = q.size(1), Hq = q.size(2), d = q.size(3), pages = kp.size(0), Hkv = kp.size(1);
  if (kp.size(2) != 128 || table.size(0) != B) raise(PyExc_AssertionError, "treeverify: pages of 128 rows, one table row per sequence");
  const int blocks = table.size(1);
  const auto *pq = x.ptr<tv_bf16>(0), *pk = x.ptr<tv_bf16>(1), *pv = x.ptr<tv_bf16>(2);
  const auto* bt = x.ptr<int32_t>(3);
  const auto *kt = x.ptr<tv_bf16>(4), *vt = x.ptr<tv_bf16>(5);
  const auto *S = x.ptr<int32_t>(6), *nn = x.ptr<int32_t>(7);
  const auto* bits = x.ptr<uint32_t>(8);
  const float scale = x.number(9);
  auto* out = x.ptr<tv_bf16>(10);
  void* ws = x.ptr(11);
  const size_t wsb = x.bytes(11);
  auto* st = x.ptr<int32_t>(12);
  auto* lse = x.ptr<float>(13);
  const tv_stream s = x.stream(14);
  return call([&] {
    return tree_verify_attn_paged(pq, pk, pv, bt, kt, vt, S, nn, bits, B, N, Hq, Hkv, d, pages, blocks, scale, out, lse, ws, wsb,
                                  st, s);
  });
}

// ... with flags in front of the stream
PyObject* verify_attn_paged_layers(PyObject* const* a, Py_ssize_t n) {
  Args x(a, n, 16);
  const at::Tensor &q = x.tensor(0, 5), &kp = x.tensor(1, 5), &table = x.tensor(3, 2);
  const int L = q.size(0), B = q.size(1), N = q.size(2), Hq = q.size(3), d = q.size(4), pages = kp.size(1), Hkv = kp.size(2),
            blocks = table.size(1);
  // the first L layers of pools, trees and outputs that may have more
  const auto *pq = x.layers<tv_bf16>(0, L), *pk = x.layers<tv_bf16>(1, L, true), *pv = x.layers<tv_bf16>(2, L, true);
  const auto* bt = x.ptr<int32_t>(3);
  const auto *kt = x.layers<tv_bf16>(4, L, true), *vt = x.layers<tv_bf16>(5, L, true);
  if (L > 1 && (x.layer_stride(1) != x.layer_stride(2) || x.layer_stride(4) != x.layer_stride(5)))
    raise(PyExc_AssertionError, "treeverify: K and V need the same layer stride");
  const auto *S = x.ptr<int32_t>(6), *nn = x.ptr<int32_t>(7);
  const auto* bits = x.ptr<uint32_t>(8);
  const float scale = x.number(9);
  auto* out = x.layers<tv_bf16>(10, L, true);
  void* ws = x.ptr(11);
  const size_t wsb = x.bytes(11);
  auto* st = x.ptr<int32_t>(12);
  x.layers(13, L, true);
  auto* lse = x.ptr<float>(13);
  const unsigned flags = (unsigned)x.integer(14);
  const tv_stream s = x.stream(15);
  const int64_t ql = x.layer_stride(0), cl = x.layer_stride(1), tl = x.layer_stride(4), ol = x.layer_stride(10);
  return call([&] {
    return tree_verify_attn_paged_layers(pq, pk, pv, bt, kt, vt, S, nn, bits, L, B, N, Hq, Hkv, d, pages, blocks, scale, ql, cl,
                                         tl, out, ol, lse, ws, wsb, st, flags, s);
  });
}

// logits, tokens, retrieve_indices, n_nodes, argmax_tok, safe_idx, candidates, accept_len, best_path, accepted_nodes,
// next_token, workspace, status, behind_attn, stream
PyObject* accept(PyObject* const* a, Py_ssize_t n) {
  Args x(a, n, 15);
  const at::Tensor &lg = x.tensor(0, 3), &r = x.tensor(2, 3);
  const int B = lg.size(0), N = lg.size(1), V = lg.size(2), P = r.size(1), Dp1 = r.size(2);
  const auto* logits = x.ptr<tv_bf16>(0);
  const auto *tok = x.ptr<int32_t>(1), *rows = P > 0 ? x.ptr<int32_t>(2) : nullptr, *nn = x.ptr<int32_t>(3);
  auto *am = x.ptr<int32_t>(4), *safe = x.ptr<int32_t>(5), *cand = x.ptr<int32_t>(6), *al = x.ptr<int32_t>(7),
       *best = x.ptr<int32_t>(8), *nodes = x.ptr<int32_t>(9), *next = x.ptr<int32_t>(10);
  void* ws = x.ptr(11);
  const size_t wsb = x.bytes(11);
  auto* st = x.ptr<int32_t>(12);
  const auto entry = x.integer(13) ? tree_accept_behind_attn : tree_accept;
  const tv_stream s = x.stream(14);
  return call([&] {
    return entry(logits, tok, rows, nn, B, N, V, P, Dp1, am, safe, cand, al, best, nodes, next, ws, wsb, st, s);
  });
}

// logits, tokens, parent, n_nodes, u_node, u_bonus, temperature, accept_len, accepted_nodes, next_token, workspace, status, stream
PyObject* accept_sample(PyObject* const* a, Py_ssize_t n) {
  Args x(a, n, 13);
  const at::Tensor &lg = x.tensor(0, 3), &acc = x.tensor(8, 2);
  const int B = lg.size(0), N = lg.size(1), V = lg.size(2), Dp1 = acc.size(1);
  const auto* logits = x.ptr<tv_bf16>(0);
  const auto *tok = x.ptr<int32_t>(1), *par = x.ptr<int32_t>(2), *nn = x.ptr<int32_t>(3);
  const auto *un = x.ptr<float>(4), *ub = x.ptr<float>(5);
  const float T = x.number(6);
  auto *al = x.ptr<int32_t>(7), *nodes = x.ptr<int32_t>(8), *next = x.ptr<int32_t>(9);
  void* ws = x.ptr(10);
  const size_t wsb = x.bytes(10);
  auto* st = x.ptr<int32_t>(11);
  const tv_stream s = x.stream(12);
  return call([&] { return tree_accept_sample(logits, tok, par, nn, un, ub, T, B, N, V, Dp1, al, nodes, next, ws, wsb, st, s); });
}

// o_parts, lse_parts, out, lse, stream
PyObject* merge_partials(PyObject* const* a, Py_ssize_t n) {
  Args x(a, n, 5);
  const at::Tensor& o = x.tensor(0, 5);
  const int R = o.size(0), B = o.size(1), N = o.size(2), Hq = o.size(3), d = o.size(4);
  const auto* op = x.ptr<tv_bf16>(0);
  const auto* lp = x.ptr<float>(1);
  auto* out = x.ptr<tv_bf16>(2);
  auto* lse = x.ptr<float>(3);
  const tv_stream s = x.stream(4);
  return call([&] { return tree_merge_partials(op, lp, R, B, N, Hq, d, out, lse, s); });
}

// k_cache, v_cache, k_tree, v_tree, accepted_nodes, accept_len, prefix_len, status, stream
PyObject* commit(PyObject* const* a, Py_ssize_t n) {
  Args x(a, n, 9);
  const at::Tensor &kc = x.tensor(0, 5), &kt = x.tensor(2, 5), &acc = x.tensor(4, 2);
  const int L = kc.size(0), B = kc.size(1), Hkv = kc.size(2), Scap = kc.size(3), d = kc.size(4), N = kt.size(2), Dp1 = acc.size(1);
  auto *pk = x.ptr<tv_bf16>(0), *pv = x.ptr<tv_bf16>(1);
  const auto *tk = x.ptr<tv_bf16>(2), *tvp = x.ptr<tv_bf16>(3);
  const auto *nodes = x.ptr<int32_t>(4), *al = x.ptr<int32_t>(5);
  auto *S = x.ptr<int32_t>(6), *st = x.ptr<int32_t>(7);
  const tv_stream s = x.stream(8);
  const int64_t cl = kc.stride(0), tl = kt.stride(0);
  return call([&] { return kv_commit(pk, pv, tk, tvp, nodes, al, S, L, B, N, Hkv, d, Scap, Dp1, cl, tl, st, s); });
}

// k_pages, v_pages, block_table, k_tree, v_tree, accepted_nodes, accept_len, prefix_len, status, stream
PyObject* commit_paged(PyObject* const* a, Py_ssize_t n) {
  Args x(a, n, 10);
  const at::Tensor &kp = x.tensor(0, 5), &table = x.tensor(2, 2), &kt = x.tensor(3, 5), &acc = x.tensor(5, 2);
  const int L = kp.size(0), pages = kp.size(1), Hkv = kp.size(2), d = kp.size(4), blocks = table.size(1), B = kt.size(1),
            N = kt.size(2), Dp1 = acc.size(1);
  auto *pk = x.ptr<tv_bf16>(0), *pv = x.ptr<tv_bf16>(1);
  const auto* bt = x.ptr<int32_t>(2);
  const auto *tk = x.ptr<tv_bf16>(3), *tvp = x.ptr<tv_bf16>(4);
  const auto *nodes = x.ptr<int32_t>(5), *al = x.ptr<int32_t>(6);
  auto *S = x.ptr<int32_t>(7), *st = x.ptr<int32_t>(8);
  const tv_stream s = x.stream(9);
  const int64_t cl = kp.stride(0), tl = kt.stride(0);
  return call([&] { return kv_commit_paged(pk, pv, bt, tk, tvp, nodes, al, S, L, B, N, Hkv, d, pages, blocks, Dp1, cl, tl, st, s); });
}

// k_cache, v_cache, accepted_nodes, accept_len, prefix_len, Nmax, status, stream
PyObject* commit_inplace(PyObject* const* a, Py_ssize_t n) {
  Args x(a, n, 8);
  const at::Tensor &kc = x.tensor(0, 5), &acc = x.tensor(2, 2);
  const int L = kc.size(0), B = kc.size(1), Hkv = kc.size(2), Scap = kc.size(3), d = kc.size(4), Dp1 = acc.size(1);
  auto *pk = x.ptr<tv_bf16>(0), *pv = x.ptr<tv_bf16>(1);
  const auto *nodes = x.ptr<int32_t>(2), *al = x.ptr<int32_t>(3);
  auto* S = x.ptr<int32_t>(4);
  const int N = x.integer(5);
  auto* st = x.ptr<int32_t>(6);
  const tv_stream s = x.stream(7);
  const int64_t cl = kc.stride(0);
  return call([&] { return kv_commit_inplace(pk, pv, nodes, al, S, L, B, N, Hkv, d, Scap, Dp1, cl, st, s); });
}

// host (dict of pinned tensors), k_cache, v_cache, prefix_len, staging, scale, V, stream
PyObject* step_host(PyObject* const* a, Py_ssize_t n) {
  Args x(a, n, 8);
  if (!PyDict_Check(a[0])) raise(PyExc_TypeError, "treeverify: the host buffers are a dict of tensors");
  static const char* const names[] = {"parent", "n_nodes", "tokens", "retrieve_indices", "q", "k_tree", "v_tree", "logits", "out",
                                      "accept_len", "accepted_nodes", "next_token", "status", "P"};
  PyObject* h[14];
  for (int i = 0; i < 14; ++i) {
    h[i] = PyDict_GetItemString(a[0], names[i]);
    if (!h[i]) {
      if (i != 3 && i != 13) raise(PyExc_KeyError, names[i]);
      h[i] = Py_None;
    }
  }
  Args y(h, 14, 14);
  const at::Tensor &q = y.tensor(4, 5), &kc = x.tensor(1, 5), &acc = y.tensor(10, 2);
  tv_step_host_args s{};
  s.parent = y.ptr<int32_t>(0);
  s.n_nodes = y.ptr<int32_t>(1);
  s.tokens = y.ptr<int32_t>(2);
  s.retrieve_indices = y.ptr<int32_t>(3);
  s.q = y.ptr<tv_bf16>(4);
  s.k_tree = y.ptr<tv_bf16>(5);
  s.v_tree = y.ptr<tv_bf16>(6);
  s.logits = y.ptr<tv_bf16>(7);
  s.out = y.ptr<tv_bf16>(8);
  s.accept_len = y.ptr<int32_t>(9);
  s.accepted_nodes = y.ptr<int32_t>(10);
  s.next_token = y.ptr<int32_t>(11);
  s.status = y.ptr<int32_t>(12);
  s.k_cache = x.ptr<tv_bf16>(1);
  s.v_cache = x.ptr<tv_bf16>(2);
  s.prefix_len = x.ptr<int32_t>(3);
  s.staging = x.ptr(4);
  s.staging_bytes = x.bytes(4);
  s.L = q.size(0);
  s.B = q.size(1);
  s.Nmax = q.size(2);
  s.Hq = q.size(3);
  s.d = q.size(4);
  s.Hkv = kc.size(2);
  s.Scap = kc.size(3);
  s.V = x.integer(6);
  s.P = y.none(3) ? y.integer(13) : (int)y.tensor(3, 3).size(1);
  s.Dp1 = acc.size(1);
  s.scale = x.number(5);
  s.stream = x.stream(7);
  return call([&] { return tv_verify_step_host(&s); });
}

#define TV_METHOD(name, body) {name, reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(&guarded<body>)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {
    TV_METHOD("tree_build_mask", build_mask),
    TV_METHOD("tree_verify_attn", verify_attn),
    TV_METHOD("tree_verify_attn_layers", verify_attn_layers),
    TV_METHOD("tree_verify_attn_paged", verify_attn_paged),
    TV_METHOD("tree_verify_attn_paged_layers", verify_attn_paged_layers),
    TV_METHOD("tree_accept", accept),
    TV_METHOD("tree_accept_sample", accept_sample),
    TV_METHOD("tree_merge_partials", merge_partials),
    TV_METHOD("kv_commit", commit),
    TV_METHOD("kv_commit_paged", commit_paged),
    TV_METHOD("kv_commit_inplace", commit_inplace),
    TV_METHOD("tv_verify_step_host", step_host),
    {nullptr, nullptr, 0, nullptr}};

PyModuleDef module = {PyModuleDef_HEAD_INIT, "_calls", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__calls() { return PyModule_Create(&module); }
