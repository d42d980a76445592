// Native half of the Python binding: torch tensors in, calls of the C ABI (include/mixkv.h), torch
// tensors out.  Argument marshalling only, as in binding.py, which wraps every function of this module
// and documents it.
//
// Why it is native: a call of the library enqueues two to six kernels, and the smallest calls keep the
// GPU busy for less time than interpreted marshalling takes.  Through ctypes one decode call cost 15 us of
// host time for 7 us of GPU time and a scores + select pair 89 us; here they cost 3.2 and 18 us, one
// layer's compression 7.4 us, a similarity map 7.1 us.  Output tensors come from torch's caching allocator without the dispatcher.
//
// The interpreter lock is given up around everything that can block (Unlocked, below): a launch waits while the
// stream's queue is full, an allocation may wait for the device, and a host callback on that stream, or any
// other thread of the program, may need the interpreter before either goes on.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/ATen.h>
#include <ATen/cuda/EmptyTensor.h>
#include <c10/cuda/CUDAFunctions.h>
#include <c10/cuda/CUDAGuard.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <dlfcn.h>

#include <optional>
#include <vector>

#include "../internal_api.h"
#include "mixkv.h"

// What this module was compiled against (build.py looks for the string in the file).
extern "C" __attribute__((used)) const char mixkv_host_tag[] = MIXKV_HOST_TAG;

namespace {

// ---- the library and what comes from Python at start-up
struct Api {
  decltype(&mixkv_internal_scores) scores;
  decltype(&mixkv_internal_select) select;
  decltype(&mixkv_compress_layer_traced) layer;
  decltype(&mixkv_compress_layers) layers;
  decltype(&mixkv_compress_layers_budgeted) budgeted;
  decltype(&mixkv_workspace_size_layers) ws_size;
  decltype(&mixkv_similarity_workspace_size) sim_ws_size;
  decltype(&mixkv_similarity_map) sim_map;
  decltype(&mixkv_decode_attention) decode;
} api;
PyObject* g_error = nullptr;   // binding.MixKVError

// Interned names, created once.
struct Names {
  PyObject *kv_heads, *gqa_ratio, *head_dim, *window, *pool_kernel, *pool_mode, *use_vnorm, *mix_mode,
      *budget_mode, *budget, *ada_floor, *eps, *softmax_scale, *cuda_stream;
  PyObject *s_comp, *s_ex, *s_div, *rbar, *status, *idx, *counts, *idx_offsets, *K_out, *V_out,
      *out_row_offsets;
} nm;

// A Python exception is set; unwinds to the entry point.
struct Raised {};

// No interpreter lock in this scope.
struct Unlocked {
  PyThreadState* state = PyEval_SaveThread();
  ~Unlocked() { PyEval_RestoreThread(state); }
};

[[noreturn]] void fail(PyObject* type, const char* what) {
  PyErr_SetString(type, what);
  throw Raised();
}
void check_status(const int rc, const char* what) {
  if (rc == MIXKV_OK) return;
  PyObject* e = PyObject_CallFunction(g_error, "is", rc, what);
  if (e) {
    PyErr_SetObject(g_error, e);
    Py_DECREF(e);
  }
  throw Raised();
}

const at::Tensor& tensor(PyObject* o) {
  if (!THPVariable_Check(o)) fail(PyExc_TypeError, "a tensor is expected");
  return THPVariable_Unpack(o);
}
void want_contiguous(const at::Tensor& t) {
  if (!t.is_contiguous()) fail(PyExc_AssertionError, "tensors handed to the library must be contiguous");
}
template <typename T = void>
T* ptr(PyObject* o) {   // None -> nullptr
  if (o == nullptr || o == Py_None) return nullptr;
  const at::Tensor& t = tensor(o);
  want_contiguous(t);
  return static_cast<T*>(t.data_ptr());
}
template <typename T = void>
T* item(PyObject* dict, PyObject* key, const bool required) {   // entry of an output dict
  PyObject* o = PyDict_GetItemWithError(dict, key);
  if (!o) {
    if (PyErr_Occurred()) throw Raised();
    if (required) {
      PyErr_SetObject(PyExc_KeyError, key);
      throw Raised();
    }
    return nullptr;
  }
  return ptr<T>(o);
}

bool truth(PyObject* o) {
  const int t = PyObject_IsTrue(o);
  if (t < 0) throw Raised();
  return t != 0;
}
// The library takes 32 bits: of a larger number it would see the lower ones, another problem than the caller's.
int32_t int32(const long x, const char* what) {
  if (x != (int32_t)x) check_status(MIXKV_ERR_INVALID_ARG, what);
  return (int32_t)x;
}
int32_t int32(PyObject* o, const char* what) {
  const long x = PyLong_AsLong(o);
  if (x == -1 && PyErr_Occurred()) throw Raised();
  return int32(x, what);
}
int32_t attr_int(PyObject* o, PyObject* name) {
  PyObject* v = PyObject_GetAttr(o, name);
  if (!v) throw Raised();
  const long x = PyLong_AsLong(v);
  Py_DECREF(v);
  if (x == -1 && PyErr_Occurred()) throw Raised();
  return int32(x, "mixkv_params");
}
float attr_float(PyObject* o, PyObject* name) {
  PyObject* v = PyObject_GetAttr(o, name);
  if (!v) throw Raised();
  const double x = PyFloat_AsDouble(v);
  Py_DECREF(v);
  if (x == -1.0 && PyErr_Occurred()) throw Raised();
  return (float)x;
}
mixkv_params params(PyObject* o) {
  mixkv_params p;
  p.kv_heads = attr_int(o, nm.kv_heads);
  p.gqa_ratio = attr_int(o, nm.gqa_ratio);
  p.head_dim = attr_int(o, nm.head_dim);
  p.window = attr_int(o, nm.window);
  p.pool_kernel = attr_int(o, nm.pool_kernel);
  p.pool_mode = attr_int(o, nm.pool_mode);
  p.use_vnorm = attr_int(o, nm.use_vnorm);
  p.mix_mode = attr_int(o, nm.mix_mode);
  p.budget_mode = attr_int(o, nm.budget_mode);
  p.budget = attr_int(o, nm.budget);
  p.ada_floor = attr_float(o, nm.ada_floor);
  p.eps = attr_float(o, nm.eps);
  p.softmax_scale = attr_float(o, nm.softmax_scale);
  return p;
}

// Sequence offsets (None: one sequence).
struct Offsets {
  std::vector<int32_t> v;
  int batch = 1;
  explicit Offsets(PyObject* o) {
    if (o == Py_None) return;
    PyObject* seq = PySequence_Fast(o, "cu_seqlens must be a sequence");
    if (!seq) throw Raised();
    const Py_ssize_t n = PySequence_Fast_GET_SIZE(seq);
    v.reserve((size_t)n);
    for (Py_ssize_t i = 0; i < n; ++i) {
      long x = PyLong_AsLong(PySequence_Fast_GET_ITEM(seq, i));
      if (x == -1 && PyErr_Occurred()) {   // e.g. a tensor element or a numpy integer
        PyErr_Clear();
        PyObject* as_int = PyNumber_Long(PySequence_Fast_GET_ITEM(seq, i));
        if (as_int) {
          x = PyLong_AsLong(as_int);
          Py_DECREF(as_int);
        }
        if (PyErr_Occurred()) {
          Py_DECREF(seq);
          throw Raised();
        }
      }
      if (x != (int32_t)x) {
        Py_DECREF(seq);
        check_status(MIXKV_ERR_INVALID_ARG, "cu_seqlens");
      }
      v.push_back((int32_t)x);
    }
    Py_DECREF(seq);
    batch = (int)n - 1;
  }
  const int32_t* data() const { return v.empty() ? nullptr : v.data(); }
  int len(int b, int Ltot) const { return v.empty() ? Ltot : v[(size_t)b + 1] - v[(size_t)b]; }
  int max_len(int Ltot) const {   // (0 where there is no sequence: the library refuses that)
    int m = 0;
    for (int b = 0; b < batch; ++b) m = std::max(m, len(b, Ltot));
    return m;
  }
};

// The stream of a call: the one it is given, else the current one.  While this lives it is the current one, so that what
// the call allocates, fills and gives back (a workspace of its own is free again when the call returns, long before the
// GPU is done with it) is ordered on the stream its kernels run on.
struct CallStream {
  void* handle;
  std::optional<c10::cuda::CUDAStreamGuard> guard;
  CallStream(PyObject* o, const at::Tensor& like) {
    if (o == Py_None) {
      handle = (void*)c10::cuda::getCurrentCUDAStream().stream();
      return;
    }
    PyObject* v = PyObject_GetAttr(o, nm.cuda_stream);
    if (!v) throw Raised();
    handle = PyLong_AsVoidPtr(v);
    Py_DECREF(v);
    if (!handle && PyErr_Occurred()) throw Raised();
    if (!like.is_cuda()) return;
    const c10::DeviceIndex device = c10::cuda::current_device();
    if (handle != (void*)c10::cuda::getCurrentCUDAStream(device).stream())
      guard.emplace(c10::cuda::getStreamFromExternal((cudaStream_t)handle, device));
  }
};

// (called without the interpreter lock)
at::Tensor empty(at::IntArrayRef size, at::ScalarType type, const at::Tensor& like) {
  return at::Tensor(at::detail::empty_cuda(size, type, like.device(), std::nullopt));
}
int32_t* ip(const at::Tensor& t) { return static_cast<int32_t*>(t.data_ptr()); }
float* fp(const at::Tensor& t) { return static_cast<float*>(t.data_ptr()); }

void put(PyObject* dict, PyObject* key, const at::Tensor& t) {
  PyObject* o = THPVariable_Wrap(t);
  if (!o) throw Raised();
  const int rc = PyDict_SetItem(dict, key, o);
  Py_DECREF(o);
  if (rc != 0) throw Raised();
}

// The caller's workspace, or one of the size the call needs (kept alive by `own`).
struct Space {
  at::Tensor own;
  void* data;
  size_t bytes;
  Space(PyObject* o, const mixkv_params& p, int layers, const Offsets& cu, int Ltot, const at::Tensor& like) {
    if (o == Py_None) {
      size_t need = 0;
      check_status(api.ws_size(&p, layers, cu.batch, Ltot, cu.max_len(Ltot), &need), "mixkv_workspace_size");
      const Unlocked u;
      own = empty({(int64_t)need}, at::kByte, like);
      data = own.data_ptr();
      bytes = need;
    } else {
      const at::Tensor& t = tensor(o);
      want_contiguous(t);
      data = t.data_ptr();
      bytes = (size_t)t.numel();
    }
  }
};

void want_dims(const at::Tensor& t, int64_t n, const char* what) {
  if (t.dim() != n) fail(PyExc_ValueError, what);
}

template <typename F>
PyObject* guarded(Py_ssize_t n, Py_ssize_t want, F&& body) {
  if (n != want) {
    PyErr_SetString(PyExc_TypeError, "wrong number of arguments");
    return nullptr;
  }
  try {
    return body();
  } catch (const Raised&) {
    return nullptr;
  } catch (const c10::OutOfMemoryError& e) {
    PyObject* torch = PyImport_ImportModule("torch");
    PyObject* type = torch ? PyObject_GetAttrString(torch, "OutOfMemoryError") : nullptr;
    PyErr_SetString(type ? type : PyExc_MemoryError, e.what_without_backtrace());
    Py_XDECREF(type);
    Py_XDECREF(torch);
    return nullptr;
  } catch (const std::exception& e) {
    PyErr_SetString(PyExc_RuntimeError, e.what());
    return nullptr;
  }
}

// A dict under construction, released unless handed over.
struct Dict {
  PyObject* d = PyDict_New();
  Dict() {
    if (!d) throw Raised();
  }
  ~Dict() { Py_XDECREF(d); }
  PyObject* release() {
    PyObject* r = d;
    d = nullptr;
    return r;
  }
};

// scores(K, V, Q, params, cu, rbar_in, workspace, stream, want_parts, fixed_scratch)
PyObject* py_scores(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded(n, 10, [&]() -> PyObject* {
    const at::Tensor& K = tensor(a[0]);
    want_dims(K, 3, "K must have three dimensions [H, Ltot, d]");
    const mixkv_params p = params(a[3]);
    const Offsets cu(a[4]);
    const bool parts = truth(a[8]), fixed = truth(a[9]);
    const int64_t H = K.size(0), Ltot = K.size(1), Ptot = Ltot - (int64_t)cu.batch * p.window;
    const CallStream stream(a[7], K);
    std::optional<Space> ws;
    if (!fixed) ws.emplace(a[6], p, 1, cu, (int)Ltot, K);
    if (Ptot < 0) check_status(MIXKV_ERR_INVALID_ARG, fixed ? "mixkv_scores_static" : "mixkv_scores");
    at::Tensor s_comp, s_ex, s_div, rbar, status;
    void *k = ptr(a[0]), *v = ptr(a[1]), *q = ptr(a[2]);
    const float* rin = ptr<float>(a[5]);
    int rc;
    {
      const Unlocked u;
      s_comp = empty({H, Ptot}, at::kFloat, K);
      if (parts) {
        s_ex = empty({H, Ptot}, at::kFloat, K);
        s_div = empty({H, Ptot}, at::kFloat, K);
        rbar = empty({cu.batch, H}, at::kFloat, K);
      }
      status = empty({1}, at::kInt, K);
      rc = api.scores(k, v, q, cu.data(), cu.batch, (int)Ltot, &p, fixed ? 1 : 0, fixed ? nullptr : ws->data,
                      fixed ? 0 : ws->bytes, fp(s_comp), parts ? fp(s_ex) : nullptr, parts ? fp(s_div) : nullptr,
                      parts ? fp(rbar) : nullptr, rin, ip(status), stream.handle);
    }
    check_status(rc, fixed ? "mixkv_scores_static" : "mixkv_scores");
    Dict out;
    put(out.d, nm.s_comp, s_comp);
    if (parts) {
      put(out.d, nm.s_ex, s_ex);
      put(out.d, nm.s_div, s_div);
      put(out.d, nm.rbar, rbar);
    }
    put(out.d, nm.status, status);
    return out.release();
  });
}

// select(s, params, cu, workspace, stream)
PyObject* py_select(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded(n, 5, [&]() -> PyObject* {
    const at::Tensor& s = tensor(a[0]);
    want_dims(s, 2, "scores must have two dimensions [H, Ptot]");
    const mixkv_params p = params(a[1]);
    const Offsets cu(a[2]);
    const int64_t H = s.size(0), Ltot = s.size(1) + (int64_t)cu.batch * p.window, BH = cu.batch * H;
    const CallStream stream(a[4], s);
    const Space ws(a[3], p, 1, cu, (int)Ltot, s);
    const int64_t cap = std::max<int64_t>(BH * (p.budget - p.window), 1);
    const float* scores = ptr<const float>(a[0]);
    at::Tensor idx, counts, offs, status;
    int rc;
    {
      const Unlocked u;
      idx = empty({cap}, at::kInt, s);
      counts = empty({BH}, at::kInt, s);
      offs = empty({BH + 1}, at::kInt, s);
      status = empty({1}, at::kInt, s);
      rc = api.select(scores, cu.data(), cu.batch, (int)Ltot, &p, ws.data, ws.bytes, ip(idx), ip(counts), ip(offs),
                      ip(status), stream.handle);
    }
    check_status(rc, "mixkv_select");
    Dict out;
    put(out.d, nm.idx, idx);
    put(out.d, nm.counts, counts);
    put(out.d, nm.idx_offsets, offs);
    put(out.d, nm.status, status);
    return out.release();
  });
}

// Outputs of a compression call: the caller's dict, or a new one.  `lead` is the layer dimension (-1: the
// one-layer call, whose tensors have none).
PyObject* compress_outputs(PyObject* given, PyObject* aux, const int64_t lead, const int64_t rows,
                           const int64_t cap, const int64_t BH, const int64_t H, const int64_t Ptot,
                           const at::Tensor& K) {
  if (given != Py_None) {
    if (!PyDict_Check(given)) fail(PyExc_TypeError, "out must be a dict of tensors");
    Py_INCREF(given);
    return given;
  }
  const bool with_aux = truth(aux);
  struct {
    PyObject* key;
    at::ScalarType type;
    std::vector<int64_t> size;
    at::Tensor t;
  } outputs[] = {{nm.K_out, at::kBFloat16, {rows, K.size(-1)}, {}},
                 {nm.V_out, at::kBFloat16, {rows, K.size(-1)}, {}},
                 {nm.out_row_offsets, at::kInt, {BH + 1}, {}},
                 {nm.idx, at::kInt, {cap}, {}},
                 {nm.counts, at::kInt, {BH}, {}},
                 {nm.idx_offsets, at::kInt, {BH + 1}, {}},
                 {nm.s_comp, at::kFloat, {H, Ptot}, {}}};
  const int n = with_aux ? 7 : 3;
  at::Tensor status;
  {
    const Unlocked u;
    for (int i = 0; i < n; ++i) {
      if (lead >= 0) outputs[i].size.insert(outputs[i].size.begin(), lead);
      outputs[i].t = empty(outputs[i].size, outputs[i].type, K);
    }
    status = at::zeros({1}, K.options().dtype(at::kInt));   // (enqueues a fill)
  }
  Dict out;
  for (int i = 0; i < n; ++i) put(out.d, outputs[i].key, outputs[i].t);
  put(out.d, nm.status, status);
  return out.release();
}
struct Ref {   // an owned reference
  PyObject* o;
  explicit Ref(PyObject* x) : o(x) {}
  ~Ref() { Py_XDECREF(o); }
  PyObject* release() {
    PyObject* r = o;
    o = nullptr;
    return r;
  }
};
struct OutPtrs {
  void *K, *V;
  int32_t *row_offsets, *idx, *counts, *idx_offsets, *status;
  float* s_comp;
  explicit OutPtrs(PyObject* d) {
    K = item(d, nm.K_out, true);
    V = item(d, nm.V_out, true);
    row_offsets = item<int32_t>(d, nm.out_row_offsets, true);
    idx = item<int32_t>(d, nm.idx, false);
    counts = item<int32_t>(d, nm.counts, false);
    idx_offsets = item<int32_t>(d, nm.idx_offsets, false);
    s_comp = item<float>(d, nm.s_comp, false);
    status = item<int32_t>(d, nm.status, true);
  }
};

// compress_layer(K, V, Q, params, cu, rbar_in, workspace, stream, out, want_aux, events, n_events)
PyObject* py_compress_layer(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded(n, 12, [&]() -> PyObject* {
    const at::Tensor& K = tensor(a[0]);
    want_dims(K, 3, "K must have three dimensions [H, Ltot, d]");
    const mixkv_params p = params(a[3]);
    const Offsets cu(a[4]);
    const int64_t H = K.size(0), Ltot = K.size(1), BH = cu.batch * H;
    const CallStream stream(a[7], K);
    const Space ws(a[6], p, 1, cu, (int)Ltot, K);
    Ref out(compress_outputs(a[8], a[9], -1, BH * p.budget,
                             std::max<int64_t>(BH * (p.budget - p.window), 1), BH, H,
                             Ltot - (int64_t)cu.batch * p.window, K));
    const OutPtrs o(out.o);
    const long long events = PyLong_AsLongLong(a[10]);
    const long n_events = PyLong_AsLong(a[11]);
    if (PyErr_Occurred()) throw Raised();
    void *k = ptr(a[0]), *v = ptr(a[1]), *q = ptr(a[2]);
    const float* rin = ptr<const float>(a[5]);
    int rc;
    {
      const Unlocked u;
      rc = api.layer(k, v, q, cu.data(), cu.batch, (int)Ltot, &p, ws.data, ws.bytes, rin, o.K, o.V, o.row_offsets,
                     o.idx, o.counts, o.idx_offsets, o.s_comp, o.status, stream.handle,
                     reinterpret_cast<void* const*>(events), (int)n_events);
    }
    check_status(rc, "mixkv_compress_layer");
    return out.release();
  });
}

// Whether everything but the leading (layer) dimension is packed.
void want_layer_contiguous(const at::Tensor& t) {
  int64_t packed = 1;
  for (int64_t i = t.dim() - 1; i >= 1; --i) {
    if (t.size(i) != 1 && t.stride(i) != packed) fail(PyExc_AssertionError, "each layer must be contiguous");
    packed *= t.size(i);
  }
}

// compress_layers(K, V, Q, params, cu, rbar_in, workspace, stream, out, want_aux, events, n_events,
//                 head_budgets)
PyObject* py_compress_layers(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded(n, 13, [&]() -> PyObject* {
    const at::Tensor &K = tensor(a[0]), &V = tensor(a[1]), &Q = tensor(a[2]);
    want_dims(K, 4, "K must have four dimensions [layers, H, Ltot, d]");
    if (V.dim() < 2 || Q.dim() < 2) fail(PyExc_ValueError, "V and Q need a leading layer dimension");
    want_layer_contiguous(K);
    want_layer_contiguous(V);
    want_layer_contiguous(Q);
    if (V.stride(0) != K.stride(0)) fail(PyExc_AssertionError, "K and V must share their layer stride");
    const mixkv_params p = params(a[3]);
    const Offsets cu(a[4]);
    const int64_t NL = K.size(0), H = K.size(1), Ltot = K.size(2), BH = cu.batch * H;
    const CallStream stream(a[7], K);
    const Space ws(a[6], p, (int)NL, cu, (int)Ltot, K);
    int64_t cap = 0;
    for (int b = 0; b < cu.batch; ++b)
      cap += H * std::min<int64_t>(p.budget - p.window, cu.len(b, (int)Ltot) - p.window);
    Ref out(compress_outputs(a[8], a[9], NL, BH * p.budget, std::max<int64_t>(cap, 1), BH,
                             H, Ltot - (int64_t)cu.batch * p.window, K));
    const OutPtrs o(out.o);
    const long long events = PyLong_AsLongLong(a[10]);
    const long n_events = PyLong_AsLong(a[11]);
    if (PyErr_Occurred()) throw Raised();
    const float* rin = ptr<const float>(a[5]);
    const int32_t* budgets = nullptr;
    if (a[12] != Py_None) {
      const at::Tensor& hb = tensor(a[12]);
      want_contiguous(hb);
      if (hb.scalar_type() != at::kInt || hb.dim() != 2 || hb.size(0) != NL || hb.size(1) != BH || n_events)
        fail(PyExc_AssertionError, "head_budgets must be an int32 tensor [layers, batch * H], without events");
      budgets = ip(hb);
    }
    void *k = K.data_ptr(), *v = V.data_ptr(), *q = Q.data_ptr();
    const int64_t kv_stride = K.stride(0), q_stride = Q.stride(0);
    int rc;
    {
      const Unlocked u;
      rc = budgets ? api.budgeted(k, v, q, (int)NL, kv_stride, q_stride, cu.data(), cu.batch, (int)Ltot, &p, ws.data,
                                  ws.bytes, rin, budgets, o.K, o.V, o.row_offsets, o.idx, o.counts, o.idx_offsets,
                                  o.s_comp, o.status, stream.handle)
                   : api.layers(k, v, q, (int)NL, kv_stride, q_stride, cu.data(), cu.batch, (int)Ltot, &p, ws.data,
                                ws.bytes, rin, o.K, o.V, o.row_offsets, o.idx, o.counts, o.idx_offsets, o.s_comp,
                                o.status, stream.handle, reinterpret_cast<void* const*>(events), (int)n_events);
    }
    check_status(rc, budgets ? "mixkv_compress_layers_budgeted" : "mixkv_compress_layers");
    return out.release();
  });
}

// similarity_map(X, block, want_mean, stream) -> (cells, mean or None)
PyObject* py_similarity_map(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded(n, 4, [&]() -> PyObject* {
    const at::Tensor& X = tensor(a[0]);
    want_dims(X, 3, "X must have three dimensions [heads, L, d]");
    if (!X.is_contiguous() || X.scalar_type() != at::kBFloat16)
      fail(PyExc_AssertionError, "X must be a contiguous bf16 tensor");
    const int64_t block = int32(a[1], "mixkv_similarity_map");
    const int heads = (int)X.size(0), L = (int)X.size(1);
    size_t need = 0;
    check_status(api.sim_ws_size(heads, L, (int)block, &need), "mixkv_similarity_workspace_size");
    const int64_t T = (L + block - 1) / block;
    const bool want_mean = truth(a[2]);
    const CallStream stream(a[3], X);
    void* x = X.data_ptr();
    const int d = (int)X.size(2);
    at::Tensor ws, cells, mean;
    int rc;
    {
      const Unlocked u;
      ws = empty({(int64_t)need}, at::kByte, X);
      cells = empty({heads, T, T}, at::kFloat, X);
      if (want_mean) mean = empty({heads}, at::kFloat, X);
      rc = api.sim_map(x, heads, L, d, (int)block, ws.data_ptr(), need, fp(cells), want_mean ? fp(mean) : nullptr,
                       stream.handle);
    }
    check_status(rc, "mixkv_similarity_map");
    Ref c(THPVariable_Wrap(cells)), m(want_mean ? THPVariable_Wrap(mean) : Py_NewRef(Py_None));
    if (!c.o || !m.o) throw Raised();
    return PyTuple_Pack(2, c.o, m.o);
  });
}

// decode_attention(K_cache, V_cache, offsets, q, kv_heads, gqa_ratio, max_rows, softmax_scale, stream)
PyObject* py_decode_attention(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded(n, 9, [&]() -> PyObject* {
    const at::Tensor &K = tensor(a[0]), &V = tensor(a[1]), &offs = tensor(a[2]), &q = tensor(a[3]);
    want_dims(K, 3, "K_cache must have three dimensions [layers, rows, d]");
    if (q.dim() < 2) fail(PyExc_IndexError, "q must have a batch dimension");
    if (!K.is_contiguous() || !V.is_contiguous() || !q.is_contiguous())
      fail(PyExc_AssertionError, "the caches and q must be contiguous");
    if (offs.scalar_type() != at::kInt || !offs.is_contiguous())
      fail(PyExc_AssertionError, "out_row_offsets must be a contiguous int32 tensor");
    const char* what = "mixkv_decode_attention";
    const int32_t H = int32(a[4], what), G = int32(a[5], what), rows = int32(a[6], what);
    const double scale = PyFloat_AsDouble(a[7]);
    if (PyErr_Occurred()) throw Raised();
    const CallStream stream(a[8], K);
    void *k = K.data_ptr(), *v = V.data_ptr(), *query = q.data_ptr();
    const int32_t* offsets = ip(offs);
    const int layers = (int)K.size(0), batch = (int)q.size(1), d = (int)K.size(2);
    const int64_t cap = K.size(1);
    at::Tensor out;
    int rc;
    {
      const Unlocked u;
      out = empty(q.sizes(), at::kFloat, q);
      rc = api.decode(k, v, offsets, cap, query, layers, batch, H, G, d, (float)scale, rows, fp(out), stream.handle);
    }
    check_status(rc, what);
    return THPVariable_Wrap(out);
  });
}

// setup(path of libmixkv.so, error class): resolves the library's entry points.
PyObject* py_setup(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded(n, 2, [&]() -> PyObject* {
    const char* path = PyUnicode_AsUTF8(a[0]);
    if (!path) throw Raised();
    void* lib = dlopen(path, RTLD_NOW | RTLD_LOCAL);
    if (!lib) fail(PyExc_OSError, dlerror());
    auto get = [&](auto& fn, const char* name) {
      fn = reinterpret_cast<std::decay_t<decltype(fn)>>(dlsym(lib, name));
      if (!fn) fail(PyExc_OSError, name);
    };
    get(api.scores, "mixkv_internal_scores");
    get(api.select, "mixkv_internal_select");
    get(api.layer, "mixkv_compress_layer_traced");
    get(api.layers, "mixkv_compress_layers");
    get(api.budgeted, "mixkv_compress_layers_budgeted");
    get(api.ws_size, "mixkv_workspace_size_layers");
    get(api.sim_ws_size, "mixkv_similarity_workspace_size");
    get(api.sim_map, "mixkv_similarity_map");
    get(api.decode, "mixkv_decode_attention");
    Py_XSETREF(g_error, Py_NewRef(a[1]));
    Py_RETURN_NONE;
  });
}

#define FAST(f) reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(f)), METH_FASTCALL, nullptr
PyMethodDef methods[] = {{"setup", FAST(py_setup)},
                         {"scores", FAST(py_scores)},
                         {"select", FAST(py_select)},
                         {"compress_layer", FAST(py_compress_layer)},
                         {"compress_layers", FAST(py_compress_layers)},
                         {"similarity_map", FAST(py_similarity_map)},
                         {"decode_attention", FAST(py_decode_attention)},
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_mixkv_host", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__mixkv_host() {
#define NAME(x) nm.x = PyUnicode_InternFromString(#x)
  NAME(kv_heads), NAME(gqa_ratio), NAME(head_dim), NAME(window), NAME(pool_kernel), NAME(pool_mode),
      NAME(use_vnorm), NAME(mix_mode), NAME(budget_mode), NAME(budget), NAME(ada_floor), NAME(eps),
      NAME(softmax_scale), NAME(cuda_stream), NAME(s_comp), NAME(s_ex), NAME(s_div), NAME(rbar), NAME(status),
      NAME(idx), NAME(counts), NAME(idx_offsets), NAME(K_out), NAME(V_out), NAME(out_row_offsets);
#undef NAME
  return PyModule_Create(&module);
}
