// Argument marshalling of the Python binding for the calls that a program makes again and again: tensors become pointers,
// sizes and strides here instead of through a dozen Python attribute look-ups per tensor.  One call of tq_attend_decode
// with two channel groups unpacks 20 tensors: 14-17 us of host time through ctypes, more than its kernels take on a short
// context.  No computation happens here; binding.py keeps the signatures and raises the errors.
#include <Python.h>
#include <dlfcn.h>

#include <ATen/ATen.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "tq.h"

namespace {

struct Api {
#define TQ_API(name) decltype(&::name) name = nullptr;
#define TQ_API_LIST(X)                                                                                                   \
  X(tq_quantize_mse) X(tq_quantize_prod) X(tq_dequantize) X(tq_score) X(tq_score_static) X(tq_query_prepare)             \
  X(tq_score_prepared) X(tq_topk) X(tq_select_topk) X(tq_wsum) X(tq_softmax) X(tq_attend_decode) X(tq_kv_append)         \
  X(tq_entropy_workspace_bytes) X(tq_entropy_measure) X(tq_entropy_pack) X(tq_entropy_unpack)
  TQ_API_LIST(TQ_API)
} api;

// ---- a failed conversion sets the Python error and makes the caller return nullptr
struct Failed {};
[[noreturn]] void fail(const char* msg) {
  PyErr_SetString(PyExc_ValueError, msg);
  throw Failed();
}

const at::Tensor& tensor(PyObject* o) {
  if (!THPVariable_Check(o)) fail("expected a CUDA tensor (this library has no CPU path)");
  return THPVariable_Unpack(o);
}
void* dev(PyObject* o) {
  if (o == Py_None || o == nullptr) return nullptr;
  const at::Tensor& t = tensor(o);
  if (!t.is_cuda()) fail("expected a CUDA tensor (this library has no CPU path)");
  return t.data_ptr();
}
template <typename T>
T* dev(PyObject* o) { return static_cast<T*>(dev(o)); }

struct Rows {
  void* p;
  int64_t n, ld, cols;
  at::ScalarType type;
};
Rows rows(PyObject* o) {
  const at::Tensor& t = tensor(o);
  if (!t.is_cuda()) fail("expected a CUDA tensor (this library has no CPU path)");
  if (t.dim() != 2 || t.stride(1) != 1) fail("expected a 2-D tensor with unit inner stride");
  const int64_t n = t.size(0), cols = t.size(1);
  return {t.data_ptr(), n, n > 1 ? t.stride(0) : std::max(t.stride(0), cols), cols, t.scalar_type()};
}
int dtype_code(const Rows& r) {
  if (r.type == at::kFloat) return TQ_F32;
  if (r.type == at::kBFloat16) return TQ_BF16;
  fail("unsupported dtype: expected torch.float32 or torch.bfloat16");
}
struct Bytes {
  void* p;
  size_t n;
};
Bytes scratch(PyObject* o) {
  if (o == Py_None || o == nullptr) return {nullptr, 0};
  const at::Tensor& t = tensor(o);
  return {dev(o), (size_t)t.numel() * t.element_size()};
}
int64_t integer(PyObject* o) {
  const long long v = PyLong_AsLongLong(o);
  if (v == -1 && PyErr_Occurred()) throw Failed();
  return v;
}
int int32(PyObject* o) {
  const int64_t v = integer(o);
  if (v != (int)v) fail("integer argument out of range");
  return (int)v;
}
double real(PyObject* o) {
  const double v = PyFloat_AsDouble(o);
  if (v == -1.0 && PyErr_Occurred()) throw Failed();
  return v;
}
const tq_plan* plan_of(PyObject* o) {
  return o == Py_None ? nullptr : reinterpret_cast<const tq_plan*>(static_cast<uintptr_t>(integer(o)));
}
const uint8_t* host_bytes(PyObject* o) { return reinterpret_cast<const uint8_t*>(static_cast<uintptr_t>(integer(o))); }
void* stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

// Runs `call` without the interpreter lock and returns its status as a Python integer.
template <typename F>
PyObject* run(F&& call) {
  int rc;
  Py_BEGIN_ALLOW_THREADS;
  rc = call();
  Py_END_ALLOW_THREADS;
  return PyLong_FromLong(rc);
}

#define TQ_FN(name, count)                                                                   \
  PyObject* name##_impl(PyObject* const* a);                                                 \
  PyObject* name(PyObject*, PyObject* const* a, Py_ssize_t n) {                              \
    if (n != (count)) return PyErr_Format(PyExc_TypeError, #name ": expected %d arguments", (count)); \
    try {                                                                                    \
      return name##_impl(a);                                                                 \
    } catch (const Failed&) {                                                                \
      return nullptr;                                                                        \
    } catch (const std::exception& e) {                                                      \
      PyErr_SetString(PyExc_RuntimeError, e.what());                                         \
      return nullptr;                                                                        \
    }                                                                                        \
  }                                                                                          \
  PyObject* name##_impl(PyObject* const* a)

TQ_FN(quantize_mse, 5) {   // plan, X, idx, norms, scratch
  const Rows x = rows(a[1]);
  const int dt = dtype_code(x);
  uint8_t* idx = dev<uint8_t>(a[2]);
  float* norms = dev<float>(a[3]);
  const Bytes s = scratch(a[4]);
  const tq_plan* p = plan_of(a[0]);
  void* st = stream();
  return run([&] { return api.tq_quantize_mse(p, x.p, dt, x.n, x.ld, idx, norms, s.p, s.n, st); });
}

TQ_FN(quantize_prod, 7) {   // plan, X, idx, qjl, gamma, norms, scratch
  const Rows x = rows(a[1]);
  const int dt = dtype_code(x);
  uint8_t *idx = dev<uint8_t>(a[2]), *qjl = dev<uint8_t>(a[3]);
  float *gamma = dev<float>(a[4]), *norms = dev<float>(a[5]);
  const Bytes s = scratch(a[6]);
  const tq_plan* p = plan_of(a[0]);
  void* st = stream();
  return run([&] { return api.tq_quantize_prod(p, x.p, dt, x.n, x.ld, idx, qjl, gamma, norms, s.p, s.n, st); });
}

struct Codes {
  const uint8_t *idx, *qjl;
  const float *gamma, *norms;
};
Codes codes(PyObject* const* a) { return {dev<uint8_t>(a[0]), dev<uint8_t>(a[1]), dev<float>(a[2]), dev<float>(a[3])}; }

TQ_FN(dequantize, 7) {   // plan, n, idx, qjl, gamma, norms, Xhat
  const Rows x = rows(a[6]);
  const Codes c = codes(a + 2);
  const tq_plan* p = plan_of(a[0]);
  const int64_t n = integer(a[1]);
  void* st = stream();
  return run([&] { return api.tq_dequantize(p, n, c.idx, c.qjl, c.gamma, c.norms, static_cast<float*>(x.p), x.ld, st); });
}

TQ_FN(score, 9) {   // plan, Q, n, idx, qjl, gamma, norms, scores, workspace
  const Rows q = rows(a[1]), s = rows(a[7]);
  const int dt = dtype_code(q);
  const Codes c = codes(a + 3);
  const Bytes w = scratch(a[8]);
  const tq_plan* p = plan_of(a[0]);
  const int64_t n = integer(a[2]);
  void* st = stream();
  return run([&] {
    return api.tq_score(p, q.p, dt, (int)q.n, q.ld, n, c.idx, c.qjl, c.gamma, c.norms, static_cast<float*>(s.p), s.ld, w.p, w.n, st);
  });
}

TQ_FN(score_static, 8) {   // plan, Q, n, idx, qjl, gamma, norms, scores
  const Rows q = rows(a[1]), s = rows(a[7]);
  const int dt = dtype_code(q);
  const Codes c = codes(a + 3);
  const tq_plan* p = plan_of(a[0]);
  const int64_t n = integer(a[2]);
  void* st = stream();
  return run([&] {
    return api.tq_score_static(p, q.p, dt, (int)q.n, q.ld, n, c.idx, c.qjl, c.gamma, c.norms, static_cast<float*>(s.p), s.ld, st);
  });
}

TQ_FN(query_prepare, 3) {   // plan, Q, prepared
  const Rows q = rows(a[1]);
  const int dt = dtype_code(q);
  const Bytes w = scratch(a[2]);
  const tq_plan* p = plan_of(a[0]);
  void* st = stream();
  return run([&] { return api.tq_query_prepare(p, q.p, dt, (int)q.n, q.ld, w.p, w.n, st); });
}

TQ_FN(score_prepared, 9) {   // plan, prepared, nq, n, idx, qjl, gamma, norms, scores
  const Rows s = rows(a[8]);
  const void* prepared = dev(a[1]);
  const Codes c = codes(a + 4);
  const tq_plan* p = plan_of(a[0]);
  const int nq = int32(a[2]);
  const int64_t n = integer(a[3]);
  void* st = stream();
  return run([&] { return api.tq_score_prepared(p, prepared, nq, n, c.idx, c.qjl, c.gamma, c.norms, static_cast<float*>(s.p), s.ld, st); });
}

TQ_FN(topk, 11) {   // plan, Q, n, idx, qjl, gamma, norms, k, top_scores, top_ids, workspace
  const Rows q = rows(a[1]);
  const int dt = dtype_code(q);
  const Codes c = codes(a + 3);
  float* ts = dev<float>(a[8]);
  int32_t* ti = dev<int32_t>(a[9]);
  const Bytes w = scratch(a[10]);
  const tq_plan* p = plan_of(a[0]);
  const int64_t n = integer(a[2]);
  const int k = int32(a[7]);
  void* st = stream();
  return run([&] { return api.tq_topk(p, q.p, dt, (int)q.n, q.ld, n, c.idx, c.qjl, c.gamma, c.norms, k, ts, ti, w.p, w.n, st); });
}

TQ_FN(select_topk, 5) {   // cand_scores, cand_ids, k, top_scores, top_ids
  const Rows s = rows(a[0]), i = rows(a[1]);
  if (i.ld != s.ld || i.n != s.n || i.cols != s.cols) fail("cand_ids must have the shape and row stride of cand_scores");
  float* ts = dev<float>(a[3]);
  int32_t* ti = dev<int32_t>(a[4]);
  const int k = int32(a[2]);
  void* st = stream();
  return run([&] {
    return api.tq_select_topk(static_cast<const float*>(s.p), static_cast<const int32_t*>(i.p), (int)s.n, s.cols, s.ld, k, ts, ti, st);
  });
}

TQ_FN(wsum, 9) {   // plan, W, n, idx, qjl, gamma, norms, out, workspace
  const Rows o = rows(a[7]);
  const int64_t n = integer(a[2]);
  const float* W = dev<float>(a[1]);
  const int64_t ldw = W ? rows(a[1]).ld : n;
  const Codes c = codes(a + 3);
  const Bytes w = scratch(a[8]);
  const tq_plan* p = plan_of(a[0]);
  void* st = stream();
  return run([&] { return api.tq_wsum(p, W, (int)o.n, ldw, n, c.idx, c.qjl, c.gamma, c.norms, static_cast<float*>(o.p), o.ld, w.p, w.n, st); });
}

TQ_FN(softmax, 4) {   // s1, s2, scale, W
  const Rows s = rows(a[0]), w = rows(a[3]);
  const float* s2 = nullptr;
  if (a[1] != Py_None) {
    const Rows t = rows(a[1]);
    if (t.ld != s.ld || t.n != s.n || t.cols != s.cols) fail("s2 must have the shape and row stride of s1");
    s2 = static_cast<const float*>(t.p);
  }
  const float scale = (float)real(a[2]);
  void* st = stream();
  return run([&] {
    return api.tq_softmax(static_cast<const float*>(s.p), s2, (int)s.n, s.cols, s.ld, scale, static_cast<float*>(w.p), w.ld, st);
  });
}

// ---- channel groups of a compressed KV layer: a sequence of dicts (or of other mappings, which are copied into dicts)
enum { kPlanK, kPlanV, kKIdx, kKQjl, kKGamma, kKNorms, kVIdx, kVNorms, kKChan, kVChan, kKeys };
PyObject* keys[kKeys];
PyObject* handle_name;

struct Groups {
  tq_kv_group g[TQ_MAX_KV_GROUPS];
  int n;
  PyObject* copies[TQ_MAX_KV_GROUPS] = {};   // they keep the tensors until the call has returned
  ~Groups() {
    for (PyObject* c : copies) Py_XDECREF(c);
  }
};

PyObject* item(PyObject* dict, int key, bool needed) {
  PyObject* v = PyDict_GetItemWithError(dict, keys[key]);   // borrowed
  if (v == nullptr) {
    if (PyErr_Occurred()) throw Failed();
    if (needed) {
      PyErr_SetObject(PyExc_KeyError, keys[key]);
      throw Failed();
    }
  }
  return v;
}
const tq_plan* group_plan(PyObject* dict, int key) {
  PyObject* h = PyObject_GetAttr(item(dict, key, true), handle_name);
  if (h == nullptr) throw Failed();
  const void* p = h == Py_None ? nullptr : PyLong_AsVoidPtr(h);
  Py_DECREF(h);
  if (p == nullptr && PyErr_Occurred()) throw Failed();
  return static_cast<const tq_plan*>(p);
}
const int32_t* channels(PyObject* dict, int key) {
  PyObject* o = item(dict, key, true);
  const at::Tensor& t = tensor(o);
  if (t.scalar_type() != at::kInt || !t.is_contiguous()) fail("k_channels and v_channels must be contiguous int32 tensors");
  return dev<int32_t>(o);
}
void kv_groups(PyObject* seq, Groups* out) {
  PyObject* fast = PySequence_Fast(seq, "groups must be a sequence of dicts");
  if (fast == nullptr) throw Failed();
  struct Release {
    PyObject* o;
    ~Release() { Py_DECREF(o); }
  } release{fast};
  const Py_ssize_t n = PySequence_Fast_GET_SIZE(fast);
  out->n = (int)n;
  for (Py_ssize_t i = 0; i < n && i < TQ_MAX_KV_GROUPS; ++i) {   // more groups than that: the library rejects the count
    PyObject* d = PySequence_Fast_GET_ITEM(fast, i);
    if (!PyDict_Check(d)) {
      d = out->copies[i] = PyDict_New();
      if (d == nullptr || PyDict_Update(d, PySequence_Fast_GET_ITEM(fast, i)) != 0) throw Failed();
    }
    tq_kv_group& g = out->g[i];
    g.plan_k = group_plan(d, kPlanK);
    g.plan_v = group_plan(d, kPlanV);
    g.k_idx = dev<uint8_t>(item(d, kKIdx, false));
    g.k_qjl = dev<uint8_t>(item(d, kKQjl, false));
    g.k_gamma = dev<float>(item(d, kKGamma, false));
    g.k_norms = dev<float>(item(d, kKNorms, false));
    g.v_idx = dev<uint8_t>(item(d, kVIdx, false));
    g.v_norms = dev<float>(item(d, kVNorms, false));
    g.k_channels = channels(d, kKChan);
    g.v_channels = channels(d, kVChan);
  }
}

TQ_FN(attend_decode, 9) {   // groups, heads, tokens, head_stride, q_per_kv, Q, scale, out, workspace
  Groups g;
  kv_groups(a[0], &g);
  const Rows q = rows(a[5]), o = rows(a[7]);
  const int dt = dtype_code(q), heads = int32(a[1]), q_per_kv = int32(a[4]);
  const int64_t tokens = integer(a[2]), stride = integer(a[3]);
  const float scale = (float)real(a[6]);
  const Bytes w = scratch(a[8]);
  void* st = stream();
  return run([&] {
    return api.tq_attend_decode(g.g, g.n, heads, tokens, stride, q_per_kv, q.p, dt, q.ld, scale, static_cast<float*>(o.p), o.ld, w.p, w.n, st);
  });
}

TQ_FN(kv_append, 6) {   // groups, heads, head_stride, position, K, V
  Groups g;
  kv_groups(a[0], &g);
  const Rows k = rows(a[4]), v = rows(a[5]);
  if (k.type != v.type) fail("K and V must have one dtype");
  const int dt = dtype_code(k), heads = int32(a[1]);
  const int64_t stride = integer(a[2]), position = integer(a[3]);
  void* st = stream();
  return run([&] { return api.tq_kv_append(g.g, g.n, heads, stride, position, k.p, v.p, dt, k.ld, v.ld, st); });
}

// Measures, reads the total back and packs.  Returns (packed, offsets), or the failed call's status.
TQ_FN(entropy_pack, 4) {   // plan, lengths (host address), n, idx
  const tq_plan* p = plan_of(a[0]);
  const uint8_t* lengths = host_bytes(a[1]);
  const int64_t n = integer(a[2]);
  const uint8_t* idx = dev<uint8_t>(a[3]);
  const auto cuda = tensor(a[3]).device();
  at::Tensor offsets = at::empty({n + 1}, at::TensorOptions().dtype(at::kLong).device(cuda));
  at::Tensor total = at::empty({1}, at::TensorOptions().dtype(at::kLong).pinned_memory(true));
  const size_t need = api.tq_entropy_workspace_bytes(n);
  at::Tensor ws = at::empty({(int64_t)std::max<size_t>(need, 256)}, at::TensorOptions().dtype(at::kByte).device(cuda));
  uint64_t* off = reinterpret_cast<uint64_t*>(offsets.data_ptr());
  const cudaStream_t st = c10::cuda::getCurrentCUDAStream().stream();
  int rc;
  cudaError_t e = cudaSuccess;
  Py_BEGIN_ALLOW_THREADS;
  rc = api.tq_entropy_measure(p, lengths, n, idx, off, ws.data_ptr(), (size_t)ws.numel(), st);
  if (rc == TQ_OK) {
    e = cudaMemcpyAsync(total.data_ptr(), off + n, 8, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  }
  Py_END_ALLOW_THREADS;
  if (rc != TQ_OK) return PyLong_FromLong(rc);
  if (e != cudaSuccess) {
    PyErr_SetString(PyExc_RuntimeError, cudaGetErrorString(e));
    return nullptr;
  }
  const int64_t bytes = *static_cast<const int64_t*>(total.data_ptr());
  at::Tensor out = at::empty({std::max<int64_t>(bytes, 4)}, at::TensorOptions().dtype(at::kByte).device(cuda));
  uint8_t* dst = static_cast<uint8_t*>(out.data_ptr());
  Py_BEGIN_ALLOW_THREADS;
  rc = api.tq_entropy_pack(p, lengths, n, idx, off, dst, (size_t)bytes, st);
  Py_END_ALLOW_THREADS;
  if (rc != TQ_OK) return PyLong_FromLong(rc);
  return Py_BuildValue("(NN)", THPVariable_Wrap(bytes == out.numel() ? out : out.narrow(0, 0, bytes)), THPVariable_Wrap(offsets));
}

TQ_FN(entropy_unpack, 6) {   // plan, lengths (host address), n, packed, offsets, idx
  const tq_plan* p = plan_of(a[0]);
  const uint8_t* lengths = host_bytes(a[1]);
  const int64_t n = integer(a[2]);
  const uint8_t* packed = dev<uint8_t>(a[3]);
  const uint64_t* off = reinterpret_cast<const uint64_t*>(dev(a[4]));
  uint8_t* idx = dev<uint8_t>(a[5]);
  void* st = stream();
  return run([&] { return api.tq_entropy_unpack(p, lengths, n, packed, off, idx, st); });
}

// Resolves the library's entry points in the shared object that binding.py has loaded.
PyObject* bind(PyObject*, PyObject* path) {
  const char* file = PyUnicode_AsUTF8(path);
  if (file == nullptr) return nullptr;
  void* h = dlopen(file, RTLD_NOW);
  if (h == nullptr) return PyErr_Format(PyExc_RuntimeError, "%s", dlerror());
#define TQ_RESOLVE(name)                                                                          \
  api.name = reinterpret_cast<decltype(api.name)>(dlsym(h, #name));                               \
  if (api.name == nullptr) return PyErr_Format(PyExc_RuntimeError, "%s does not export " #name, file);
  TQ_API_LIST(TQ_RESOLVE)
  Py_RETURN_NONE;
}

#define TQ_DEF(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(name)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {{"bind", bind, METH_O, nullptr},
                         TQ_DEF(quantize_mse), TQ_DEF(quantize_prod), TQ_DEF(dequantize), TQ_DEF(score), TQ_DEF(score_static),
                         TQ_DEF(query_prepare), TQ_DEF(score_prepared), TQ_DEF(topk), TQ_DEF(select_topk), TQ_DEF(wsum),
                         TQ_DEF(softmax), TQ_DEF(attend_decode), TQ_DEF(kv_append), TQ_DEF(entropy_pack), TQ_DEF(entropy_unpack),
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_tqbind", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__tqbind() {
  static const char* names[kKeys] = {"plan_k", "plan_v", "k_idx", "k_qjl", "k_gamma", "k_norms", "v_idx", "v_norms", "k_channels", "v_channels"};
  for (int i = 0; i < kKeys; ++i)
    if ((keys[i] = PyUnicode_InternFromString(names[i])) == nullptr) return nullptr;
  if ((handle_name = PyUnicode_InternFromString("handle")) == nullptr) return nullptr;
  return PyModule_Create(&module);
}
