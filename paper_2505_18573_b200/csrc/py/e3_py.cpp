// Python binding of the device calls (module `_native`): argument checks, output tensors, scratch and the call through
// the C ABI of include/e3.h, all in native code.  The wrappers with their signatures and defaults are in binding.py.
//
// Why native: a rollout step of a few microseconds of GPU work was bound by the host.  Marshalling in Python (attribute
// reads, torch.empty, an 18-argument ctypes call) took 18-20 us per e3_sample.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/cuda/EmptyTensor.h>
#include <ATen/core/Tensor.h>
#include <ATen/ops/empty_like.h>
#include <c10/cuda/CUDAException.h>
#include <c10/cuda/CUDAGuard.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <map>
#include <memory>
#include <mutex>
#include <utility>
#include <vector>

#include "e3.h"
#include "e3_internal.h"

namespace {

struct PyFailed {};  // a Python error has been set

[[noreturn]] void value_error(const char *text) {
  PyErr_SetString(PyExc_ValueError, text);
  throw PyFailed();
}

PyObject *g_error_class = nullptr;  // binding.E3Error

void check(const char *call, e3_status st) {
  if (st == E3_OK) return;
  PyObject *e = g_error_class ? PyObject_CallFunction(g_error_class, "si", call, static_cast<int>(st)) : nullptr;
  if (e) {
    PyErr_SetObject(g_error_class, e);
    Py_DECREF(e);
  } else if (!PyErr_Occurred()) {
    PyErr_Format(PyExc_RuntimeError, "%s failed: %s", call, e3_status_string(st));
  }
  throw PyFailed();
}

// ---- arguments -------------------------------------------------------------------------------------------------
const at::Tensor *optional_tensor(PyObject *o, const char *name) {
  if (o == Py_None) return nullptr;
  if (!THPVariable_Check(o)) {
    PyErr_Format(PyExc_TypeError, "%s must be a tensor", name);
    throw PyFailed();
  }
  return &THPVariable_Unpack(o);
}
const at::Tensor *device_tensor(PyObject *o, const char *name) {
  const at::Tensor *t = optional_tensor(o, name);
  if (t && !t->is_cuda()) {
    PyErr_Format(PyExc_ValueError, "%s must be a CUDA tensor (there is no CPU path)", name);
    throw PyFailed();
  }
  return t;
}
const at::Tensor &required_tensor(PyObject *o, const char *name) {
  const at::Tensor *t = device_tensor(o, name);
  if (!t) {
    PyErr_Format(PyExc_TypeError, "%s must be a tensor", name);
    throw PyFailed();
  }
  return *t;
}
template <class T = void>
T *pointer(const at::Tensor *t) {
  return t ? static_cast<T *>(t->data_ptr()) : nullptr;
}
template <class T = void>
T *pointer(const at::Tensor &t) {
  return static_cast<T *>(t.data_ptr());
}
uint64_t integer(PyObject *o) {  // any width: taken modulo 2^64
  const uint64_t v = PyLong_AsUnsignedLongLongMask(o);
  if (PyErr_Occurred()) throw PyFailed();
  return v;
}
float number(PyObject *o) {
  const double v = PyFloat_AsDouble(o);
  if (v == -1.0 && PyErr_Occurred()) throw PyFailed();
  return static_cast<float>(v);
}
bool truth(PyObject *o) {
  const int v = PyObject_IsTrue(o);
  if (v < 0) throw PyFailed();
  return v != 0;
}
bool has_dtype(const at::Tensor &t, at::ScalarType s) { return t.scalar_type() == s; }

struct Logits {
  void *data;
  e3_dtype dt;
  int64_t rows, V, stride;
  at::Device device;
};
Logits logits_of(const at::Tensor &t) {
  if (t.dim() != 2 || (t.size(1) > 1 && t.stride(1) != 1)) value_error("logits must be 2-D with a contiguous last dimension");
  Logits l{t.data_ptr(), E3_F32, t.size(0), t.size(1), t.stride(0), t.device()};
  if (has_dtype(t, at::kBFloat16)) l.dt = E3_BF16;
  else if (!has_dtype(t, at::kFloat)) value_error("logits must be float32 or bfloat16");
  if (l.rows <= 1 && l.stride < l.V) l.stride = l.V;
  return l;
}

cudaStream_t stream_of(PyObject *o) {
  if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
  PyObject *h = PyObject_GetAttrString(o, "cuda_stream");
  if (!h) throw PyFailed();
  const uint64_t v = PyLong_AsUnsignedLongLongMask(h);
  Py_DECREF(h);
  if (PyErr_Occurred()) throw PyFailed();
  return reinterpret_cast<cudaStream_t>(static_cast<uintptr_t>(v));
}

// ---- outputs ---------------------------------------------------------------------------------------------------
// A tensor that is returned: the caller's, or a new one (`make`), or None.
struct Output {
  PyObject *object = nullptr;  // borrowed, where the caller gave one
  at::Tensor made;
  bool any = false;
  template <class T>
  T *data() const {
    if (object) return static_cast<T *>(THPVariable_Unpack(object).data_ptr());
    return any ? static_cast<T *>(made.data_ptr()) : nullptr;
  }
  PyObject *release() const {  // new reference
    if (object) {
      Py_INCREF(object);
      return object;
    }
    if (any) return THPVariable_Wrap(made);
    Py_RETURN_NONE;
  }
};
at::Tensor empty(at::IntArrayRef size, at::ScalarType dtype, at::Device device) {
  return at::detail::empty_cuda(size, dtype, device, std::nullopt);
}
Output output(PyObject *given, const char *name, bool make, at::IntArrayRef size, at::ScalarType dtype, at::Device device) {
  Output o;
  if (optional_tensor(given, name)) {
    o.object = given;
    o.any = true;
  } else if (make) {
    o.made = empty(size, dtype, device);
    o.any = true;
  }
  return o;
}
PyObject *tuple_of(std::initializer_list<const Output *> outs) {
  PyObject *t = PyTuple_New(static_cast<Py_ssize_t>(outs.size()));
  if (!t) throw PyFailed();
  Py_ssize_t i = 0;
  for (const Output *o : outs) {
    PyObject *v = o->release();
    if (!v) {
      Py_DECREF(t);
      throw PyFailed();
    }
    PyTuple_SET_ITEM(t, i++, v);
  }
  return t;
}

// ---- scratch ---------------------------------------------------------------------------------------------------
// One buffer per (device, stream), grown on demand: calls that may overlap on the GPU must not share one.  It is allocated on
// the stream of the call, so that a buffer that is dropped (at most kMostKept are kept) is only ever used again in that stream's
// order.  A call into a stream that is being captured gets a buffer of that capture instead (one per capture and stream), which
// belongs to the graph: it lives until the graph and what has been instantiated from it are gone.  Callers that manage memory
// themselves pass `workspace=` instead.
constexpr size_t kMostKept = 64;
using Key = std::pair<int, cudaStream_t>;
std::map<Key, at::Tensor> *g_kept = new std::map<Key, at::Tensor>();  // used with the GIL held; never destroyed (torch may be gone by then)
std::mutex g_launch_lock;                                             // a call's kernels go to the stream together

at::Tensor buffer_on(cudaStream_t stream, size_t bytes, at::Device device) {
  const c10::cuda::CUDAStreamGuard guard(stream == nullptr || stream == cudaStreamLegacy
                                             ? c10::cuda::getDefaultCUDAStream(device.index())
                                             : c10::cuda::getStreamFromExternal(stream, device.index()));
  return empty({static_cast<int64_t>(bytes < 16 ? 16 : bytes)}, at::kByte, device);
}

// Buffers of captures.
using CaptureKey = std::pair<unsigned long long, cudaStream_t>;
struct GraphBuffer {
  CaptureKey key;
  at::Tensor tensor;
};
std::map<CaptureKey, GraphBuffer *> *g_captured = new std::map<CaptureKey, GraphBuffer *>();  // the largest of each; with the GIL held
std::mutex g_orphans_lock;
std::vector<GraphBuffer *> *g_orphans = new std::vector<GraphBuffer *>();  // their graphs are gone
// Called by the CUDA runtime, on a thread of its own that must not call it: the buffer waits for the next call.
void CUDART_CB orphan(void *b) {
  std::lock_guard<std::mutex> hold(g_orphans_lock);
  g_orphans->push_back(static_cast<GraphBuffer *>(b));
}
void free_orphans() {
  std::vector<GraphBuffer *> gone;
  {
    std::lock_guard<std::mutex> hold(g_orphans_lock);
    gone.swap(*g_orphans);
  }
  for (GraphBuffer *b : gone) {
    auto it = g_captured->find(b->key);
    if (it != g_captured->end() && it->second == b) g_captured->erase(it);
    delete b;
  }
}
at::Tensor graph_buffer(unsigned long long id, cudaGraph_t graph, cudaStream_t stream, size_t need, at::Device device) {
  const CaptureKey key(id, stream);
  auto it = g_captured->find(key);
  if (it != g_captured->end() && static_cast<size_t>(it->second->tensor.numel()) >= need) return it->second->tensor;
  auto b = std::make_unique<GraphBuffer>(GraphBuffer{key, buffer_on(stream, need, device)});
  cudaUserObject_t object;
  C10_CUDA_CHECK(cudaUserObjectCreate(&object, b.get(), orphan, 1, cudaUserObjectNoDestructorSync));
  GraphBuffer *const owned = b.release();
  const cudaError_t e = cudaGraphRetainUserObject(graph, object, 1, cudaGraphUserObjectMove);
  if (e != cudaSuccess) (void)cudaUserObjectRelease(object, 1);
  C10_CUDA_CHECK(e);
  (*g_captured)[key] = owned;
  return owned->tensor;
}

struct Scratch {
  at::Tensor hold;
  void *data = nullptr;
  size_t bytes = 0;
};
Scratch scratch(PyObject *given, size_t need, at::Device device, cudaStream_t stream) {
  Scratch s;
  if (const at::Tensor *t = optional_tensor(given, "workspace")) {
    s.data = t->data_ptr();
    s.bytes = static_cast<size_t>(t->numel()) * t->element_size();
    return s;
  }
  free_orphans();
  cudaStreamCaptureStatus status = cudaStreamCaptureStatusNone;
  unsigned long long id = 0;
  cudaGraph_t graph = nullptr;
  if (cudaStreamGetCaptureInfo_v2(stream, &status, &id, &graph, nullptr, nullptr) != cudaSuccess) {
    (void)cudaGetLastError();  // (the launch will say what is wrong with the stream)
    status = cudaStreamCaptureStatusNone;
  }
  if (status == cudaStreamCaptureStatusActive) {
    s.hold = graph_buffer(id, graph, stream, need, device);
  } else {
    const Key key(device.index(), stream);
    auto it = g_kept->find(key);
    if (it == g_kept->end() || static_cast<size_t>(it->second.numel()) < need) {
      at::Tensor fresh = buffer_on(stream, need, device);
      if (it != g_kept->end()) {
        it->second = std::move(fresh);
      } else {
        if (g_kept->size() >= kMostKept) g_kept->clear();
        it = g_kept->emplace(key, std::move(fresh)).first;
      }
    }
    s.hold = it->second;
  }
  s.data = s.hold.data_ptr();
  s.bytes = static_cast<size_t>(s.hold.numel());
  return s;
}

// Runs a call of the library without the GIL (a full launch queue may make it wait).  The call may throw (a tensor without
// memory of its own, as under vmap): the GIL is back before that leaves.
template <class F>
e3_status launch(F call) {
  struct Released {
    PyThreadState *save = PyEval_SaveThread();
    ~Released() { PyEval_RestoreThread(save); }
  } released;
  std::lock_guard<std::mutex> hold(g_launch_lock);
  return call();
}

// ---- calls -----------------------------------------------------------------------------------------------------
// Positional arguments, in the order of the wrappers of binding.py.
PyObject *sample(PyObject *const *a) {
  enum { kLogits, kTemps, kSeed, kCounter, kRowBase, kSampler, kTok, kLogp, kEnt, kWantLogp, kWantEnt, kGap, kWantGap, kStatus, kWorkspace, kStream };
  const Logits l = logits_of(required_tensor(a[kLogits], "logits"));
  const at::Tensor &temps = required_tensor(a[kTemps], "temps");
  if (!has_dtype(temps, at::kFloat) || temps.numel() != l.rows || !temps.is_contiguous())
    value_error("temps must be a contiguous float32 tensor with one entry per row");
  const uint64_t seed = integer(a[kSeed]), counter = integer(a[kCounter]);
  const int64_t row_base = static_cast<int64_t>(integer(a[kRowBase]));
  const e3_sampler sampler = static_cast<e3_sampler>(static_cast<int>(integer(a[kSampler])));
  const at::Tensor *status = optional_tensor(a[kStatus], "status");
  if (status && (!status->is_cuda() || !has_dtype(*status, at::kInt) || status->numel() < 1))
    value_error("status must be an int32 CUDA tensor");
  const Output tok = output(a[kTok], "out_tok", true, {l.rows}, at::kInt, l.device);
  const Output logp = output(a[kLogp], "out_logp", truth(a[kWantLogp]), {l.rows}, at::kFloat, l.device);
  const Output ent = output(a[kEnt], "out_ent", truth(a[kWantEnt]), {l.rows}, at::kFloat, l.device);
  const Output gap = output(a[kGap], "out_gap", truth(a[kWantGap]), {l.rows}, at::kFloat, l.device);
  const cudaStream_t stream = stream_of(a[kStream]);
  // the blocked sampler asks for its full size; for the others the room for cut rows is enough (that of a training pass of no rows)
  const size_t need = sampler == E3_SAMPLER_BLOCK ? e3_workspace_bytes(E3_CALL_SAMPLE, l.rows, l.V, l.dt)
                                                  : e3_workspace_bytes(E3_CALL_TOKEN_LOGP_ENTROPY, 0, l.V, l.dt);
  const Scratch ws = scratch(a[kWorkspace], need, l.device, stream);
  check("e3_sample", launch([&] {
          return e3_sample(l.data, l.dt, l.rows, l.V, l.stride, pointer<float>(temps), seed, counter, row_base, sampler,
                           tok.data<int32_t>(), logp.data<float>(), ent.data<float>(), gap.data<float>(),
                           pointer<int32_t>(status), ws.data, ws.bytes, stream);
        }));
  return gap.any ? tuple_of({&tok, &logp, &ent, &gap}) : tuple_of({&tok, &logp, &ent});
}

PyObject *token_logp_entropy(PyObject *const *a) {
  enum { kLogits, kTargets, kMask, kTemps, kTempScalar, kLogp, kEnt, kGap, kWantGap, kSum, kStatus, kWorkspace, kStream };
  const Logits l = logits_of(required_tensor(a[kLogits], "logits"));
  const at::Tensor &targets = required_tensor(a[kTargets], "targets");
  const at::Tensor *mask = device_tensor(a[kMask], "mask"), *temps = device_tensor(a[kTemps], "temps");
  if (!has_dtype(targets, at::kInt) || targets.numel() != l.rows) value_error("targets must be int32 with one entry per row");
  if (mask && (!has_dtype(*mask, at::kByte) || mask->numel() != l.rows)) value_error("mask must be uint8 with one entry per row");
  if (temps && (!has_dtype(*temps, at::kFloat) || temps->numel() != l.rows)) value_error("temps must be float32 with one entry per row");
  const float tau = number(a[kTempScalar]);
  const at::Tensor *sum = optional_tensor(a[kSum], "out_sum"), *status = optional_tensor(a[kStatus], "status");
  if (sum && (!sum->is_cuda() || !has_dtype(*sum, at::kDouble) || sum->numel() != 2 || !sum->is_contiguous()))
    value_error("out_sum must be a contiguous float64 CUDA tensor with two entries");
  if (status && (!status->is_cuda() || !has_dtype(*status, at::kInt) || status->numel() < 1))
    value_error("status must be an int32 CUDA tensor");
  const Output logp = output(a[kLogp], "out_logp", true, {l.rows}, at::kFloat, l.device);
  const Output ent = output(a[kEnt], "out_ent", true, {l.rows}, at::kFloat, l.device);
  const Output gap = output(a[kGap], "out_gap", truth(a[kWantGap]), {l.rows}, at::kFloat, l.device);
  const cudaStream_t stream = stream_of(a[kStream]);
  const Scratch ws = scratch(a[kWorkspace], e3_workspace_bytes(E3_CALL_TOKEN_LOGP_ENTROPY, l.rows, l.V, l.dt), l.device, stream);
  double *const s = pointer<double>(sum);
  check("e3_token_logp_entropy", launch([&] {
          return e3_token_logp_entropy(l.data, l.dt, l.rows, l.V, l.stride, pointer<int32_t>(targets), pointer<uint8_t>(mask),
                                       pointer<float>(temps), tau, logp.data<float>(), ent.data<float>(), gap.data<float>(), s,
                                       s ? s + 1 : nullptr, pointer<int32_t>(status), ws.data, ws.bytes, stream);
        }));
  return gap.any ? tuple_of({&logp, &ent, &gap}) : tuple_of({&logp, &ent});
}

PyObject *token_logp_entropy_backward(PyObject *const *a) {
  enum { kLogits, kTargets, kLogp, kEnt, kGLogp, kGEnt, kMask, kTemps, kTempScalar, kOut, kStream };
  static const char *const names[] = {"logits", "targets", "logp", "ent", "g_logp", "g_ent", "mask", "temps"};
  const at::Tensor &logits = required_tensor(a[kLogits], "logits");
  const Logits l = logits_of(logits);
  const at::Tensor *t[kTemps + 1] = {&logits};
  for (int i = kTargets; i <= kTemps; ++i) {
    t[i] = i <= kEnt ? &required_tensor(a[i], names[i]) : device_tensor(a[i], names[i]);
    if (t[i] && (t[i]->numel() != l.rows || !t[i]->is_contiguous())) {
      PyErr_Format(PyExc_ValueError, "%s must be contiguous with one entry per row", names[i]);
      throw PyFailed();
    }
  }
  if (!has_dtype(*t[kTargets], at::kInt) || !has_dtype(*t[kLogp], at::kFloat) || !has_dtype(*t[kEnt], at::kFloat))
    value_error("targets must be int32, logp and ent float32");
  const float tau = number(a[kTempScalar]);
  const Output out = output(a[kOut], "out", true, {l.rows, l.V}, logits.scalar_type(), l.device);
  Logits o = out.object ? logits_of(required_tensor(a[kOut], "out")) : logits_of(out.made);
  if (o.dt != l.dt || o.rows != l.rows || o.V != l.V) value_error("out must have the shape and dtype of logits");
  const cudaStream_t stream = stream_of(a[kStream]);
  check("e3_token_logp_entropy_backward", launch([&] {
          return e3_token_logp_entropy_backward(l.data, l.dt, l.rows, l.V, l.stride, pointer<int32_t>(t[kTargets]),
                                                pointer<uint8_t>(t[kMask]), pointer<float>(t[kTemps]), tau, pointer<float>(t[kLogp]),
                                                pointer<float>(t[kEnt]), pointer<float>(t[kGLogp]), pointer<float>(t[kGEnt]), o.data,
                                                o.stride, stream);
        }));
  return out.release();
}

// ent and mask of the mean entropies
void check_tokens(const at::Tensor &ent, const at::Tensor *mask) {
  if (!has_dtype(ent, at::kFloat) || !ent.is_contiguous()) value_error("ent must be a contiguous float32 tensor");
  if (mask && (!has_dtype(*mask, at::kByte) || mask->numel() != ent.numel())) value_error("mask must be uint8 with one entry per token");
}

PyObject *masked_mean_entropy(PyObject *const *a) {
  enum { kEnt, kMask, kOut, kWorkspace, kStream };
  const at::Tensor &ent = required_tensor(a[kEnt], "ent");
  const at::Tensor *mask = device_tensor(a[kMask], "mask");
  check_tokens(ent, mask);
  const int64_t n = ent.numel();
  const Output out = output(a[kOut], "out", true, {2}, at::kDouble, ent.device());
  const cudaStream_t stream = stream_of(a[kStream]);
  const Scratch ws = scratch(a[kWorkspace], e3_workspace_bytes(E3_CALL_MASKED_MEAN_ENTROPY, n, 0, E3_F32), ent.device(), stream);
  double *const o = out.data<double>();
  check("e3_masked_mean_entropy", launch([&] {
          return e3_masked_mean_entropy(pointer<float>(ent), pointer<uint8_t>(mask), n, o, o + 1, ws.data, ws.bytes, stream);
        }));
  return out.release();
}

PyObject *sequence_mean_entropy(PyObject *const *a) {
  enum { kEnt, kMask, kOut, kWorkspace, kStream };
  const at::Tensor &ent = required_tensor(a[kEnt], "ent");
  const at::Tensor *mask = device_tensor(a[kMask], "mask");
  if (ent.dim() != 2 || !has_dtype(ent, at::kFloat) || !ent.is_contiguous())
    value_error("ent must be a contiguous float32 tensor [n_seq, seq_len]");
  if (mask && (!has_dtype(*mask, at::kByte) || mask->numel() != ent.numel() || !mask->is_contiguous()))
    value_error("mask must be contiguous uint8 with one entry per token");
  const Output out = output(a[kOut], "out", true, {2}, at::kDouble, ent.device());
  const cudaStream_t stream = stream_of(a[kStream]);
  const Scratch ws = scratch(a[kWorkspace], e3_workspace_bytes(E3_CALL_SEQUENCE_MEAN_ENTROPY, ent.size(0), 0, E3_F32), ent.device(), stream);
  double *const o = out.data<double>();
  check("e3_sequence_mean_entropy", launch([&] {
          return e3_sequence_mean_entropy(pointer<float>(ent), pointer<uint8_t>(mask), ent.size(0), ent.size(1), o, o + 1, ws.data,
                                          ws.bytes, stream);
        }));
  return out.release();
}

PyObject *masked_mean_entropy_static(PyObject *const *a) {
  enum { kEnt, kMask, kOut, kStream };
  const at::Tensor &ent = required_tensor(a[kEnt], "ent");
  const at::Tensor *mask = device_tensor(a[kMask], "mask");
  check_tokens(ent, mask);
  const Output out = output(a[kOut], "out", true, {2}, at::kDouble, ent.device());
  const cudaStream_t stream = stream_of(a[kStream]);
  double *const o = out.data<double>();
  check("e3_masked_mean_entropy_static", launch([&] {
          return e3_masked_mean_entropy_static(pointer<float>(ent), pointer<uint8_t>(mask), ent.numel(), o, o + 1, stream);
        }));
  return out.release();
}

PyObject *group_advantage(PyObject *const *a) {
  enum { kRewards, kOffsets, kEps, kUnbiased, kAdv, kFlags, kWantFlags, kStream };
  const at::Tensor &rewards = required_tensor(a[kRewards], "rewards"), &offsets = required_tensor(a[kOffsets], "group_offsets");
  if (!has_dtype(rewards, at::kFloat) || !has_dtype(offsets, at::kLong))
    value_error("rewards must be float32 and group_offsets int64");
  const int64_t ng = offsets.numel() - 1;
  const float eps = number(a[kEps]);
  const int unbiased = truth(a[kUnbiased]) ? 1 : 0;
  const bool own_adv = a[kAdv] == Py_None, own_flags = a[kFlags] == Py_None && truth(a[kWantFlags]);
  Output adv = output(a[kAdv], "out_adv", rewards.is_contiguous(), rewards.sizes(), at::kFloat, rewards.device());
  if (!adv.any) {  // groups go by the order in memory: permuted rewards give advantages permuted alike
    adv.made = at::empty_like(rewards);
    adv.any = true;
  }
  const Output flags = output(a[kFlags], "out_flags", own_flags, {ng < 0 ? 0 : ng}, at::kByte, rewards.device());
  const cudaStream_t stream = stream_of(a[kStream]);
  check("e3_group_advantage", launch([&] {
          if (own_adv && (own_flags || !flags.any))  // new tensors: what no group covers reads 0
            return e3::group_advantage_filled(pointer<float>(rewards), rewards.numel(), pointer<int64_t>(offsets), ng, eps, unbiased,
                                              adv.data<float>(), flags.data<uint8_t>(), stream);
          // a new tensor beside one of the caller's: cleared, then the groups' entries are written
          if (own_adv && cudaMemsetAsync(adv.data<float>(), 0, rewards.numel() * sizeof(float), stream) != cudaSuccess) return E3_ERR_CUDA;
          if (own_flags && ng > 0 && cudaMemsetAsync(flags.data<uint8_t>(), 0, ng, stream) != cudaSuccess) return E3_ERR_CUDA;
          return e3_group_advantage(pointer<float>(rewards), pointer<int64_t>(offsets), ng, eps, unbiased, adv.data<float>(),
                                    flags.data<uint8_t>(), stream);
        }));
  return tuple_of({&adv, &flags});
}

PyObject *grpo_objective(PyObject *const *a) {
  enum { kLogp, kLogpOld, kAdv, kOffsets, kMask, kClip, kGrad, kWantGrad, kOut, kWorkspace, kStream };
  const at::Tensor &logp = required_tensor(a[kLogp], "logp"), &old = required_tensor(a[kLogpOld], "logp_old");
  const at::Tensor &adv = required_tensor(a[kAdv], "adv"), &offsets = required_tensor(a[kOffsets], "group_offsets");
  const at::Tensor *mask = device_tensor(a[kMask], "mask");
  if (logp.dim() != 2 || !logp.sizes().equals(old.sizes()) || !logp.is_contiguous() || !old.is_contiguous())
    value_error("logp and logp_old must be contiguous [n_seq, seq_len] tensors of the same shape");
  if (!has_dtype(logp, at::kFloat) || !has_dtype(old, at::kFloat) || !has_dtype(adv, at::kFloat))
    value_error("logp, logp_old and adv must be float32");
  const int64_t n_seq = logp.size(0), seq_len = logp.size(1);
  if (adv.numel() != n_seq || !has_dtype(offsets, at::kLong))
    value_error("adv needs one entry per response, group_offsets must be int64");
  if (mask && (!has_dtype(*mask, at::kByte) || mask->numel() != n_seq * seq_len || !mask->is_contiguous()))
    value_error("mask must be contiguous uint8 with one entry per token");
  const float clip = number(a[kClip]);
  const Output grad = output(a[kGrad], "out_g_logp", truth(a[kWantGrad]), {n_seq, seq_len}, at::kFloat, logp.device());
  const Output out = output(a[kOut], "out", true, {2}, at::kDouble, logp.device());
  const cudaStream_t stream = stream_of(a[kStream]);
  const Scratch ws = scratch(a[kWorkspace], e3_workspace_bytes(E3_CALL_GRPO_OBJECTIVE, n_seq, 0, E3_F32), logp.device(), stream);
  double *const o = out.data<double>();
  check("e3_grpo_objective", launch([&] {
          return e3_grpo_objective(pointer<float>(logp), pointer<float>(old), pointer<uint8_t>(mask), n_seq, seq_len, pointer<float>(adv),
                                   pointer<int64_t>(offsets), offsets.numel() - 1, clip, grad.data<float>(), o, o + 1, ws.data, ws.bytes,
                                   stream);
        }));
  return tuple_of({&out, &grad});
}

// ---- module ----------------------------------------------------------------------------------------------------
template <PyObject *(*F)(PyObject *const *), int N>
PyObject *entry(PyObject *, PyObject *const *args, Py_ssize_t n) {
  if (n != N) {
    PyErr_Format(PyExc_TypeError, "%d arguments expected, got %zd", N, n);
    return nullptr;
  }
  try {
    return F(args);
  } catch (const PyFailed &) {
    return nullptr;
  } catch (const std::exception &e) {
    PyErr_SetString(PyExc_RuntimeError, e.what());
    return nullptr;
  }
}
PyObject *set_error_class(PyObject *, PyObject *cls) {
  Py_INCREF(cls);
  Py_XSETREF(g_error_class, cls);
  Py_RETURN_NONE;
}

#define E3_ENTRY(f, n) {#f, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(entry<f, n>)), METH_FASTCALL, nullptr}
PyMethodDef g_methods[] = {
    E3_ENTRY(sample, 16), E3_ENTRY(token_logp_entropy, 13), E3_ENTRY(token_logp_entropy_backward, 11),
    E3_ENTRY(masked_mean_entropy, 5), E3_ENTRY(sequence_mean_entropy, 5), E3_ENTRY(masked_mean_entropy_static, 4),
    E3_ENTRY(group_advantage, 8), E3_ENTRY(grpo_objective, 11), {"set_error_class", set_error_class, METH_O, nullptr},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef g_module = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, g_methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native() { return PyModule_Create(&g_module); }
