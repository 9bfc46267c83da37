// _qbert: the Python entry to libqbert's C ABI for the calls that a model makes on every pass.
//
// A quantized linear at a few dozen tokens keeps the GPU busy for about ten microseconds; through ctypes,
// torch.empty and torch.cuda.current_stream the same two calls took the host more than thirty (an output
// allocated from Python 2.5 us each, the stream 3.2 us, seventeen converted arguments 1.5 us).  Here the
// tensors are read, the outputs allocated and the stream looked up in C++, so that a call costs the host
// little more than its launches.  Marshalling only: no arithmetic, no state, no fallback.  The interpreter's lock is
// released while outputs are allocated and the library runs: both can block (a full launch queue, an allocation that has to
// free first), and other threads go on meanwhile.
//
// Every function takes its arguments by position (the wrappers in __init__.py give them names and
// defaults) and raises what the wrapper's own checks would: AssertionError for a tensor of the wrong kind,
// QbertError (through the function set by set_raise) for a status.
#include <Python.h>

#include <ATen/cuda/EmptyTensor.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include <algorithm>
#include <utility>

#include "qbert.h"

namespace {

PyObject* g_raise = nullptr;  // __init__._raise(status, what)

struct Failed {};  // a Python error is set

[[noreturn]] void fail(PyObject* type, const char* text) {
  PyErr_SetString(type, text);
  throw Failed{};
}
void need(bool ok, const char* text) {
  if (!ok) fail(PyExc_AssertionError, text);
}
void check(qb_status st, const char* what) {
  if (st == QB_OK) return;
  PyObject* r = PyObject_CallFunction(g_raise, "is", (int)st, what);
  Py_XDECREF(r);
  if (!PyErr_Occurred()) PyErr_SetString(PyExc_RuntimeError, what);
  throw Failed{};
}

const at::Tensor& tensor(PyObject* o) {
  if (!THPVariable_Check(o)) fail(PyExc_TypeError, "expected a torch.Tensor");
  return THPVariable_Unpack(o);
}
const at::Tensor& input(PyObject* o, at::ScalarType type, const char* what) {
  const at::Tensor& t = tensor(o);
  need(t.is_cuda() && t.scalar_type() == type && t.is_contiguous(), what);
  return t;
}
void* ptr(PyObject* o) { return o == Py_None ? nullptr : tensor(o).data_ptr(); }
int64_t integer(PyObject* o) {
  const long long v = PyLong_AsLongLong(o);
  if (v == -1 && PyErr_Occurred()) throw Failed{};
  return v;
}
void* stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

// Other Python threads run while one of these lives; no Python object may be touched.
struct Unlocked {
  PyThreadState* const state = PyEval_SaveThread();
  Unlocked() = default;
  Unlocked(const Unlocked&) = delete;
  ~Unlocked() { PyEval_RestoreThread(state); }
};

// An output: the caller's tensor, or a new one that `make` allocates (a caller's tensor stays).  `get` hands over a new
// reference.
struct Out {
  PyObject* obj = nullptr;
  void* data = nullptr;
  at::Tensor made;
  explicit Out(PyObject* given) {
    if (given == Py_None) return;
    data = tensor(given).data_ptr();
    obj = Py_NewRef(given);
  }
  Out(const Out&) = delete;
  ~Out() { Py_XDECREF(obj); }
  void make(at::IntArrayRef shape, at::ScalarType type, at::Device device) {
    if (obj) return;
    made = at::Tensor(at::detail::empty_cuda(shape, type, device, std::nullopt));
    data = made.data_ptr();
  }
  void wrap() {
    if (!obj) obj = THPVariable_Wrap(std::move(made));
    if (!obj) throw Failed{};
  }
  PyObject* get() {
    wrap();
    return std::exchange(obj, nullptr);
  }
};
PyObject* triple(Out& a, Out& b, Out& c) {
  a.wrap();
  b.wrap();
  c.wrap();
  PyObject* r = PyTuple_New(3);
  if (!r) throw Failed{};
  PyTuple_SET_ITEM(r, 0, a.get());
  PyTuple_SET_ITEM(r, 1, b.get());
  PyTuple_SET_ITEM(r, 2, c.get());
  return r;
}

struct Workspace {
  void* data;
  size_t bytes;
  explicit Workspace(PyObject* o) {
    const at::Tensor& t = tensor(o);
    data = t.data_ptr();
    bytes = (size_t)t.numel();
  }
};

// A ctypes array of descriptors.
struct Descs {
  Py_buffer b;
  explicit Descs(PyObject* o) {
    if (PyObject_GetBuffer(o, &b, PyBUF_SIMPLE) != 0) throw Failed{};
  }
  Descs(const Descs&) = delete;
  ~Descs() { PyBuffer_Release(&b); }
  template <class T>
  const T* as(int32_t* count) const {
    *count = (int32_t)(b.len / (Py_ssize_t)sizeof(T));
    return static_cast<const T*>(b.buf);
  }
};

typedef PyObject* const* Args;

// quantize_act(x, ws, xq, act_scale, rowsum) -> (xq, act_scale, rowsum)
PyObject* quantize_act(Args a) {
  const at::Tensor& x = input(a[0], at::kFloat, "x: a contiguous fp32 CUDA tensor of two dimensions");
  need(x.dim() == 2, "x: a contiguous fp32 CUDA tensor of two dimensions");
  const int64_t M = x.size(0), K = x.size(1);
  const at::Device device = x.device();
  const float* const x_data = x.const_data_ptr<float>();
  const Workspace ws(a[1]);
  Out xq(a[2]), scale(a[3]), rowsum(a[4]);
  qb_status st;
  {
    const Unlocked unlocked;
    xq.make({M, K}, at::kChar, device);
    scale.make({1}, at::kFloat, device);
    rowsum.make({M}, at::kInt, device);
    st = qb_quantize_act(x_data, M, K, static_cast<int8_t*>(xq.data), static_cast<float*>(scale.data),
                         static_cast<int32_t*>(rowsum.data), ws.data, ws.bytes, stream());
  }
  check(st, "qb_quantize_act");
  return triple(xq, scale, rowsum);
}

// gemm(kind, xq, act_scale, rowsum, packed, delta, q0, bias, N, bits, groups, ws, y, acc_out | out_scale)
// kind 0: fp32 (last argument: int32 accumulators or None), 1: bfloat16 (None), 2: int8 (the output scale)
PyObject* gemm(Args a) {
  const int64_t kind = integer(a[0]);
  const at::Tensor& xq = input(a[1], at::kChar, "xq: a contiguous int8 CUDA tensor");
  need(xq.dim() == 2, "xq: two dimensions");
  const int64_t M = xq.size(0), K = xq.size(1), N = integer(a[8]);
  const at::Device device = xq.device();
  const int bits = (int)integer(a[9]), groups = (int)integer(a[10]);
  const Workspace ws(a[11]);
  if (kind == 1 && a[12] != Py_None)
    need(tensor(a[12]).scalar_type() == at::kBFloat16 && tensor(a[12]).is_contiguous(), "y: a contiguous bfloat16 tensor");
  if (kind == 2) need(tensor(a[13]).is_cuda() && tensor(a[13]).scalar_type() == at::kFloat, "out_scale: an fp32 CUDA tensor");
  Out y(a[12]);
  const int8_t* x = xq.const_data_ptr<int8_t>();
  const float* scale = static_cast<const float*>(ptr(a[2]));
  const int32_t* rowsum = static_cast<const int32_t*>(ptr(a[3]));
  const uint32_t* packed = static_cast<const uint32_t*>(ptr(a[4]));
  const float* delta = static_cast<const float*>(ptr(a[5]));
  const float* q0 = static_cast<const float*>(ptr(a[6]));
  const float* bias = static_cast<const float*>(ptr(a[7]));
  void* const last = ptr(a[13]);
  qb_status st;
  {
    const Unlocked unlocked;
    y.make({M, N}, kind == 0 ? at::kFloat : (kind == 1 ? at::kBFloat16 : at::kChar), device);
    if (kind == 0)
      st = qb_gemm(x, scale, rowsum, packed, delta, q0, bias, M, N, K, bits, groups, static_cast<float*>(y.data),
                   static_cast<int32_t*>(last), ws.data, ws.bytes, stream());
    else if (kind == 1)
      st = qb_gemm_bf16(x, scale, rowsum, packed, delta, q0, bias, M, N, K, bits, groups, static_cast<uint16_t*>(y.data),
                        ws.data, ws.bytes, stream());
    else
      st = qb_gemm_i8(x, scale, rowsum, packed, delta, q0, bias, M, N, K, bits, groups, static_cast<const float*>(last),
                      static_cast<int8_t*>(y.data), ws.data, ws.bytes, stream());
  }
  check(st, kind == 0 ? "qb_gemm" : (kind == 1 ? "qb_gemm_bf16" : "qb_gemm_i8"));
  return y.get();
}

// rowsum_i8(xq, rowsum) -> rowsum
PyObject* rowsum_i8(Args a) {
  const at::Tensor& xq = input(a[0], at::kChar, "xq: a contiguous int8 CUDA tensor of two dimensions");
  need(xq.dim() == 2, "xq: a contiguous int8 CUDA tensor of two dimensions");
  const int64_t M = xq.size(0), K = xq.size(1);
  const at::Device device = xq.device();
  const int8_t* const x = xq.const_data_ptr<int8_t>();
  Out rowsum(a[1]);
  qb_status st;
  {
    const Unlocked unlocked;
    rowsum.make({M}, at::kInt, device);
    st = qb_rowsum_i8(x, M, K, static_cast<int32_t*>(rowsum.data), stream());
  }
  check(st, "qb_rowsum_i8");
  return rowsum.get();
}

// quantize_pack_weights(w, bits, groups, ws, range_lo, range_hi, packed, delta, q0) -> (packed, delta, q0)
PyObject* quantize_pack_weights(Args a) {
  const at::Tensor& w = input(a[0], at::kFloat, "w: a contiguous fp32 CUDA tensor of two dimensions");
  need(w.dim() == 2, "w: a contiguous fp32 CUDA tensor of two dimensions");
  const int64_t N = w.size(0), K = w.size(1), bits = integer(a[1]), groups = integer(a[2]);
  const at::Device device = w.device();
  const float* const w_data = w.const_data_ptr<float>();
  const Workspace ws(a[3]);
  const float* const lo = static_cast<const float*>(ptr(a[4]));
  const float* const hi = static_cast<const float*>(ptr(a[5]));
  Out packed(a[6]), delta(a[7]), q0(a[8]);
  qb_status st;
  {
    const Unlocked unlocked;
    packed.make({N, std::max<int64_t>(1, K * bits / 32)}, at::kInt, device);
    delta.make({std::max<int64_t>(groups, 1)}, at::kFloat, device);
    q0.make({std::max<int64_t>(groups, 1)}, at::kFloat, device);
    st = qb_quantize_pack_weights(w_data, N, K, (int)bits, (int)groups, lo, hi, static_cast<uint32_t*>(packed.data),
                                  static_cast<float*>(delta.data), static_cast<float*>(q0.data), ws.data, ws.bytes, stream());
  }
  check(st, "qb_quantize_pack_weights");
  return triple(packed, delta, q0);
}

// fake_quantize_weights(w, bits, groups, ws, range_lo, range_hi, wq) -> (wq, delta, q0)
PyObject* fake_quantize_weights(Args a) {
  const at::Tensor& w = input(a[0], at::kFloat, "w: a contiguous fp32 CUDA tensor of two dimensions");
  need(w.dim() == 2, "w: a contiguous fp32 CUDA tensor of two dimensions");
  const int64_t N = w.size(0), K = w.size(1), bits = integer(a[1]), groups = integer(a[2]);
  const at::Device device = w.device();
  const float* const w_data = w.const_data_ptr<float>();
  const Workspace ws(a[3]);
  const float* const lo = static_cast<const float*>(ptr(a[4]));
  const float* const hi = static_cast<const float*>(ptr(a[5]));
  Out wq(a[6]), delta(Py_None), q0(Py_None);
  qb_status st;
  {
    const Unlocked unlocked;
    wq.make({N, K}, at::kFloat, device);
    delta.make({std::max<int64_t>(groups, 0)}, at::kFloat, device);
    q0.make({std::max<int64_t>(groups, 0)}, at::kFloat, device);
    st = qb_fake_quantize_weights(w_data, N, K, (int)bits, (int)groups, lo, hi, static_cast<float*>(wq.data),
                                  static_cast<float*>(delta.data), static_cast<float*>(q0.data), ws.data, ws.bytes, stream());
  }
  check(st, "qb_fake_quantize_weights");
  return triple(wq, delta, q0);
}

// ste_backward(grad_wq, w, groups, range_lo, range_hi, grad_w) -> grad_w
PyObject* ste_backward(Args a) {
  const at::Tensor& g = input(a[0], at::kFloat, "grad_wq: a contiguous fp32 CUDA tensor of the shape of w");
  const at::Tensor& w = tensor(a[1]);
  need(g.dim() == 2 && g.sizes() == w.sizes(), "grad_wq: a contiguous fp32 CUDA tensor of the shape of w");
  const int64_t N = w.size(0), K = w.size(1), groups = integer(a[2]);
  const at::Device device = w.device();
  const float* const g_data = g.const_data_ptr<float>();
  const float* const w_data = static_cast<const float*>(w.const_data_ptr());
  const float* const lo = static_cast<const float*>(ptr(a[3]));
  const float* const hi = static_cast<const float*>(ptr(a[4]));
  Out grad_w(a[5]);
  qb_status st;
  {
    const Unlocked unlocked;
    grad_w.make({N, K}, at::kFloat, device);
    st = qb_ste_backward(g_data, w_data, N, K, (int)groups, lo, hi, static_cast<float*>(grad_w.data), stream());
  }
  check(st, "qb_ste_backward");
  return grad_w.get();
}

// quantize_embedding(table, bits, groups, ws, packed) -> (packed, delta, q0)
PyObject* quantize_embedding(Args a) {
  const at::Tensor& t = input(a[0], at::kFloat, "table: a contiguous fp32 CUDA tensor of two dimensions");
  need(t.dim() == 2, "table: a contiguous fp32 CUDA tensor of two dimensions");
  const int64_t V = t.size(0), D = t.size(1), bits = integer(a[1]), groups = integer(a[2]);
  const at::Device device = t.device();
  const float* const table = t.const_data_ptr<float>();
  const Workspace ws(a[3]);
  Out packed(a[4]), delta(Py_None), q0(Py_None);
  qb_status st;
  {
    const Unlocked unlocked;
    packed.make({V, D * bits / 32}, at::kInt, device);
    delta.make({std::max<int64_t>(groups, 0)}, at::kFloat, device);
    q0.make({std::max<int64_t>(groups, 0)}, at::kFloat, device);
    st = qb_quantize_embedding(table, V, D, (int)bits, (int)groups, static_cast<uint32_t*>(packed.data),
                               static_cast<float*>(delta.data), static_cast<float*>(q0.data), ws.data, ws.bytes, stream());
  }
  check(st, "qb_quantize_embedding");
  return triple(packed, delta, q0);
}

// embedding_lookup(ids, packed, delta, q0, D, bits, groups, ws, out, accumulate) -> out
PyObject* embedding_lookup(Args a) {
  const at::Tensor& ids = input(a[0], at::kInt, "ids: a contiguous int32 CUDA tensor");
  const at::Tensor& packed = tensor(a[1]);
  const int64_t T = ids.numel(), V = packed.size(0), D = integer(a[4]), bits = integer(a[5]), groups = integer(a[6]);
  const at::Device device = ids.device();
  const int32_t* const id_data = ids.const_data_ptr<int32_t>();
  const uint32_t* const codes = static_cast<const uint32_t*>(packed.const_data_ptr());
  const float* const delta = static_cast<const float*>(ptr(a[2]));
  const float* const q0 = static_cast<const float*>(ptr(a[3]));
  const Workspace ws(a[7]);
  const int accumulate = PyObject_IsTrue(a[9]);
  if (accumulate < 0) throw Failed{};
  if (a[8] == Py_None) need(!accumulate, "accumulate needs `out`");
  Out out(a[8]);
  qb_status st;
  {
    const Unlocked unlocked;
    out.make({T, D}, at::kFloat, device);
    st = qb_embedding_lookup(id_data, T, codes, delta, q0, V, D, (int)bits, (int)groups, accumulate ? 1 : 0,
                             static_cast<float*>(out.data), ws.data, ws.bytes, stream());
  }
  check(st, "qb_embedding_lookup");
  return out.get();
}

// The calls over an array of descriptors: (array, ws)
template <class T, qb_status (*F)(const T*, int32_t, void*, size_t, void*)>
PyObject* over_descs(Args a, const char* what) {
  const Descs d(a[0]);
  const Workspace ws(a[1]);
  int32_t count = 0;
  const T* p = d.as<T>(&count);
  qb_status st;
  {
    const Unlocked unlocked;
    st = F(p, count, ws.data, ws.bytes, stream());
  }
  check(st, what);
  Py_RETURN_NONE;
}
PyObject* quantize_act_batch(Args a) { return over_descs<qb_act_desc, qb_quantize_act_batch>(a, "qb_quantize_act_batch"); }
PyObject* quantize_pack_weights_batch(Args a) {
  return over_descs<qb_weight_desc, qb_quantize_pack_weights_batch>(a, "qb_quantize_pack_weights_batch");
}
PyObject* fake_quantize_weights_batch(Args a) {
  return over_descs<qb_weight_desc, qb_fake_quantize_weights_batch>(a, "qb_fake_quantize_weights_batch");
}
PyObject* layer_linears(Args a) { return over_descs<qb_linear_desc, qb_layer_linears>(a, "qb_layer_linears"); }
PyObject* layer_linears_bf16(Args a) { return over_descs<qb_linear_desc, qb_layer_linears_bf16>(a, "qb_layer_linears_bf16"); }

PyObject* set_raise(Args a) {
  Py_XSETREF(g_raise, Py_NewRef(a[0]));
  Py_RETURN_NONE;
}

template <PyObject* (*F)(Args), int N>
PyObject* entry(PyObject*, PyObject* const* args, Py_ssize_t n) {
  if (n != N) {
    PyErr_Format(PyExc_TypeError, "expected %d arguments, got %zd", N, n);
    return nullptr;
  }
  HANDLE_TH_ERRORS  // what torch throws (out of memory, no device) becomes the exception torch raises for it
  try {
    return F(args);
  } catch (const Failed&) {
    return nullptr;
  }
  END_HANDLE_TH_ERRORS
}
#define QB_ENTRY(f, n) {#f, (PyCFunction)(void (*)(void))entry<f, n>, METH_FASTCALL, nullptr}
PyMethodDef g_methods[] = {QB_ENTRY(quantize_act, 5),
                           QB_ENTRY(gemm, 14),
                           QB_ENTRY(rowsum_i8, 2),
                           QB_ENTRY(quantize_pack_weights, 9),
                           QB_ENTRY(fake_quantize_weights, 7),
                           QB_ENTRY(ste_backward, 6),
                           QB_ENTRY(quantize_embedding, 5),
                           QB_ENTRY(embedding_lookup, 10),
                           QB_ENTRY(quantize_act_batch, 2),
                           QB_ENTRY(quantize_pack_weights_batch, 2),
                           QB_ENTRY(fake_quantize_weights_batch, 2),
                           QB_ENTRY(layer_linears, 2),
                           QB_ENTRY(layer_linears_bf16, 2),
                           QB_ENTRY(set_raise, 1),
                           {nullptr, nullptr, 0, nullptr}};
PyModuleDef g_module = {PyModuleDef_HEAD_INIT, "_qbert", nullptr, -1, g_methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__qbert(void) { return PyModule_Create(&g_module); }
