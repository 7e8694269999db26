// The dense calls of binding.py as one native step: check the tensors, allocate outputs and workspace, call the library.
//
// A call returns None wherever anything is out of the ordinary (another type, shape, layout or device than the kernels take,
// tensor subclasses, active function or dispatch modes, an argument that is not a plain number); binding.py then goes its own
// way, with its own checks and messages.  It returns a status code where the library refuses the call.
// What for: the smallest steps are bound by the host.  Forward and backward of 2 heads x 256 x 64 took 31.2 us of host time in
// Python and ctypes and take 16.9 here (three launches, eleven tensor maps, six allocations), 20.3 with the GPU's share.
#include <Python.h>

#include "gproj_attn.h"

#include <ATen/ATen.h>
#include <ATen/PythonTorchFunctionTLS.h>
#include <c10/core/impl/TorchDispatchModeTLS.h>
#include <c10/cuda/CUDAFunctions.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <algorithm>
#include <cstddef>

namespace {

// In the library that binding.py loaded; its types are the header's, so a signature that changes there does not compile here.
decltype(&gproj_attn_fwd_rect) fwd_fn = nullptr;
decltype(&gproj_attn_bwd_rect) bwd_fn = nullptr;
decltype(&gproj_attn_bwd_workspace_bytes) bytes_fn = nullptr;

struct Unusual {};            // leave the call to binding.py

const at::Tensor &tensor(PyObject *o, at::ScalarType type, int64_t dims) {
  if (!THPVariable_CheckExact(o)) throw Unusual{};
  const at::Tensor &t = THPVariable_Unpack(o);
  if (!t.is_cuda() || t.scalar_type() != type || t.dim() != dims || !t.is_contiguous()) throw Unusual{};
  return t;
}

struct Sizes { int B, H, Hkv, Nq, Nk, d; };
Sizes sizes_of(const at::Tensor &Q, const at::Tensor &K, const at::Tensor &V, bool square) {
  const auto q = Q.sizes(), k = K.sizes();
  for (int64_t n : q) if (n < 0 || n > INT32_MAX) throw Unusual{};
  if (V.sizes() != k || k[0] != q[0] || k[3] != q[3] || k[1] <= 0 || q[1] % k[1] != 0 || k[2] > INT32_MAX || (square && k[2] != q[2])) throw Unusual{};
  return Sizes{static_cast<int>(q[0]), static_cast<int>(q[1]), static_cast<int>(k[1]), static_cast<int>(q[2]), static_cast<int>(k[2]), static_cast<int>(q[3])};
}

struct Options { float scale; int causal; unsigned flags; };
Options options_of(PyObject *scale, PyObject *causal, PyObject *flags) {
  if (!PyFloat_CheckExact(scale) || !PyBool_Check(causal) || !PyLong_CheckExact(flags)) throw Unusual{};
  const long f = PyLong_AsLong(flags);
  if (f < 0 || f > INT32_MAX) { PyErr_Clear(); throw Unusual{}; }
  return Options{static_cast<float>(PyFloat_AS_DOUBLE(scale)), causal == Py_True, static_cast<unsigned>(f)};
}

// The device of the call, current and the same for all tensors, and its current stream.
template <typename... Ts>
void *stream_on(const at::Tensor &first, const Ts &...others) {
  const auto index = first.device().index();
  if (index != c10::cuda::current_device() || ((others.device().index() != index) || ...)) throw Unusual{};
  if (at::impl::torch_function_mode_enabled() || c10::impl::TorchDispatchModeTLS::any_modes_set()) throw Unusual{};
  return c10::cuda::getCurrentCUDAStream(index).stream();
}

PyObject *tuple_of(std::initializer_list<at::Tensor> ts) {
  PyObject *out = PyTuple_New(static_cast<Py_ssize_t>(ts.size()));
  if (out == nullptr) return nullptr;
  Py_ssize_t i = 0;
  for (const at::Tensor &t : ts) {
    PyObject *o = THPVariable_Wrap(t);
    if (o == nullptr) { Py_DECREF(out); return nullptr; }
    PyTuple_SET_ITEM(out, i++, o);
  }
  return out;
}

// Other Python threads may run while this lives; it ends by an exception as well.
struct NoGil {
  PyThreadState *state = PyEval_SaveThread();
  ~NoGil() { PyEval_RestoreThread(state); }
};

template <typename Body>
PyObject *guarded(Body body) {
  try {
    return body();
  } catch (...) {             // binding.py meets the same condition and reports it
    PyErr_Clear();
    Py_RETURN_NONE;
  }
}

// (Q, K, V, softmax_scale, causal, fwd_flags, square) -> (O, LSE)
PyObject *fwd(PyObject *, PyObject *const *a, Py_ssize_t n) {
  return guarded([&]() -> PyObject * {
    if (n != 7 || fwd_fn == nullptr) throw Unusual{};
    const at::Tensor &Q = tensor(a[0], at::kBFloat16, 4), &K = tensor(a[1], at::kBFloat16, 4), &V = tensor(a[2], at::kBFloat16, 4);
    const Sizes s = sizes_of(Q, K, V, a[6] == Py_True);
    const Options o = options_of(a[3], a[4], a[5]);
    void *stream = stream_on(Q, K, V);
    const void *q = Q.const_data_ptr(), *k = K.const_data_ptr(), *v = V.const_data_ptr();
    at::Tensor O = at::empty_like(Q), LSE = at::empty({s.B, s.H, s.Nq}, Q.options().dtype(at::kFloat));
    void *out = O.mutable_data_ptr();
    float *lse = static_cast<float *>(LSE.mutable_data_ptr());
    const int rc = [&] { const NoGil free; return fwd_fn(q, k, v, out, lse, s.B, s.H, s.Hkv, s.Nq, s.Nk, s.d, o.scale, o.causal, o.flags, stream); }();
    return rc == 0 ? tuple_of({O, LSE}) : PyLong_FromLong(rc);
  });
}

// (Q, K, V, O, LSE, dO, softmax_scale, causal, flags, square) -> (dQ, dK, dV)
PyObject *bwd(PyObject *, PyObject *const *a, Py_ssize_t n) {
  return guarded([&]() -> PyObject * {
    if (n != 10 || bwd_fn == nullptr) throw Unusual{};
    const at::Tensor &Q = tensor(a[0], at::kBFloat16, 4), &K = tensor(a[1], at::kBFloat16, 4), &V = tensor(a[2], at::kBFloat16, 4);
    const at::Tensor &O = tensor(a[3], at::kBFloat16, 4), &LSE = tensor(a[4], at::kFloat, 3), &dO = tensor(a[5], at::kBFloat16, 4);
    const Sizes s = sizes_of(Q, K, V, a[9] == Py_True);
    if (O.sizes() != Q.sizes() || dO.sizes() != Q.sizes() || LSE.size(0) != s.B || LSE.size(1) != s.H || LSE.size(2) != s.Nq) throw Unusual{};
    const Options o = options_of(a[6], a[7], a[8]);
    void *stream = stream_on(Q, K, V, O, LSE, dO);
    const void *q = Q.const_data_ptr(), *k = K.const_data_ptr(), *v = V.const_data_ptr(), *out = O.const_data_ptr(), *u = dO.const_data_ptr();
    const float *lse = static_cast<const float *>(LSE.const_data_ptr());
    const size_t bytes = std::max<size_t>(bytes_fn(s.B, s.H, s.Nq, s.d), 256);
    at::Tensor ws = at::empty({static_cast<int64_t>(bytes)}, Q.options().dtype(at::kByte));
    at::Tensor dQ = at::empty_like(Q), dK = at::empty_like(K), dV = at::empty_like(V);
    void *pq = dQ.mutable_data_ptr(), *pk = dK.mutable_data_ptr(), *pv = dV.mutable_data_ptr(), *pw = ws.mutable_data_ptr();
    const int rc = [&] { const NoGil free; return bwd_fn(q, k, v, out, lse, u, pq, pk, pv, s.B, s.H, s.Hkv, s.Nq, s.Nk, s.d, o.scale, o.causal, pw, bytes, o.flags, stream); }();
    return rc == 0 ? tuple_of({dQ, dK, dV}) : PyLong_FromLong(rc);
  });
}

// Addresses of gproj_attn_fwd_rect, gproj_attn_bwd_rect and gproj_attn_bwd_workspace_bytes in the loaded library.
PyObject *bind(PyObject *, PyObject *args) {
  unsigned long long f, b, w;
  if (!PyArg_ParseTuple(args, "KKK", &f, &b, &w)) return nullptr;
  fwd_fn = reinterpret_cast<decltype(fwd_fn)>(f);
  bwd_fn = reinterpret_cast<decltype(bwd_fn)>(b);
  bytes_fn = reinterpret_cast<decltype(bytes_fn)>(w);
  Py_RETURN_NONE;
}

PyMethodDef methods[] = {
    {"fwd", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(fwd)), METH_FASTCALL, nullptr},
    {"bwd", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(bwd)), METH_FASTCALL, nullptr},
    {"bind", bind, METH_VARARGS, nullptr},
    {nullptr, nullptr, 0, nullptr},
};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_torch_calls", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__torch_calls() { return PyModule_Create(&module); }
