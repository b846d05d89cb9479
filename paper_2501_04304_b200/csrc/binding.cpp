// Native half of binding.py: the hot-path calls of libdgq with their output and workspace allocations, as
// positional CPython functions.  A layer pass is two library calls, five allocations and two or three kernel
// launches; marshalling them through ctypes and torch.empty took 38 us of host time (256 x 320 x 320, static
// tables), more than the kernels of every small layer.  Keyword handling, defaults and the meaning of
// every argument live in binding.py.
#include <Python.h>

#include <ATen/cuda/EmptyTensor.h>
#include <c10/cuda/CUDAGuard.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/dgq.h"

namespace {

at::Tensor empty(std::initializer_list<int64_t> shape, at::ScalarType type, const at::Tensor& like) {
  return at::Tensor(at::detail::empty_cuda(at::IntArrayRef(shape.begin(), shape.size()), type, like.device(), std::nullopt));
}

// Scratch memory for a call on stream `st` that is dropped when the call returns: it belongs to that stream, so that torch
// gives it to nobody else before the call's kernels have run.  `given` is the stream argument (None: the current
// stream, to which torch's allocations belong anyway).
at::Tensor scratch(int64_t bytes, const at::Tensor& like, PyObject* given, void* st) {
  if (given == Py_None) return empty({bytes}, at::kByte, like);
  c10::cuda::CUDAStreamGuard on(c10::cuda::getStreamFromExternal(static_cast<cudaStream_t>(st), like.device().index()));
  return empty({bytes}, at::kByte, like);
}

// A tensor argument, or an undefined tensor for None.  Sets a TypeError for anything else.
bool tensor(PyObject* o, at::Tensor* t) {
  if (o == Py_None) return true;
  if (!THPVariable_Check(o)) {
    PyErr_Format(PyExc_TypeError, "expected a tensor or None, got %s", Py_TYPE(o)->tp_name);
    return false;
  }
  *t = THPVariable_Unpack(o);
  return true;
}

template <typename T = void>
T* ptr(const at::Tensor& t) { return t.defined() ? static_cast<T*>(t.data_ptr()) : nullptr; }

PyObject* wrap(const at::Tensor& t) {
  if (!t.defined()) Py_RETURN_NONE;
  return THPVariable_Wrap(t);
}

bool integer(PyObject* o, int* v) {
  const long x = PyLong_AsLong(o);
  if (x == -1 && PyErr_Occurred()) return false;
  *v = static_cast<int>(x);
  return true;
}

// The argument of a stream parameter: None (the current stream) or an object with a `cuda_stream` handle.
bool stream_arg(PyObject* o, void** s) {
  if (o == Py_None) {
    *s = c10::cuda::getCurrentCUDAStream().stream();
    return true;
  }
  static PyObject* name = PyUnicode_InternFromString("cuda_stream");
  PyObject* v = PyObject_GetAttr(o, name);
  if (!v) return false;
  *s = PyLong_AsVoidPtr(v);
  Py_DECREF(v);
  return !PyErr_Occurred();
}

bool handle(PyObject* o, void** h) {
  *h = PyLong_AsVoidPtr(o);
  return !PyErr_Occurred();
}

// binding.py raises DgqError from a status returned in place of a result.
PyObject* status(dgq_status st) { return PyLong_FromLong(st); }

// A function of the module: what torch's C++ API throws (no CUDA device, a tensor without storage, a dimension that
// is not there) becomes a Python exception.  For that everything that may throw, taking a tensor's address included,
// runs with the GIL held: between Py_BEGIN_ALLOW_THREADS and its end stands nothing but the library call.
template <PyObject* (*BODY)(PyObject* const*, Py_ssize_t)>
PyObject* entry(PyObject*, PyObject* const* a, Py_ssize_t n) {
  try {
    return BODY(a, n);
  } catch (python_error& e) {
    e.restore();
  } catch (const std::exception& e) {
    PyErr_SetString(PyExc_RuntimeError, e.what());
  }
  return nullptr;
}

// A tuple of the objects, whose references it takes over; null if one of them is.
PyObject* tuple(std::initializer_list<PyObject*> items) {
  PyObject* r = PyTuple_New(static_cast<Py_ssize_t>(items.size()));
  bool ok = r != nullptr;
  Py_ssize_t i = 0;
  for (PyObject* o : items) {
    ok = ok && o;
    if (r) PyTuple_SET_ITEM(r, i++, o);
    else Py_XDECREF(o);
  }
  if (!ok) Py_CLEAR(r);
  return r;
}

// An output: the caller's buffer as the object it is, or the tensor made for it.
PyObject* output(PyObject* given, const at::Tensor& t) { return given == Py_None ? wrap(t) : Py_NewRef(given); }

bool require(bool ok, const char* what) {
  if (!ok) PyErr_SetString(PyExc_AssertionError, what);
  return ok;
}

bool arity(Py_ssize_t n, Py_ssize_t want) {
  if (n == want) return true;
  PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, n);
  return false;
}

// (groups, K_pad, G, timestep, mode, layout, X, out | None, scale | None, zp | None, allocate, stream) -> (Xq, scale, zp)
PyObject* quantize_act(PyObject* const* a, Py_ssize_t n) {
  void *g, *st;
  int k_pad, n_groups, timestep, mode, layout, allocate;
  at::Tensor x, out, scale, zp;
  if (!arity(n, 12) || !handle(a[0], &g) || !integer(a[1], &k_pad) || !integer(a[2], &n_groups) ||
      !integer(a[3], &timestep) || !integer(a[4], &mode) || !integer(a[5], &layout) || !tensor(a[6], &x) ||
      !tensor(a[7], &out) || !tensor(a[8], &scale) || !tensor(a[9], &zp) || !integer(a[10], &allocate) ||
      !stream_arg(a[11], &st))
    return nullptr;
  if (!require(x.defined() && x.is_cuda() && x.scalar_type() == at::kHalf && x.dim() == 2 && x.stride(1) == 1,
               "X is a CUDA fp16 matrix with contiguous rows"))
    return nullptr;
  const int64_t m = x.size(0);
  if (allocate) {
    if (!out.defined()) out = empty({m, k_pad}, at::kByte, x);
    if (mode == DGQ_MODE_DYNAMIC_TOKEN) {
      scale = empty({m, n_groups}, at::kFloat, x);
      zp = empty({m, n_groups}, at::kInt, x);
    }
  }
  const int64_t ld = x.stride(0);
  void *p_x = ptr(x), *p_out = ptr(out);
  float* p_scale = ptr<float>(scale);
  int32_t* p_zp = ptr<int32_t>(zp);
  dgq_status rc;
  Py_BEGIN_ALLOW_THREADS
  rc = dgq_quantize_act(static_cast<const dgq_groups*>(g), timestep, mode, layout, p_x, m, ld, p_out, p_scale, p_zp, st);
  Py_END_ALLOW_THREADS
  if (rc != DGQ_OK) return status(rc);
  return tuple({output(a[7], out), wrap(scale), wrap(zp)});
}

// (groups, weight, N, timestep, mode, layout, Xq, scale, zp, bias, out | None, conv | None, workspace, stream) -> Y
// workspace: a tensor, None (one of the size the library asks for) or False (none).
PyObject* linear(PyObject* const* a, Py_ssize_t n) {
  void *g, *w, *st;
  int n_out, timestep, mode, layout;
  at::Tensor xq, scale, zp, bias, y, ws;
  if (!arity(n, 14) || !handle(a[0], &g) || !handle(a[1], &w) || !integer(a[2], &n_out) || !integer(a[3], &timestep) ||
      !integer(a[4], &mode) || !integer(a[5], &layout) || !tensor(a[6], &xq) || !tensor(a[7], &scale) ||
      !tensor(a[8], &zp) || !tensor(a[9], &bias) || !tensor(a[10], &y) ||
      (a[12] != Py_False && !tensor(a[12], &ws)) || !stream_arg(a[13], &st))
    return nullptr;
  dgq_conv_desc conv;
  if (a[11] != Py_None) {
    PyObject* t = PySequence_Tuple(a[11]);
    if (!t) return nullptr;
    const bool ok = PyArg_ParseTuple(t, "iiii", &conv.n, &conv.h, &conv.w, &conv.c);
    Py_DECREF(t);
    if (!ok) return nullptr;
  }
  if (!require(xq.defined() && xq.dim() >= 1, "Xq is a matrix of codes")) return nullptr;
  const int64_t m = xq.size(0);
  if (!y.defined()) y = empty({m, n_out}, at::kHalf, xq);
  dgq_status rc = DGQ_OK;
  if (a[12] == Py_None) {
    size_t need = 0;
    rc = dgq_linear_workspace_bytes(static_cast<const dgq_groups*>(g), static_cast<const dgq_weight*>(w), m, &need);
    if (rc != DGQ_OK) return status(rc);
    if (need) ws = scratch(static_cast<int64_t>(need), xq, a[13], st);
  }
  const int64_t ldy = y.stride(0);
  const size_t ws_bytes = ws.defined() ? static_cast<size_t>(ws.numel()) : 0;
  void *p_xq = ptr(xq), *p_bias = ptr(bias), *p_y = ptr(y), *p_ws = ptr(ws);
  float* p_scale = ptr<float>(scale);
  int32_t* p_zp = ptr<int32_t>(zp);
  Py_BEGIN_ALLOW_THREADS
  rc = dgq_linear(static_cast<const dgq_groups*>(g), static_cast<const dgq_weight*>(w), timestep, mode, layout, p_xq, p_scale,
                  p_zp, p_bias, p_y, m, ldy, a[11] != Py_None ? &conv : nullptr, p_ws, ws_bytes, st);
  Py_END_ALLOW_THREADS
  if (rc != DGQ_OK) return status(rc);
  return output(a[10], y);
}

// (Q, K, V, score_bits, scale_gran, fixed_scale, out | None, want_scale, want_codes, workspace | None, v_bits, stream)
// -> (O, scale, codes)
PyObject* cross_attn_logq(PyObject* const* a, Py_ssize_t n) {
  void* st;
  int bits, gran, want_scale, want_codes, v_bits;
  at::Tensor q, k, v, fixed, o, scale, codes, ws;
  if (!arity(n, 12) || !tensor(a[0], &q) || !tensor(a[1], &k) || !tensor(a[2], &v) || !integer(a[3], &bits) ||
      !integer(a[4], &gran) || !tensor(a[5], &fixed) || !tensor(a[6], &o) || !integer(a[7], &want_scale) ||
      !integer(a[8], &want_codes) || !tensor(a[9], &ws) || !integer(a[10], &v_bits) || !stream_arg(a[11], &st))
    return nullptr;
  if (!require(q.defined() && k.defined() && v.defined() && q.dim() == 4 && q.is_contiguous() && k.is_contiguous() &&
                   v.is_contiguous(),
               "Q, K and V are contiguous [B, n, H, d] tensors"))
    return nullptr;
  const int64_t B = q.size(0), nq = q.size(1), H = q.size(2), d = q.size(3), nk = k.size(1);
  if (!o.defined()) o = empty({B, nq, H, d}, q.scalar_type(), q);
  if (want_scale) {
    const int64_t scopes = gran == DGQ_SCALE_PER_PROMPT ? B : gran == DGQ_SCALE_PER_PROMPT_HEAD ? B * H : 1;
    scale = empty({scopes}, at::kFloat, q);
  }
  if (want_codes) codes = empty({B, H, nq, nk - 1}, at::kByte, q);
  if (!ws.defined()) {
    size_t need = 256;
    if (nk >= 2) {
      const dgq_status rc = dgq_cross_attn_workspace_bytes(B, H, nq, nk, d, &need);
      if (rc != DGQ_OK) return status(rc);
    }
    ws = scratch(static_cast<int64_t>(need), q, a[11], st);
  }
  void *p_q = ptr(q), *p_k = ptr(k), *p_v = ptr(v), *p_o = ptr(o), *p_ws = ptr(ws);
  float *p_fixed = ptr<float>(fixed), *p_scale = ptr<float>(scale);
  uint8_t* p_codes = ptr<uint8_t>(codes);
  const size_t ws_bytes = ws.numel();
  dgq_status rc;
  Py_BEGIN_ALLOW_THREADS
  if (v_bits)
    rc = dgq_cross_attn_logq_qv(p_q, p_k, p_v, B, H, nq, nk, d, bits, gran, p_fixed, v_bits, p_o, p_scale, p_codes, p_ws, ws_bytes, st);
  else
    rc = dgq_cross_attn_logq(p_q, p_k, p_v, B, H, nq, nk, d, bits, gran, p_fixed, p_o, p_scale, p_codes, p_ws, ws_bytes, st);
  Py_END_ALLOW_THREADS
  if (rc != DGQ_OK) return status(rc);
  return tuple({output(a[6], o), wrap(scale), wrap(codes)});
}

// (Q, K, V, score_bits, fixed_scale, out | None, want_codes, stream) -> (O, codes)
PyObject* self_attn_logq(PyObject* const* a, Py_ssize_t n) {
  void* st;
  int bits, want_codes;
  at::Tensor q, k, v, fixed, o, codes;
  if (!arity(n, 8) || !tensor(a[0], &q) || !tensor(a[1], &k) || !tensor(a[2], &v) || !integer(a[3], &bits) ||
      !tensor(a[4], &fixed) || !tensor(a[5], &o) || !integer(a[6], &want_codes) || !stream_arg(a[7], &st))
    return nullptr;
  if (!require(q.defined() && k.defined() && v.defined() && q.dim() == 4 && q.is_contiguous() && k.is_contiguous() &&
                   v.is_contiguous(),
               "Q, K and V are contiguous [B, n, H, d] tensors"))
    return nullptr;
  const int64_t B = q.size(0), nq = q.size(1), H = q.size(2), d = q.size(3), nk = k.size(1);
  if (!o.defined()) o = empty({B, nq, H, d}, q.scalar_type(), q);
  if (want_codes) codes = empty({B, H, nq, nk}, at::kByte, q);
  void *p_q = ptr(q), *p_k = ptr(k), *p_v = ptr(v), *p_o = ptr(o);
  float* p_fixed = ptr<float>(fixed);
  uint8_t* p_codes = ptr<uint8_t>(codes);
  dgq_status rc;
  Py_BEGIN_ALLOW_THREADS
  rc = dgq_self_attn_logq(p_q, p_k, p_v, B, H, nq, nk, d, bits, p_fixed, p_o, p_codes, st);
  Py_END_ALLOW_THREADS
  if (rc != DGQ_OK) return status(rc);
  return tuple({output(a[5], o), wrap(codes)});
}

template <PyObject* (*BODY)(PyObject* const*, Py_ssize_t)>
PyMethodDef method(const char* name) {
  return {name, reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(entry<BODY>)), METH_FASTCALL, nullptr};
}
PyMethodDef methods[] = {method<quantize_act>("quantize_act"), method<linear>("linear"),
                         method<cross_attn_logq>("cross_attn_logq"), method<self_attn_logq>("self_attn_logq"),
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native() { return PyModule_Create(&module); }
