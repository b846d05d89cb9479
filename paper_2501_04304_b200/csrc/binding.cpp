// Native half of binding.py: the hot-path calls of libdgq with their output and workspace allocations, as
// positional CPython functions.  A layer pass is two library calls, five allocations and two or three kernel
// launches; marshalling them through ctypes and torch.empty took 38 us of host time (256 x 320 x 320, static
// tables), more than the kernels of every small layer.  Keyword handling, defaults and the meaning of
// every argument live in binding.py.
#include <Python.h>

#include <ATen/cuda/EmptyTensor.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/dgq.h"

namespace {

at::Tensor empty(std::initializer_list<int64_t> shape, at::ScalarType type, const at::Tensor& like) {
  return at::Tensor(at::detail::empty_cuda(at::IntArrayRef(shape.begin(), shape.size()), type, like.device(), std::nullopt));
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

PyObject* guard_error(const std::exception& e) {
  PyErr_SetString(PyExc_RuntimeError, e.what());
  return nullptr;
}

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
PyObject* quantize_act(PyObject*, PyObject* const* a, Py_ssize_t n) {
  void *g, *st;
  int k_pad, n_groups, timestep, mode, layout, allocate;
  at::Tensor x, out, scale, zp;
  if (!arity(n, 12) || !handle(a[0], &g) || !integer(a[1], &k_pad) || !integer(a[2], &n_groups) ||
      !integer(a[3], &timestep) || !integer(a[4], &mode) || !integer(a[5], &layout) || !tensor(a[6], &x) ||
      !tensor(a[7], &out) || !tensor(a[8], &scale) || !tensor(a[9], &zp) || !integer(a[10], &allocate) ||
      !stream_arg(a[11], &st))
    return nullptr;
  try {
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
    dgq_status rc;
    Py_BEGIN_ALLOW_THREADS
    rc = dgq_quantize_act(static_cast<const dgq_groups*>(g), timestep, mode, layout, ptr(x), m, x.stride(0), ptr(out),
                          ptr<float>(scale), ptr<int32_t>(zp), st);
    Py_END_ALLOW_THREADS
    if (rc != DGQ_OK) return status(rc);
    PyObject* r = PyTuple_New(3);
    if (!r) return nullptr;
    // an output buffer of the caller's is handed back as the object it is
    PyTuple_SET_ITEM(r, 0, a[7] == Py_None ? wrap(out) : Py_NewRef(a[7]));
    PyTuple_SET_ITEM(r, 1, wrap(scale));
    PyTuple_SET_ITEM(r, 2, wrap(zp));
    return r;
  } catch (const std::exception& e) {
    return guard_error(e);
  }
}

// (groups, weight, N, timestep, mode, layout, Xq, scale, zp, bias, out | None, conv | None, workspace, stream) -> Y
// workspace: a tensor, None (one of the size the library asks for) or False (none).
PyObject* linear(PyObject*, PyObject* const* a, Py_ssize_t n) {
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
  try {
    if (!require(xq.defined() && xq.dim() >= 1, "Xq is a matrix of codes")) return nullptr;
    const int64_t m = xq.size(0);
    if (!y.defined()) y = empty({m, n_out}, at::kHalf, xq);
    dgq_status rc = DGQ_OK;
    if (a[12] == Py_None) {
      size_t need = 0;
      rc = dgq_linear_workspace_bytes(static_cast<const dgq_groups*>(g), static_cast<const dgq_weight*>(w), m, &need);
      if (rc != DGQ_OK) return status(rc);
      if (need) ws = empty({static_cast<int64_t>(need)}, at::kByte, xq);
    }
    Py_BEGIN_ALLOW_THREADS
    rc = dgq_linear(static_cast<const dgq_groups*>(g), static_cast<const dgq_weight*>(w), timestep, mode, layout, ptr(xq),
                    ptr<float>(scale), ptr<int32_t>(zp), ptr(bias), ptr(y), m, y.stride(0),
                    a[11] != Py_None ? &conv : nullptr, ptr(ws), ws.defined() ? static_cast<size_t>(ws.numel()) : 0, st);
    Py_END_ALLOW_THREADS
    if (rc != DGQ_OK) return status(rc);
    return a[10] == Py_None ? wrap(y) : Py_NewRef(a[10]);
  } catch (const std::exception& e) {
    return guard_error(e);
  }
}

// (Q, K, V, score_bits, scale_gran, fixed_scale, out | None, want_scale, want_codes, workspace | None, v_bits, stream)
// -> (O, scale, codes)
PyObject* cross_attn_logq(PyObject*, PyObject* const* a, Py_ssize_t n) {
  void* st;
  int bits, gran, want_scale, want_codes, v_bits;
  at::Tensor q, k, v, fixed, o, scale, codes, ws;
  if (!arity(n, 12) || !tensor(a[0], &q) || !tensor(a[1], &k) || !tensor(a[2], &v) || !integer(a[3], &bits) ||
      !integer(a[4], &gran) || !tensor(a[5], &fixed) || !tensor(a[6], &o) || !integer(a[7], &want_scale) ||
      !integer(a[8], &want_codes) || !tensor(a[9], &ws) || !integer(a[10], &v_bits) || !stream_arg(a[11], &st))
    return nullptr;
  try {
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
      ws = empty({static_cast<int64_t>(need)}, at::kByte, q);
    }
    dgq_status rc;
    Py_BEGIN_ALLOW_THREADS
    if (v_bits)
      rc = dgq_cross_attn_logq_qv(ptr(q), ptr(k), ptr(v), B, H, nq, nk, d, bits, gran, ptr<float>(fixed), v_bits, ptr(o),
                                  ptr<float>(scale), ptr<uint8_t>(codes), ptr(ws), ws.numel(), st);
    else
      rc = dgq_cross_attn_logq(ptr(q), ptr(k), ptr(v), B, H, nq, nk, d, bits, gran, ptr<float>(fixed), ptr(o),
                               ptr<float>(scale), ptr<uint8_t>(codes), ptr(ws), ws.numel(), st);
    Py_END_ALLOW_THREADS
    if (rc != DGQ_OK) return status(rc);
    PyObject* r = PyTuple_New(3);
    if (!r) return nullptr;
    PyTuple_SET_ITEM(r, 0, a[6] == Py_None ? wrap(o) : Py_NewRef(a[6]));
    PyTuple_SET_ITEM(r, 1, wrap(scale));
    PyTuple_SET_ITEM(r, 2, wrap(codes));
    return r;
  } catch (const std::exception& e) {
    return guard_error(e);
  }
}

// (Q, K, V, score_bits, fixed_scale, out | None, want_codes, stream) -> (O, codes)
PyObject* self_attn_logq(PyObject*, PyObject* const* a, Py_ssize_t n) {
  void* st;
  int bits, want_codes;
  at::Tensor q, k, v, fixed, o, codes;
  if (!arity(n, 8) || !tensor(a[0], &q) || !tensor(a[1], &k) || !tensor(a[2], &v) || !integer(a[3], &bits) ||
      !tensor(a[4], &fixed) || !tensor(a[5], &o) || !integer(a[6], &want_codes) || !stream_arg(a[7], &st))
    return nullptr;
  try {
    if (!require(q.defined() && k.defined() && v.defined() && q.dim() == 4 && q.is_contiguous() && k.is_contiguous() &&
                     v.is_contiguous(),
                 "Q, K and V are contiguous [B, n, H, d] tensors"))
      return nullptr;
    const int64_t B = q.size(0), nq = q.size(1), H = q.size(2), d = q.size(3), nk = k.size(1);
    if (!o.defined()) o = empty({B, nq, H, d}, q.scalar_type(), q);
    if (want_codes) codes = empty({B, H, nq, nk}, at::kByte, q);
    dgq_status rc;
    Py_BEGIN_ALLOW_THREADS
    rc = dgq_self_attn_logq(ptr(q), ptr(k), ptr(v), B, H, nq, nk, d, bits, ptr<float>(fixed), ptr(o), ptr<uint8_t>(codes), st);
    Py_END_ALLOW_THREADS
    if (rc != DGQ_OK) return status(rc);
    PyObject* r = PyTuple_New(2);
    if (!r) return nullptr;
    PyTuple_SET_ITEM(r, 0, a[5] == Py_None ? wrap(o) : Py_NewRef(a[5]));
    PyTuple_SET_ITEM(r, 1, wrap(codes));
    return r;
  } catch (const std::exception& e) {
    return guard_error(e);
  }
}

PyMethodDef methods[] = {
    {"quantize_act", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(quantize_act)), METH_FASTCALL, nullptr},
    {"linear", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(linear)), METH_FASTCALL, nullptr},
    {"cross_attn_logq", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(cross_attn_logq)), METH_FASTCALL, nullptr},
    {"self_attn_logq", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(self_attn_logq)), METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native() { return PyModule_Create(&module); }
