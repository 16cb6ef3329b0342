// Python entry points of the C ABI for torch tensors: argument marshalling only, in C++ because it is on the path of
// every call. A small layer's two kernels take about 8 us on the device; marshalled in Python (ctypes, one wrapper object
// per pointer, torch.cuda.current_stream()) a call took 13-18 us of host time, so the host set the pace of every layer
// below some 15 us. Each function takes exactly the positional arguments its wrapper in binding.py passes, checks that
// tensors are contiguous CUDA tensors, and returns the sdgp_status as an int.
#include <ATen/PythonTorchFunctionTLS.h>
#include <ATen/TensorSubclassLikeUtils.h>
#include <Python.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>
#include <torch/csrc/jit/frontend/tracer.h>

#include "../../include/sdgp.h"
#include "torch_autograd.h"

namespace {

// Reads positional arguments in order; after the first failure (a Python exception is set) every read returns zero.
struct Args {
  PyObject* const* a;
  Py_ssize_t left;
  bool ok = true;

  Args(PyObject* const* args, Py_ssize_t n, Py_ssize_t want) : a(args), left(n) {
    if (n != want) {
      PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, n);
      ok = false;
    }
  }
  int64_t i64() {
    if (!ok) return 0;
    const long long v = PyLong_AsLongLong(*a++);
    if (v == -1 && PyErr_Occurred()) ok = false;
    return v;
  }
  int i32() {
    const int64_t v = i64();
    if (ok && (v > INT32_MAX || v < INT32_MIN)) {
      PyErr_SetString(PyExc_OverflowError, "integer argument does not fit 32 bits");
      ok = false;
    }
    return (int)v;
  }
  uint64_t u64() {  // seeds: any Python int, modulo 2^64
    if (!ok) return 0;
    PyObject* o = *a++;
    const unsigned long long v = PyLong_AsUnsignedLongLongMask(o);
    if (v == (unsigned long long)-1 && PyErr_Occurred()) ok = false;
    return v;
  }
  // A contiguous CUDA tensor, or nullptr for None.
  const at::Tensor* tensor(const char* name) {
    if (!ok) return nullptr;
    PyObject* o = *a++;
    if (o == Py_None) return nullptr;
    if (!THPVariable_Check(o)) {
      PyErr_Format(PyExc_TypeError, "%s must be a torch tensor or None", name);
      ok = false;
      return nullptr;
    }
    const at::Tensor* t = &THPVariable_Unpack(o);
    if (!t->is_cuda() || !t->is_contiguous()) {
      PyErr_Format(PyExc_ValueError, "%s must be a contiguous CUDA tensor", name);
      ok = false;
      return nullptr;
    }
    (void)t->data_ptr();  // throws here, under the interpreter lock, if there is no memory behind the tensor
    return t;
  }
  void* pointer(const char* name) {
    const at::Tensor* t = tensor(name);
    return t ? t->data_ptr() : nullptr;
  }
  // A tensor whose shape the call reads: None is an error; it has `dims` dimensions (-d: d or more).
  const at::Tensor* shaped(const char* name, int dims) {
    const at::Tensor* t = tensor(name);
    if (ok && !t) {
      PyErr_Format(PyExc_AttributeError, "%s must be a tensor, not None", name);
      ok = false;
    }
    if (ok && (dims > 0 ? t->dim() != dims : t->dim() < -dims)) {
      PyErr_Format(PyExc_ValueError, "%s must have %s%d dimensions, has %d", name, dims > 0 ? "" : "at least ", dims > 0 ? dims : -dims,
                   (int)t->dim());
      ok = false;
      return nullptr;
    }
    return t;
  }
};

struct Workspace {
  void* ptr;
  size_t bytes;
};
Workspace workspace(Args& in) {
  const at::Tensor* t = in.tensor("workspace");
  return t ? Workspace{t->data_ptr(), (size_t)t->nbytes()} : Workspace{nullptr, 0};
}

void* stream() { return (void*)c10::cuda::getCurrentCUDAStream().stream(); }

// K = last dimension, rows = the rest
void rows_and_k(const at::Tensor* t, int64_t& rows, int64_t& K) {
  K = t->dim() ? t->size(-1) : 0;
  rows = K ? t->numel() / K : 0;
}

// Runs the library call without the interpreter lock (a launch may wait for room in the driver's queue).
template <class F>
PyObject* status_of(const Args& in, F call) {
  if (!in.ok) return nullptr;
  void* s = stream();
  sdgp_status st;
  // (`call` only reads sizes and pointers of tensors the caller holds and that Args::tensor has checked: it does not throw)
  Py_BEGIN_ALLOW_THREADS
  st = call(s);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong((long)st);
}

#define ENTRY(name) PyObject* name(PyObject*, PyObject* const* args, Py_ssize_t nargs)

ENTRY(prune) {  // dO, n, m, scheme, seed, dtype, dense, values, meta, mask
  Args in(args, nargs, 10);
  const at::Tensor* dO = in.shaped("dO", 0);
  const int n = in.i32(), m = in.i32(), scheme = in.i32();
  const uint64_t seed = in.u64();
  const int dtype = in.i32();
  void *dense = in.pointer("dense"), *values = in.pointer("values"), *meta = in.pointer("meta"), *mask = in.pointer("mask");
  int64_t rows = 0, K = 0;
  if (in.ok) rows_and_k(dO, rows, K);
  return status_of(in, [&](void* s) {
    return sdgp_prune_typed(dO->data_ptr(), rows, K, n, m, (sdgp_scheme)scheme, seed, (sdgp_dtype)dtype, dense, values, meta, mask, s);
  });
}

ENTRY(relu_backward_prune) {  // dY, dSkip, residual, act, n, m, scheme, seed, dtype, grad, dense, values, meta, mask
  Args in(args, nargs, 14);
  const at::Tensor* dY = in.shaped("dY", 0);
  const at::Tensor* skip = in.tensor("dSkip");
  const int residual = in.i32();
  const at::Tensor* act = in.shaped("act", 0);
  const int n = in.i32(), m = in.i32(), scheme = in.i32();
  const uint64_t seed = in.u64();
  const int dtype = in.i32();
  void *grad = in.pointer("grad"), *dense = in.pointer("dense"), *values = in.pointer("values"), *meta = in.pointer("meta"),
       *mask = in.pointer("mask");
  int64_t rows = 0, K = 0;
  if (in.ok) {
    if (dY->sizes() != act->sizes() || (skip && skip->sizes() != dY->sizes())) {
      PyErr_SetString(PyExc_ValueError, residual ? "dY, dSkip and act must have the same shape" : "dY and act must have the same shape");
      in.ok = false;
    } else {
      rows_and_k(dY, rows, K);
    }
  }
  return status_of(in, [&](void* s) {
    if (residual)
      return sdgp_residual_relu_backward_prune(dY->data_ptr(), skip ? skip->data_ptr() : nullptr, act->data_ptr(), rows, K, n, m,
                                               (sdgp_scheme)scheme, seed, (sdgp_dtype)dtype, grad, dense, values, meta, mask, s);
    return sdgp_relu_backward_prune(dY->data_ptr(), act->data_ptr(), rows, K, n, m, (sdgp_scheme)scheme, seed, (sdgp_dtype)dtype,
                                    grad, dense, values, meta, mask, s);
  });
}

ENTRY(maxpool_relu_backward_prune) {  // dYp, skip, act, n, m, scheme, seed, dtype, grad, dense, values, meta, mask
  Args in(args, nargs, 13);
  const at::Tensor* dY = in.shaped("dYp", 0);
  const at::Tensor* skip = in.tensor("skip");
  const at::Tensor* act = in.shaped("act", 0);
  const int n = in.i32(), m = in.i32(), scheme = in.i32();
  const uint64_t seed = in.u64();
  const int dtype = in.i32();
  void *grad = in.pointer("grad"), *dense = in.pointer("dense"), *values = in.pointer("values"), *meta = in.pointer("meta"),
       *mask = in.pointer("mask");
  if (in.ok) {
    const char* wrong = nullptr;
    if (skip && skip->sizes() != dY->sizes()) wrong = "skip must have the shape of dYp";
    else if (act->dim() != 4 || dY->dim() != 4) wrong = "dYp and act must be NHWC tensors";
    else if (dY->size(0) != act->size(0) || dY->size(1) != act->size(1) / 2 || dY->size(2) != act->size(2) / 2 ||
             dY->size(3) != act->size(3))
      wrong = "dYp must be [B, H/2, W/2, K]";
    if (wrong) {
      PyErr_SetString(PyExc_ValueError, wrong);
      in.ok = false;
    }
  }
  return status_of(in, [&](void* s) {
    return sdgp_maxpool_relu_backward_prune(dY->data_ptr(), skip ? skip->data_ptr() : nullptr, act->data_ptr(), (int)act->size(0),
                                            (int)act->size(1), (int)act->size(2), act->size(3), n, m, (sdgp_scheme)scheme, seed,
                                            (sdgp_dtype)dtype, grad, dense, values, meta, mask, s);
  });
}

ENTRY(dgrad_linear) {  // dO, W, dD, n, m, scheme, seed, dtype, workspace, flags
  Args in(args, nargs, 10);
  const at::Tensor* dO = in.shaped("dO", 2);
  const at::Tensor* W = in.shaped("W", -2);
  void* dD = in.pointer("dD");
  const int n = in.i32(), m = in.i32(), scheme = in.i32();
  const uint64_t seed = in.u64();
  const int dtype = in.i32();
  const Workspace ws = workspace(in);
  const uint32_t flags = (uint32_t)in.i32();
  return status_of(in, [&](void* s) {
    return sdgp_dgrad_linear_typed(dO->data_ptr(), W->data_ptr(), dD, dO->size(0), dO->size(1), W->size(1), n, m, (sdgp_scheme)scheme,
                                   seed, (sdgp_dtype)dtype, ws.ptr, ws.bytes, flags, s);
  });
}

ENTRY(dgrad_linear_static) {  // dO, W, dD, n, m, scheme, seed
  Args in(args, nargs, 7);
  const at::Tensor* dO = in.shaped("dO", 2);
  const at::Tensor* W = in.shaped("W", -2);
  void* dD = in.pointer("dD");
  const int n = in.i32(), m = in.i32(), scheme = in.i32();
  const uint64_t seed = in.u64();
  return status_of(in, [&](void* s) {
    return sdgp_dgrad_linear_static(dO->data_ptr(), W->data_ptr(), dD, dO->size(0), dO->size(1), W->size(1), n, m, (sdgp_scheme)scheme,
                                    seed, s);
  });
}

// dO, W, dD, stride, pad, groups (0: sdgp_dgrad_conv2d), n, m, scheme, seed, dtype, workspace, flags
ENTRY(dgrad_conv2d) {
  Args in(args, nargs, 13);
  void* dO = in.pointer("dO");
  const at::Tensor* W = in.shaped("W", 4);
  const at::Tensor* dD = in.shaped("dD", 4);
  const int stride = in.i32(), pad = in.i32(), groups = in.i32(), n = in.i32(), m = in.i32(), scheme = in.i32();
  const uint64_t seed = in.u64();
  const int dtype = in.i32();
  const Workspace ws = workspace(in);
  const uint32_t flags = (uint32_t)in.i32();
  return status_of(in, [&](void* s) {
    const int B = (int)dD->size(0), H = (int)dD->size(1), Wd = (int)dD->size(2), Cin = (int)dD->size(3);
    const int Cout = (int)W->size(0), R = (int)W->size(1), S = (int)W->size(2);
    if (groups)
      return sdgp_dgrad_conv2d_grouped(dO, W->data_ptr(), dD->data_ptr(), B, H, Wd, Cin, Cout, R, S, stride, pad, groups, n, m,
                                       (sdgp_scheme)scheme, seed, (sdgp_dtype)dtype, ws.ptr, ws.bytes, flags, s);
    return sdgp_dgrad_conv2d_typed(dO, W->data_ptr(), dD->data_ptr(), B, H, Wd, Cin, Cout, R, S, stride, pad, n, m,
                                   (sdgp_scheme)scheme, seed, (sdgp_dtype)dtype, ws.ptr, ws.bytes, flags, s);
  });
}

ENTRY(spmm_linear) {  // values, meta, W, dD, dtype
  Args in(args, nargs, 5);
  void *values = in.pointer("values"), *meta = in.pointer("meta");
  const at::Tensor* W = in.shaped("W", -1);
  const at::Tensor* dD = in.shaped("dD", 2);
  const int dtype = in.i32();
  return status_of(in, [&](void* s) {
    return sdgp_spmm_linear_typed(values, meta, W->data_ptr(), dD->data_ptr(), dD->size(0), W->size(0), dD->size(1), (sdgp_dtype)dtype, s);
  });
}

ENTRY(spmm_conv2d) {  // values, meta, W, dD, stride, pad, dtype
  Args in(args, nargs, 7);
  void *values = in.pointer("values"), *meta = in.pointer("meta");
  const at::Tensor* W = in.shaped("W", 4);
  const at::Tensor* dD = in.shaped("dD", 4);
  const int stride = in.i32(), pad = in.i32(), dtype = in.i32();
  return status_of(in, [&](void* s) {
    return sdgp_spmm_conv2d_typed(values, meta, W->data_ptr(), dD->data_ptr(), (int)dD->size(0), (int)dD->size(1), (int)dD->size(2),
                                  (int)dD->size(3), (int)W->size(0), (int)W->size(1), (int)W->size(2), stride, pad, (sdgp_dtype)dtype, s);
  });
}

// Whether the C++ layers take a tensor: what Python hands over is an ordinary tensor (no subclass) in GPU memory of a 16-bit type, and
// nothing watches or transforms the operators that run on it.
bool plain_tensor(PyObject* o, int64_t dims) {
  if (!THPVariable_CheckExact(o)) return false;
  const at::Tensor& t = THPVariable_Unpack(o);
  return t.defined() && t.is_cuda() && t.layout() == at::kStrided && (dims < 0 ? t.dim() >= -dims : t.dim() == dims) &&
         (t.scalar_type() == at::kBFloat16 || t.scalar_type() == at::kHalf) && !at::isTensorSubclassLike(t) && !t._fw_grad(0).defined();
}

bool plain_int(PyObject* o) {  // (no bool, no object with __index__: the operators' own argument parser has its rules for those)
  if (!PyLong_CheckExact(o)) return false;
  int overflow = 0;
  const long long v = PyLong_AsLongLongAndOverflow(o, &overflow);
  return overflow == 0 && v >= INT32_MIN && v <= INT32_MAX;
}

// Differentiable layers: x, weight, then `integers` numbers, the last of them a seed. NotImplemented: not a plain call, the caller takes
// the Python form (which also gives the errors of arguments that are none).
template <class F>
PyObject* layer(PyObject* const* args, Py_ssize_t nargs, int integers, int64_t x_dims, int64_t weight_dims, F call) {
  HANDLE_TH_ERRORS
  Args in(args, nargs, 2 + integers);
  if (!in.ok) return nullptr;
  bool plain = !torch::jit::tracer::isTracing() && !at::impl::torch_function_mode_enabled() && plain_tensor(args[0], x_dims) &&
               plain_tensor(args[1], weight_dims) && PyLong_CheckExact(args[1 + integers]);
  for (int k = 2; plain && k < 1 + integers; ++k) plain = plain_int(args[k]);
  at::Tensor t[2];
  for (int k = 0; plain && k < 2; ++k, ++in.a) t[k] = THPVariable_Unpack(*in.a);
  if (!plain || t[0].scalar_type() != t[1].scalar_type() || t[0].device() != t[1].device()) Py_RETURN_NOTIMPLEMENTED;
  std::vector<int64_t> numbers;
  for (int k = 0; k < integers; ++k) numbers.push_back(k + 1 < integers ? (int64_t)in.i32() : (int64_t)in.u64());
  if (!in.ok) return nullptr;
  at::Tensor y;
  {
    struct NoGil {
      PyThreadState* state = PyEval_SaveThread();
      ~NoGil() { PyEval_RestoreThread(state); }
    } no_gil;
    y = call(t[0], t[1], std::move(numbers));
  }
  return THPVariable_Wrap(std::move(y));
  END_HANDLE_TH_ERRORS
}
ENTRY(linear_layer) {  // x, weight, n, m, scheme, seed
  return layer(args, nargs, 4, -1, 2, sdgp_torch::linear);
}
ENTRY(conv2d_layer) {  // x, weight, stride, padding, kind, n, m, scheme, seed
  return layer(args, nargs, 7, 4, 4, sdgp_torch::conv2d);
}

ENTRY(workspace_size_linear) {  // rows, K, N, flags
  Args in(args, nargs, 4);
  const int64_t rows = in.i64(), K = in.i64(), N = in.i64();
  const uint32_t flags = (uint32_t)in.i64();
  return in.ok ? PyLong_FromSize_t(sdgp_workspace_size_linear(rows, K, N, flags)) : nullptr;
}

ENTRY(workspace_size_conv2d) {  // B, H, Wd, Cin, Cout, R, S, stride, pad, groups (0: sdgp_workspace_size_conv2d), flags
  Args in(args, nargs, 11);
  int v[10];
  for (int& x : v) x = in.i32();
  const uint32_t flags = (uint32_t)in.i64();
  if (!in.ok) return nullptr;
  return PyLong_FromSize_t(v[9] ? sdgp_workspace_size_conv2d_grouped(v[0], v[1], v[2], v[3], v[4], v[5], v[6], v[7], v[8], v[9], flags)
                                : sdgp_workspace_size_conv2d(v[0], v[1], v[2], v[3], v[4], v[5], v[6], v[7], v[8], flags));
}

#undef ENTRY

// A C++ exception (data_ptr() of a tensor without storage, say) becomes a Python one.
template <PyObject* (*F)(PyObject*, PyObject* const*, Py_ssize_t)>
PyObject* guarded(PyObject* self, PyObject* const* args, Py_ssize_t nargs) {
  try {
    return F(self, args, nargs);
  } catch (const std::exception& e) {
    PyErr_SetString(PyExc_RuntimeError, e.what());
    return nullptr;
  }
}

#define METHOD(name) {#name, (PyCFunction)(void (*)(void))guarded<name>, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {METHOD(prune), METHOD(relu_backward_prune), METHOD(maxpool_relu_backward_prune), METHOD(dgrad_linear),
                         METHOD(dgrad_linear_static), METHOD(dgrad_conv2d), METHOD(spmm_linear), METHOD(spmm_conv2d),
                         METHOD(workspace_size_linear), METHOD(workspace_size_conv2d), METHOD(linear_layer),
                         METHOD(conv2d_layer), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module_def = {PyModuleDef_HEAD_INIT, "_sdgp_torch", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__sdgp_torch() { return PyModule_Create(&module_def); }
