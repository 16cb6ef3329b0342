// The torch.autograd layers (see autograd.py for what they are): forward and backward passes in C++, because a training step of a
// small layer is bound by the host. As Python autograd functions a convolution + ReLU + pooling block (128 images of 16 x 16, 128
// channels: 82 us of kernels) took 168 us of host time a step, a small linear layer 120 us.
//
// Only the data gradient (and, between a ReLU and a 2 x 2 pooling, the activation) runs in this library's kernels; convolutions,
// matrix products and weight gradients are the framework's own operators.
#include "torch_autograd.h"

#include <ATen/ATen.h>
#include <Python.h>
#include <c10/cuda/CUDAGuard.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/custom_function.h>

#include "../../include/sdgp.h"
#include "sdgp_internal.cuh"

namespace sdgp_torch {
namespace {

using at::MemoryFormat;
using at::Tensor;
using torch::autograd::AutogradContext;
using torch::autograd::variable_list;

// Raises binding.SdgpError for a status that is not OK (also from the autograd engine's threads).
void check(sdgp_status st, const char* what) {
  if (st == SDGP_OK) return;
  PyGILState_STATE gil = PyGILState_Ensure();
  PyObject* module = PyImport_ImportModule("paper_2202_00774_b200.binding");
  PyObject* type = module ? PyObject_GetAttrString(module, "SdgpError") : nullptr;
  PyObject* error = type ? PyObject_CallFunction(type, "is", (int)st, what) : nullptr;
  if (error) PyErr_SetObject(type, error);
  Py_XDECREF(error);
  Py_XDECREF(type);
  Py_XDECREF(module);
  python_error e;
  e.persist();
  PyGILState_Release(gil);
  throw e;
}

sdgp_dtype dtype_of(const Tensor& t) {
  TORCH_CHECK_TYPE(t.scalar_type() == at::kBFloat16 || t.scalar_type() == at::kHalf, "SDGP layers take bfloat16 or float16 tensors, got ",
                   t.scalar_type());
  return t.scalar_type() == at::kHalf ? SDGP_FP16 : SDGP_BF16;
}

void on_gpu(const Tensor& t, const char* name) { TORCH_CHECK_VALUE(t.is_cuda(), name, " must be a contiguous CUDA tensor"); }

void* stream() { return (void*)c10::cuda::getCurrentCUDAStream().stream(); }

Tensor bytes_like(const Tensor& t, size_t n) { return at::empty({(int64_t)(n < 16 ? 16 : n)}, t.options().dtype(at::kByte)); }

struct Linear : torch::autograd::Function<Linear> {
  static Tensor forward(AutogradContext* ctx, const Tensor& x, const Tensor& weight, std::vector<int64_t> pattern) {
    ctx->save_for_backward({x, weight});
    ctx->saved_data["pattern"] = pattern;  // n, m, scheme, seed
    return at::matmul(x, weight.t());
  }

  static variable_list backward(AutogradContext* ctx, variable_list grads) {
    const auto saved = ctx->get_saved_variables();
    const Tensor &x = saved[0], &weight = saved[1];
    const auto p = ctx->saved_data["pattern"].toIntVector();
    const Tensor dO = grads[0].reshape({-1, weight.size(0)}).contiguous();
    Tensor grad_x, grad_w;
    if (ctx->needs_input_grad(0)) {
      const sdgp_dtype dt = dtype_of(dO);
      // weight is [out_features, in_features] = [K, N]: the layout sdgp_dgrad_linear wants
      const Tensor W = weight.contiguous();
      on_gpu(dO, "dO");
      on_gpu(W, "W");
      const c10::cuda::CUDAGuard guard(dO.device());
      const int64_t rows = dO.size(0), K = dO.size(1), N = W.size(1);
      const Tensor dD = at::empty({rows, N}, dO.options());
      const Tensor ws = bytes_like(dO, sdgp_workspace_size_linear(rows, K, N, SDGP_FLAG_TWO_PASS));
      check(sdgp_dgrad_linear_typed(dO.data_ptr(), W.data_ptr(), dD.data_ptr(), rows, K, N, (int)p[0], (int)p[1], (sdgp_scheme)p[2],
                                    (uint64_t)p[3], dt, ws.data_ptr(), ws.nbytes(), SDGP_FLAG_TWO_PASS, stream()),
            "sdgp_dgrad_linear_typed");
      grad_x = dD.reshape(x.sizes());
    }
    if (ctx->needs_input_grad(1)) grad_w = at::matmul(dO.t(), x.reshape({-1, x.size(-1)}));  // unpruned dL/dO (Section 3.1)
    return {grad_x, grad_w, Tensor()};
  }
};

// Weight gradient of a convolution from the unpruned dL/dO (Section 3.1).
Tensor conv_weight_grad(const Tensor& x, const Tensor& weight, const Tensor& dO, int64_t stride, int64_t padding) {
  const Tensor shape_only = dO.new_empty({1}).expand(weight.sizes());
  return std::get<1>(at::convolution_backward(dO, x, shape_only, at::OptionalIntArrayRef(), {stride, stride}, {padding, padding}, {1, 1},
                                              false, {0, 0}, 1, {false, true, false}));
}

struct Conv2d : torch::autograd::Function<Conv2d> {
  // cfg: stride, padding, kind (kPlain ...), n, m, scheme, seed
  static Tensor forward(AutogradContext* ctx, const Tensor& x, const Tensor& weight, std::vector<int64_t> cfg) {
    const int64_t kind = cfg[2];
    ctx->saved_data["cfg"] = cfg;
    Tensor out = at::conv2d(x, weight, {}, {cfg[0], cfg[0]}, {cfg[1], cfg[1]});
    if (kind == kConv) {
      ctx->save_for_backward({x, weight});
      return out;
    }
    out = out.contiguous(MemoryFormat::ChannelsLast);
    const int64_t B = out.size(0), C = out.size(1), H = out.size(2), W = out.size(3);
    const bool f16 = out.scalar_type() == at::kHalf;
    if (kind == kConvReluPool && out.is_cuda() && (f16 || out.scalar_type() == at::kBFloat16) && H % 2 == 0 && W % 2 == 0 && C % 8 == 0 &&
        out.numel() > 0 && ((uintptr_t)out.data_ptr() & 15u) == 0) {
      // ReLU and pooling in one pass; what the backward pass needs of the activation is the convolution's output itself
      const c10::cuda::CUDAGuard guard(out.device());  // (the tensors' device need not be the current one)
      const Tensor y = at::empty({B, C, H / 2, W / 2}, out.options(), MemoryFormat::ChannelsLast);
      TORCH_CHECK(sdgp::launch_relu_maxpool(out.data_ptr(), B, H, W, C, f16 ? SDGP_FP16 : SDGP_BF16, y.data_ptr(), (cudaStream_t)stream()) ==
                      cudaSuccess,
                  "relu + max pooling: launch failed");
      ctx->save_for_backward({x, weight, out});
      return y;
    }
    const Tensor act = at::relu_(out);
    ctx->save_for_backward({x, weight, act});
    return kind == kConvReluPool ? at::max_pool2d(act, {2, 2}) : act;
  }

  static variable_list backward(AutogradContext* ctx, variable_list grads) {
    const auto saved = ctx->get_saved_variables();
    const Tensor &x = saved[0], &weight = saved[1];
    const auto cfg = ctx->saved_data["cfg"].toIntVector();
    const int stride = (int)cfg[0], padding = (int)cfg[1], n = (int)cfg[3], m = (int)cfg[4];
    const int64_t kind = cfg[2];
    const sdgp_scheme scheme = (sdgp_scheme)cfg[5];
    const uint64_t seed = (uint64_t)cfg[6];
    const int B = (int)x.size(0), Cin = (int)x.size(1), H = (int)x.size(2), Wd = (int)x.size(3);
    const int Cout = (int)weight.size(0), R = (int)weight.size(2), S = (int)weight.size(3);
    const bool need_x = ctx->needs_input_grad(0), need_w = ctx->needs_input_grad(1);
    Tensor dO = grads[0], vals, meta, grad_x, grad_w;  // channels-last tensors are NHWC in memory
    if (kind != kConv) {
      // dL/dO from the gradient above the ReLU (or the pooling), its compressed pruned copy in the same pass
      const Tensor& act = saved[2];
      const sdgp_dtype dt = dtype_of(grads[0]);
      const int P = (int)act.size(2), Q = (int)act.size(3);
      const Tensor dY = grads[0].contiguous(MemoryFormat::ChannelsLast);
      on_gpu(dY, "dY");
      const c10::cuda::CUDAGuard guard(dY.device());
      const bool pool = kind == kConvReluPool;
      if (pool) {
        TORCH_CHECK_VALUE(dY.size(0) == B && dY.size(1) == Cout && dY.size(2) == P / 2 && dY.size(3) == Q / 2, "dYp must be [B, H/2, W/2, K]");
      } else {
        TORCH_CHECK_VALUE(dY.sizes() == act.sizes(), "dY and act must have the same shape");
      }
      dO = at::empty(act.sizes(), dY.options(), MemoryFormat::ChannelsLast);
      const bool compressed = n <= 2 && Cout % 128 == 0 && need_x;
      if (compressed) {
        vals = at::empty({(int64_t)B * P * Q, Cout / 2}, dY.options());
        meta = at::empty({(int64_t)B * P * Q, Cout / 16}, dY.options().dtype(at::kShort));
      }
      void *pv = compressed ? vals.data_ptr() : nullptr, *pm = compressed ? meta.data_ptr() : nullptr;
      const int pn = compressed ? n : 4, pg = compressed ? m : 4;  // n == m: nothing is pruned, the producer only writes dL/dO
      if (pool)
        check(sdgp_maxpool_relu_backward_prune(dY.data_ptr(), nullptr, act.data_ptr(), B, P, Q, Cout, pn, pg, scheme, seed, dt, dO.data_ptr(),
                                               nullptr, pv, pm, nullptr, stream()),
              "sdgp_maxpool_relu_backward_prune");
      else
        check(sdgp_relu_backward_prune(dY.data_ptr(), act.data_ptr(), (int64_t)B * P * Q, Cout, pn, pg, scheme, seed, dt, dO.data_ptr(),
                                       nullptr, pv, pm, nullptr, stream()),
              "sdgp_relu_backward_prune");
    }
    if (need_x) {
      const Tensor g = dO.contiguous(MemoryFormat::ChannelsLast);
      const Tensor W = weight.contiguous(MemoryFormat::ChannelsLast);  // [Cout,R,S,Cin]
      const sdgp_dtype dt = dtype_of(g);
      on_gpu(g, "dO");
      on_gpu(W, "W");
      const c10::cuda::CUDAGuard guard(g.device());
      grad_x = at::empty(x.sizes(), g.options(), MemoryFormat::ChannelsLast);
      if (vals.defined()) {
        check(sdgp_spmm_conv2d_typed(vals.data_ptr(), meta.data_ptr(), W.data_ptr(), grad_x.data_ptr(), B, H, Wd, Cin, Cout, R, S, stride,
                                     padding, dt, stream()),
              "sdgp_spmm_conv2d_typed");
      } else {  // a pass of its own prunes dL/dO
        const uint32_t flags = kind == kConv || n <= 2 ? SDGP_FLAG_TWO_PASS : SDGP_FLAG_MASKED;
        const Tensor ws = bytes_like(g, sdgp_workspace_size_conv2d(B, H, Wd, Cin, Cout, R, S, stride, padding, flags));
        check(sdgp_dgrad_conv2d_typed(g.data_ptr(), W.data_ptr(), grad_x.data_ptr(), B, H, Wd, Cin, Cout, R, S, stride, padding, n, m, scheme,
                                      seed, dt, ws.data_ptr(), ws.nbytes(), flags, stream()),
              "sdgp_dgrad_conv2d_typed");
      }
    }
    if (need_w) grad_w = conv_weight_grad(x, weight, dO, stride, padding);
    return {grad_x, grad_w, Tensor()};
  }
};

}  // namespace

Tensor linear(const Tensor& x, const Tensor& weight, std::vector<int64_t> pattern) { return Linear::apply(x, weight, std::move(pattern)); }

Tensor conv2d(const Tensor& x, const Tensor& weight, std::vector<int64_t> cfg) { return Conv2d::apply(x, weight, std::move(cfg)); }

}  // namespace sdgp_torch
