// Differentiable layers of the torch module.
#pragma once
#include <ATen/core/Tensor.h>

#include <vector>

namespace sdgp_torch {

constexpr int64_t kConv = 0, kConvRelu = 1, kConvReluPool = 2;

// x . weight^T; pattern: n, m, scheme, seed.
at::Tensor linear(const at::Tensor& x, const at::Tensor& weight, std::vector<int64_t> pattern);
// conv2d, or relu(conv2d), or max_pool2d(relu(conv2d), 2); cfg: stride, padding, kind, n, m, scheme, seed.
at::Tensor conv2d(const at::Tensor& x, const at::Tensor& weight, std::vector<int64_t> cfg);

}  // namespace sdgp_torch
