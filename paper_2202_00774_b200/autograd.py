"""``torch.autograd`` front end: layers whose backward pass prunes the incoming output gradient
and computes the input gradient with the SDGP kernels (Algorithm 1; Section 3.1: "SDGP only
changes the data gradient; the weight gradient uses the unpruned dL/dO").

Only the data gradient runs in this library (and ReLU + 2 x 2 pooling, in one pass). Convolutions,
matrix products and the weight gradient are the framework's own operators, which is the
integration the paper describes (Section 1: a drop-in change of the backward pass). The layers
themselves are C++ (csrc/torch_autograd.cpp): a small layer's step is bound by the host. Tensors are bf16 or fp16 CUDA tensors; convolutions use
the channels-last memory format (its physical layout is the NHWC / [Cout,R,S,Cin] layout of the
C ABI, so nothing is copied or transposed).
"""
from __future__ import annotations

from . import binding as _b

_CONV, _CONV_RELU, _CONV_RELU_POOL = 0, 1, 2


def sdgp_linear(x, weight, n=2, m=4, scheme=_b.MAGNITUDE, seed=0):
    """``x @ weight.T`` whose input gradient is ``prune(dL/dO) @ weight`` (N:M along out_features).
    in_features and out_features must be multiples of 64."""
    return (_b._torch or _b._load()).linear_layer(x, weight, n, m, scheme, seed)


def sdgp_conv2d(x, weight, stride=1, padding=0, n=2, m=4, scheme=_b.MAGNITUDE, seed=0):
    """``conv2d(x, weight)`` (NCHW tensors, channels-last storage recommended, no bias, stride 1 or 2,
    one padding value for both axes) whose input gradient is computed from dL/dO pruned N:M along
    the output channels. Channel counts must be multiples of 64."""
    return (_b._torch or _b._load()).conv2d_layer(x, weight, stride, padding, _CONV, n, m, scheme, seed)


def sdgp_conv2d_relu(x, weight, stride=1, padding=0, pool=False, n=2, m=4, scheme=_b.MAGNITUDE, seed=0):
    """``relu(conv2d(x, weight))`` - with ``pool=True`` followed by ``max_pool2d(., 2)`` - whose backward pass
    forms and prunes the convolution's dL/dO in one pass over the incoming gradient (ReLU backward, pooling
    backward and Algorithm 1 together), computes the input gradient from the pruned copy and the weight gradient
    from the unpruned one (Section 3.1). Same tensor requirements as ``sdgp_conv2d``; with ``pool=True`` the
    convolution's output height and width must be even."""
    return (_b._torch or _b._load()).conv2d_layer(x, weight, stride, padding, _CONV_RELU_POOL if pool else _CONV_RELU, n, m, scheme, seed)
