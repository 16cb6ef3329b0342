"""Workloads that stand for what a training step asks of this library, as plain descriptions.

A case names an operation, its sizes, the pruning pattern and the element type; ``prepare`` makes the tensors a
training loop holds at that point (gradients, activations, filters, caller-owned outputs and workspace) and ``run``
makes the call or calls of one backward step through the public entry points. Shapes are those of the layers of
ResNet-9 (CIFAR-sized), ResNet-50 and RegNetX-400MF and of fully connected layers; values follow
``paper_2202_00774_b200.inputs``: N(0,1) gradients for fully connected layers, Laplace(0,1) with half of the values
exactly zero (a gradient that came back through a ReLU) for convolutions, He-normal filters.
"""
import math

import torch

import paper_2202_00774_b200 as sdgp
from paper_2202_00774_b200 import autograd, binding

SCHEMES = {"random": binding.RANDOM, "magnitude": binding.MAGNITUDE, "rescaled": binding.RESCALED_MAGNITUDE}
FLAGS = {"two_pass": binding.FLAG_TWO_PASS, "fused": binding.FLAG_FUSED, "masked": binding.FLAG_MASKED,
         "channel": binding.FLAG_CHANNEL}
TYPES = {"bf16": (torch.bfloat16, binding.BF16), "fp16": (torch.float16, binding.FP16)}
PRUNE_SEED = 20220202   # seed of the random pruning function (a training loop passes its step number)


# ------------------------------------------------------------------ descriptions


def _pattern(n, m, scheme, dtype="bf16"):
    return {"n": n, "m": m, "scheme": scheme, "dtype": dtype}


def _linear(rows, K, N, mode, **pattern):
    """dO [rows, K] . W [K, N]: K output features, N input features."""
    return {"op": "linear", "rows": rows, "K": K, "N": N, "mode": mode, **pattern}


def _conv(op, batch, size, cin, cout, kernel, stride, **more):
    """cin -> cout channels on a size x size input image, ``kernel`` x ``kernel`` filter, padding (kernel - 1) / 2."""
    return {"op": op, "batch": batch, "size": size, "cin": cin, "cout": cout, "kernel": kernel, "stride": stride, **more}


def listed():
    return [
        # the smallest fully connected layer of the benchmark: a handful of microseconds, so the host's share shows
        {"name": "fc_small", **_linear(256, 512, 256, "two_pass", **_pattern(2, 4, "magnitude"))},
        # a classifier or projection layer with a batch and widths that fill no tile evenly, in the paper's precision
        {"name": "fc_ragged", **_linear(1777, 1088, 832, "two_pass", **_pattern(2, 4, "rescaled", "fp16"))},
        # the large fully connected layer of the benchmark: tensor-core bound
        {"name": "gemm_large", **_linear(16384, 4096, 4096, "two_pass", **_pattern(2, 4, "magnitude"))},
        # Algorithm 1 alone, for a caller that keeps the mask and runs the contraction later
        {"name": "prune_2of8", "op": "prune", "rows": 16384, "K": 4096, "mask": True, "dense": False,
         **_pattern(2, 8, "rescaled")},
        # ResNet-9: the widest image of the chain
        {"name": "r9_64to128_at32", **_conv("conv", 512, 32, 64, 128, 3, 1, mode="two_pass", **_pattern(2, 4, "magnitude"))},
        # ResNet-9: the deepest layers (4 x 4 images), as one fused kernel
        {"name": "r9_512to512_at4_fused", **_conv("conv", 512, 4, 512, 512, 3, 1, mode="fused", **_pattern(2, 4, "magnitude"))},
        # ResNet-9 at 4:32, the pattern of the time-to-accuracy experiment (no 2:4 form: dense copy, dense contraction)
        {"name": "r9_128to128_at16_4of32", **_conv("conv", 512, 16, 128, 128, 3, 1, mode="masked", **_pattern(4, 32, "magnitude"))},
        # ResNet-50: the expanding 1 x 1 convolution of stage 3, the shape the network holds most often
        {"name": "r50_1x1_256to1024_at14", **_conv("conv", 256, 14, 256, 1024, 1, 1, mode="two_pass", **_pattern(2, 4, "magnitude"))},
        # ResNet-50: the strided 3 x 3 convolution that opens stage 2, random pruning (the paper's control)
        {"name": "r50_3x3s2_128_at56", **_conv("conv", 256, 56, 128, 128, 3, 2, mode="two_pass", **_pattern(2, 4, "random"))},
        # ResNet-50: backward through a residual block's ReLU into the 3 x 3 convolution below it
        {"name": "r50_residual_chain_at14", **_conv("chain", 256, 14, 256, 256, 3, 1, above="residual", **_pattern(2, 4, "magnitude"))},
        # RegNetX-400MF: the grouped 3 x 3 convolution of stage 3 (160 channels, group width 16)
        {"name": "regnetx_3x3g10_at14", **_conv("grouped", 256, 14, 160, 160, 3, 1, groups=10, mode="two_pass", **_pattern(2, 4, "rescaled", "fp16"))},
        # a convolution + ReLU + pooling block trained through torch.autograd: forward, data and weight gradients
        {"name": "autograd_block_at16", **_conv("layer", 128, 16, 128, 128, 3, 1, layer="conv_relu_pool", **_pattern(2, 4, "magnitude"))},
    ]


SPARSE_PATTERNS = [(1, 4), (2, 4), (2, 4), (2, 4), (2, 8), (2, 16), (2, 32)]
MASKED_PATTERNS = [(3, 4), (4, 8), (4, 16), (8, 16), (4, 32), (16, 32)]
MOST_FLOPS, MOST_BYTES = 4e11, 2.4e8   # dense-equivalent work and traffic of a drawn case


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _multiple(rng, of, lo, hi):
    return of * max(1, round(_log_int(rng, lo, hi) / of))


def _drawn_pattern(rng, mode):
    n, m = rng.choice(MASKED_PATTERNS if mode == "masked" else SPARSE_PATTERNS)
    if mode == "fused" and m == 32:
        n, m = 2, 4
    scheme = "rescaled" if mode == "channel" else rng.choice(["magnitude", "magnitude", "rescaled", "random"])
    dtype = rng.choice(["bf16", "bf16", "fp16"])
    if mode == "fused" and scheme == "rescaled":
        dtype = "bf16"
    return _pattern(n, m, scheme, dtype)


def _drawn(rng):
    op = rng.choice(["linear", "linear", "linear", "conv", "conv", "conv", "conv", "chain", "chain", "prune", "grouped", "layer"])
    if op == "prune":
        pattern = _drawn_pattern(rng, "two_pass")
        return {"op": op, "rows": _log_int(rng, 64, 32768), "K": _multiple(rng, 64, 64, 4096), "mask": rng.random() < 0.5,
                "dense": rng.random() < 0.3, **pattern}
    if op == "linear":
        mode = rng.choice(["two_pass", "two_pass", "two_pass", "masked", "channel", "fused"])
        return _linear(_log_int(rng, 32, 16384), _multiple(rng, 64, 128, 4096), _multiple(rng, 64, 64, 4096), mode,
                       **_drawn_pattern(rng, mode))
    size, batch = rng.choice([4, 7, 8, 13, 14, 16, 27, 28, 32, 56]), _log_int(rng, 16, 512)
    kernel = rng.choice([1, 3, 3])
    stride = 2 if size > 8 and rng.random() < 0.25 else 1
    cin, cout = _multiple(rng, 64, 64, 1024), _multiple(rng, 64, 64, 1024)
    if op == "conv":
        mode = rng.choice(["two_pass", "two_pass", "two_pass", "fused", "fused", "masked", "channel"])
        return _conv(op, batch, size, cin, cout, kernel, stride, mode=mode, **_drawn_pattern(rng, mode))
    if op == "chain":
        above = rng.choice(["relu", "residual", "pool", "pool_residual"])
        size = size // 2 * 2 if "pool" in above else size
        return _conv(op, batch, size, cin, _multiple(rng, 128, 128, 1024), kernel, 1, above=above, **_drawn_pattern(rng, "two_pass"))
    if op == "grouped":
        groups = rng.randint(2, 24)
        return _conv(op, batch, size, 16 * groups, 16 * groups, 3, stride, groups=groups, mode="two_pass",
                     **_pattern(2, 4, rng.choice(["magnitude", "rescaled", "random"]), rng.choice(["bf16", "fp16"])))
    layer = rng.choice(["linear", "conv", "conv_relu", "conv_relu_pool"])
    if layer == "linear":
        return {"op": op, "layer": layer, "rows": _log_int(rng, 64, 8192), "K": _multiple(rng, 64, 128, 2048),
                "N": _multiple(rng, 64, 64, 2048), **_drawn_pattern(rng, "two_pass")}
    size = size // 2 * 2 if layer == "conv_relu_pool" else size
    return _conv(op, batch, size, cin, cout, kernel, 1, layer=layer, **_drawn_pattern(rng, "two_pass"))


def draw(rng):
    while True:
        case = _drawn(rng)
        w = work(case)
        if w["bytes"] <= MOST_BYTES and w["flops"] * case["m"] / case["n"] <= MOST_FLOPS:
            return case


# ------------------------------------------------------------------ tensors


def _out(case):
    """Output image side of the convolution."""
    return (case["size"] + 2 * (case["kernel"] // 2) - case["kernel"]) // case["stride"] + 1


class _Source:
    """Seeded device tensors."""

    def __init__(self, seed, dtype):
        self.g = torch.Generator(device="cuda")
        self.g.manual_seed(seed)
        self.dtype = dtype

    def normal(self, shape, std=1.0):
        return torch.randn(shape, generator=self.g, device="cuda", dtype=torch.float32).mul_(std).to(self.dtype)

    def relu_gradient(self, shape):
        """Laplace(0, 1), half of the values exactly zero."""
        x = torch.empty(shape, device="cuda", dtype=torch.float32).exponential_(generator=self.g)
        u = torch.randint(0, 4, shape, generator=self.g, device="cuda", dtype=torch.int8)   # 0, 1: zero; 2, 3: the sign
        return x.mul_((u >= 2).float()).mul_(1.0 - 2.0 * (u == 3).float()).to(self.dtype)

    def activation(self, shape):
        return torch.relu(self.normal(shape))

    def empty(self, shape, dtype=None):
        return torch.empty(shape, device="cuda", dtype=dtype or self.dtype)

    def workspace(self, size):
        return torch.empty(max(size, 16), device="cuda", dtype=torch.uint8)


def prepare(case, seed):
    dtype, code = TYPES[case["dtype"]]
    src = _Source(seed, dtype)
    st = {"case": case, "code": code, "args": (case["n"], case["m"], SCHEMES[case["scheme"]])}
    op = case["op"]
    if op == "prune":
        rows, K = case["rows"], case["K"]
        st["dO"] = src.relu_gradient((rows, K))
        st["out"] = {"values": src.empty((rows, K // 2)), "meta": src.empty((rows, K // 16), torch.int16)}
        if case["mask"]:
            st["out"]["mask"] = src.empty((rows, K // 32), torch.int32)
        if case["dense"]:
            st["out"]["dense"] = src.empty((rows, K))
        return st
    if op == "linear":
        rows, K, N, flags = case["rows"], case["K"], case["N"], FLAGS[case["mode"]]
        st.update(dO=src.normal((rows, K)), W=src.normal((K, N), K ** -0.5), dD=src.empty((rows, N)), flags=flags,
                  ws=src.workspace(sdgp.sdgp_workspace_size_linear(rows, K, N, flags)))
        return st
    if op == "layer" and case["layer"] == "linear":
        rows, K, N = case["rows"], case["K"], case["N"]
        st.update(x=src.normal((rows, N)).requires_grad_(), W=src.normal((K, N), N ** -0.5).requires_grad_(), dY=src.normal((rows, K)))
        return st

    B, hw, cin, cout, k, stride = (case[f] for f in ("batch", "size", "cin", "cout", "kernel", "stride"))
    pq, pad = _out(case), k // 2
    st.update(stride=stride, pad=pad)
    std = (2.0 / (k * k * cin / case.get("groups", 1))) ** 0.5
    if op == "layer":
        pooled = 2 if case["layer"] == "conv_relu_pool" else 1
        last = torch.channels_last
        st.update(x=src.activation((B, cin, hw, hw)).contiguous(memory_format=last).requires_grad_(),
                  W=src.normal((cout, cin, k, k), std).contiguous(memory_format=last).requires_grad_(),
                  dY=src.normal((B, cout, pq // pooled, pq // pooled)).contiguous(memory_format=last))
        return st
    st.update(W=src.normal((cout, k, k, cin // case.get("groups", 1)), std), dD=src.empty((B, hw, hw, cin)))
    if op == "chain":
        pooled = "pool" in case["above"]
        grads = (B, pq // 2, pq // 2, cout) if pooled else (B, pq, pq, cout)
        st.update(dY=src.normal(grads), act=src.activation((B, pq, pq, cout)), grad=src.empty((B, pq, pq, cout)),
                  values=src.empty((B, pq, pq, cout // 2)), meta=src.empty((B, pq, pq, cout // 16), torch.int16))
        if "residual" in case["above"]:
            st["skip"] = src.normal(grads)
        return st
    flags = FLAGS[case["mode"]]
    geometry = (B, hw, hw, cin, cout, k, k, stride, pad)
    size = (sdgp.sdgp_workspace_size_conv2d_grouped(*geometry, case["groups"], flags) if op == "grouped"
            else sdgp.sdgp_workspace_size_conv2d(*geometry, flags))
    st.update(dO=src.relu_gradient((B, pq, pq, cout)), flags=flags, ws=src.workspace(size))
    return st


# ------------------------------------------------------------------ one backward step


def run(st):
    case, args, code = st["case"], st["args"], st["code"]
    op, bf16 = case["op"], st["code"] == binding.BF16
    if op == "prune":
        if bf16:
            sdgp.sdgp_prune(st["dO"], *args, PRUNE_SEED, **st["out"])
        else:
            sdgp.sdgp_prune_typed(st["dO"], *args, PRUNE_SEED, code, **st["out"])
        return st["out"]
    if op == "linear":
        if bf16:
            sdgp.sdgp_dgrad_linear(st["dO"], st["W"], st["dD"], *args, PRUNE_SEED, workspace=st["ws"], flags=st["flags"])
        else:
            sdgp.sdgp_dgrad_linear_typed(st["dO"], st["W"], st["dD"], *args, PRUNE_SEED, code, workspace=st["ws"], flags=st["flags"])
        return st["dD"]
    if op == "conv":
        if bf16:
            sdgp.sdgp_dgrad_conv2d(st["dO"], st["W"], st["dD"], st["stride"], st["pad"], *args, PRUNE_SEED, workspace=st["ws"],
                                   flags=st["flags"])
        else:
            sdgp.sdgp_dgrad_conv2d_typed(st["dO"], st["W"], st["dD"], st["stride"], st["pad"], *args, PRUNE_SEED, code,
                                         workspace=st["ws"], flags=st["flags"])
        return st["dD"]
    if op == "grouped":
        sdgp.sdgp_dgrad_conv2d_grouped(st["dO"], st["W"], st["dD"], st["stride"], st["pad"], case["groups"], *args, PRUNE_SEED, code,
                                       workspace=st["ws"], flags=st["flags"])
        return st["dD"]
    if op == "chain":
        out = {"grad": st["grad"], "values": st["values"], "meta": st["meta"]}
        if case["above"] == "relu":
            sdgp.sdgp_relu_backward_prune(st["dY"], st["act"], *args, PRUNE_SEED, code, **out)
        elif case["above"] == "residual":
            sdgp.sdgp_residual_relu_backward_prune(st["dY"], st["skip"], st["act"], *args, PRUNE_SEED, code, **out)
        else:
            sdgp.sdgp_maxpool_relu_backward_prune(st["dY"], st["act"], *args, PRUNE_SEED, code, skip=st.get("skip"), **out)
        if bf16:
            sdgp.sdgp_spmm_conv2d(st["values"], st["meta"], st["W"], st["dD"], st["stride"], st["pad"])
        else:
            sdgp.sdgp_spmm_conv2d_typed(st["values"], st["meta"], st["W"], st["dD"], st["stride"], st["pad"], code)
        return {"dD": st["dD"], **out}
    layer, pattern = case["layer"], dict(zip(("n", "m", "scheme"), args), seed=PRUNE_SEED)
    if layer == "linear":
        y = autograd.sdgp_linear(st["x"], st["W"], **pattern)
    elif layer == "conv":
        y = autograd.sdgp_conv2d(st["x"], st["W"], st["stride"], st["pad"], **pattern)
    else:
        y = autograd.sdgp_conv2d_relu(st["x"], st["W"], st["stride"], st["pad"], pool=layer == "conv_relu_pool", **pattern)
    dx, dW = torch.autograd.grad(y, (st["x"], st["W"]), st["dY"])
    return {"y": y.detach(), "dx": dx, "dW": dW}


# ------------------------------------------------------------------ what a step cannot do without


def work(case):
    """Bytes: inputs read once, outputs written once. Flops: products of the surviving gradients only (dense contractions
    of a layer's forward pass and weight gradient in full)."""
    keep = case["n"] / case["m"]
    op = case["op"]
    if op == "prune":
        e = case["rows"] * case["K"]
        return {"bytes": e * (2 + 1 + 0.125 + 0.125 * case["mask"] + 2 * case["dense"]), "flops": 0}
    if op == "linear" or case.get("layer") == "linear":
        o, d, w = case["rows"] * case["K"], case["rows"] * case["N"], case["K"] * case["N"]
        flops = 2.0 * case["rows"] * w
    else:
        B, hw, cin, cout, k, pq = case["batch"], case["size"], case["cin"], case["cout"], case["kernel"], _out(case)
        g = case.get("groups", 1)
        o, d, w = B * pq * pq * cout, B * hw * hw * cin, cout * k * k * cin // g
        flops = 2.0 * B * pq * pq * w
    if op == "layer":   # forward: x, W, y; backward: dY, y or x, W again, dx, dW
        return {"bytes": 2.0 * (3 * d + 3 * o + 3 * w), "flops": flops * (2 + keep)}
    extra = 0
    if op == "chain":   # the gradients above, the activation, the compressed form (dO is the gradient that is written)
        above = o // 4 if "pool" in case["above"] else o
        extra = 2 * above * (2 if "residual" in case["above"] else 1) + 2 * o + 1.125 * o
    return {"bytes": 2.0 * (o + d + w) + extra, "flops": flops * keep}


def tolerance(case):
    """Pruning itself is exact; the contraction adds exact products in fp32 in any order and rounds once to 16 bits."""
    if case["op"] == "prune":
        return "exact"
    return {"rel": 4e-3, "max": 0.03} if case["dtype"] == "bf16" else {"rel": 1e-3, "max": 0.01}
