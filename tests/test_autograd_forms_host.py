"""Calls of the differentiable layers that are not plain CUDA calls: what the operators take, the layers take (no kernel of the library
runs here: the tensors are on the CPU or have no memory, and only the weight gradient is asked for)."""
import pytest
import torch
import torch.nn.functional as F

from paper_2202_00774_b200 import autograd

LAYERS = {"conv": (autograd.sdgp_conv2d, lambda y: y),
          "relu": (autograd.sdgp_conv2d_relu, torch.relu),
          "pool": (lambda *a, **k: autograd.sdgp_conv2d_relu(*a, pool=True, **k), lambda y: F.max_pool2d(torch.relu(y), 2))}


def tensors(dtype=torch.float32, device="cpu", k=3):
    g = torch.Generator().manual_seed(3)
    x = torch.randn((2, 64, 8, 8), generator=g).to(device, dtype)
    return x, (torch.randn((64, 64, k, k), generator=g) * 0.05).to(device, dtype).requires_grad_()


@pytest.mark.parametrize("name", LAYERS)
@pytest.mark.parametrize("stride, padding", [((1, 1), (1, 1)), ([2, 1], [1, 0]), ((1,), 1), (1, "same"), (2, "valid"), (torch.Size([1, 1]), 0)])
def test_strides_and_paddings_that_are_not_one_integer(name, stride, padding):
    layer, after = LAYERS[name]
    x, w = tensors()
    y = layer(x, w, stride, padding)
    assert torch.equal(y, after(F.conv2d(x, w, None, stride, padding)))
    if name == "conv" and not isinstance(padding, str):
        expected, = torch.autograd.grad(F.conv2d(x, w, None, stride, padding).square().sum(), w)
        assert torch.allclose(torch.autograd.grad(y.square().sum(), w)[0], expected, rtol=1e-4, atol=1e-3)  # fp32 sums in another order


@pytest.mark.parametrize("name", LAYERS)
def test_fake_tensors(name):
    from torch._subclasses.fake_tensor import FakeTensorMode
    with FakeTensorMode():
        x = torch.empty((2, 64, 8, 8), device="cuda", dtype=torch.bfloat16)
        w = torch.empty((64, 64, 3, 3), device="cuda", dtype=torch.bfloat16)
        y = LAYERS[name][0](x, w, 1, 1)
    side = 4 if name == "pool" else 8
    assert y.shape == (2, 64, side, side) and y.device.type == "cuda" and y.dtype == torch.bfloat16


@pytest.mark.parametrize("name", LAYERS)
def test_subclasses_see_the_operators(name):
    class Counting(torch.Tensor):
        calls = 0

        @classmethod
        def __torch_function__(cls, func, types, args=(), kwargs=None):
            Counting.calls += 1
            return super().__torch_function__(func, types, args, kwargs or {})

    x, w = tensors()
    y = LAYERS[name][0](x.as_subclass(Counting), w, 1, 1)
    assert type(y) is Counting and Counting.calls > 0


@pytest.mark.parametrize("name", LAYERS)
def test_transforms_are_refused_as_before(name):
    x, w = tensors()
    with pytest.raises(NotImplementedError), torch.autograd.forward_ad.dual_level():
        LAYERS[name][0](torch.autograd.forward_ad.make_dual(x, x), w, 1, 1)
    with pytest.raises(RuntimeError):
        torch.func.vmap(lambda a: LAYERS[name][0](a, w.detach(), 1, 1))(x[None])


def test_linear_compiles_as_one_graph():
    g = torch.Generator().manual_seed(4)
    x, w = torch.randn((4, 64), generator=g), torch.randn((64, 64), generator=g).requires_grad_()
    y = torch.compile(lambda a, b: autograd.sdgp_linear(a, b) + 1, backend="eager", fullgraph=True)(x, w)
    expected = x @ w.t() + 1
    assert torch.equal(y, expected)
    assert torch.equal(torch.autograd.grad(y.sum(), w)[0], torch.autograd.grad(expected.sum(), w)[0])
