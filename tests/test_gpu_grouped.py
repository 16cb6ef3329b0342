"""Data gradient of grouped convolutions and of channel counts that are not multiples of 64 (the RegNetX-400MF
shape set, Section 4) on the GPU vs the fp64 CPU oracle, through the C ABI. Tolerances as in test_gpu_dgrad.py:
relative Frobenius error <= 5e-3 and, per element, 2^-7 |ref| + 2^-16 sum |a||b|."""
import numpy as np
import pytest

import oracle
import plan_cases
from paper_2202_00774_b200 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 5e-3


def dev16(a):
    return torch.from_numpy(np.ascontiguousarray(a).view(np.int16)).cuda()


def to_f64(t):
    return inputs.bf16_bits_to_f32(t.cpu().numpy().view(np.uint16)).astype(np.float64)


def magnitudes(bits):
    return (np.asarray(bits).view(np.uint16) & np.uint16(0x7FFF)).astype(np.uint16)


def to_f16_f64(t):
    return inputs.f16_bits_to_f32(t.cpu().numpy().view(np.uint16)).astype(np.float64)


def check(got, src, W, layer, what, dtype=oracle.BF16):
    ref = oracle.dgrad_conv2d_grouped(src, W, layer.H, layer.W, layer.groups, layer.stride, layer.pad, dtype=dtype)
    absdot = oracle.dgrad_conv2d_grouped(magnitudes(src), magnitudes(W), layer.H, layer.W, layer.groups, layer.stride, layer.pad, dtype=dtype)
    assert np.linalg.norm(got - ref) <= TOL * max(np.linalg.norm(ref), 1e-30), what
    # one rounding to the 16-bit type, with a factor two to spare (binary16: 2^-11 of the value, 2^-25 below 2^-14)
    unit, least = (2.0 ** -10, 2.0 ** -24) if dtype == oracle.FP16 else (2.0 ** -7, 0.0)
    bad = ~(np.abs(got - ref) <= unit * np.abs(ref) + 2.0 ** -16 * absdot + least)
    assert not bad.any(), "%s: %d elements off, first at %s" % (what, int(bad.sum()), np.argwhere(bad)[0])


def run(layer, n, m, scheme, flags, seed=9, dtype=oracle.BF16):
    import paper_2202_00774_b200 as sdgp
    dO, W = inputs.conv_layer_tensors(layer, seed=seed)
    if dtype == oracle.FP16:
        dO, W = inputs.bf16_bits_as_f16_bits(dO), inputs.bf16_bits_as_f16_bits(W)
    size = sdgp.sdgp_workspace_size_conv2d_grouped(layer.B, layer.H, layer.W, layer.Cin, layer.Cout, layer.R, layer.S,
                                                   layer.stride, layer.pad, layer.groups, flags)
    ws = torch.empty(size, dtype=torch.uint8, device="cuda")
    dD = torch.full(layer.dD_shape(), -1, dtype=torch.int16, device="cuda")
    sdgp.sdgp_dgrad_conv2d_grouped(dev16(dO), dev16(W), dD, layer.stride, layer.pad, layer.groups, n, m, scheme, seed=77,
                                   dtype=dtype, workspace=ws, flags=flags)
    assert sdgp.sdgp_last_device_error() == 0
    if flags == sdgp.FLAG_DENSE or n == m:
        src = dO
    else:
        src = oracle.prune(dO.reshape(-1, layer.Cout), n, m, scheme, 77, want=("dense",), dtype=dtype)["dense"].reshape(dO.shape)
    check(to_f16_f64(dD) if dtype == oracle.FP16 else to_f64(dD), src, W, layer, "%s flags=%d %d:%d" % (layer.name, flags, n, m), dtype)


REGNETX = {l.name: l for l in inputs.regnetx_400mf_layers(batch=3)}


@pytest.mark.parametrize("name", sorted(REGNETX))
@pytest.mark.parametrize("mode", ["two_pass", "dense"])
def test_regnetx_400mf_layers(name, mode):
    import paper_2202_00774_b200 as sdgp
    run(REGNETX[name], 2, 4, oracle.MAGNITUDE, sdgp.FLAG_TWO_PASS if mode == "two_pass" else sdgp.FLAG_DENSE)


GROUPED = [l for l in inputs.regnetx_400mf_layers(batch=2) if l.groups > 1]


@pytest.mark.parametrize("layer", GROUPED, ids=[l.name for l in GROUPED])
@pytest.mark.parametrize("n,m,scheme", [(1, 4, oracle.RESCALED), (2, 8, oracle.RANDOM), (2, 16, oracle.MAGNITUDE)])
def test_grouped_layers_other_patterns(layer, n, m, scheme):
    import paper_2202_00774_b200 as sdgp
    run(layer, n, m, scheme, sdgp.FLAG_TWO_PASS)


@pytest.mark.parametrize("layer", GROUPED, ids=[l.name for l in GROUPED])
def test_grouped_layers_masked(layer):
    import paper_2202_00774_b200 as sdgp
    run(layer, 4, 8, oracle.MAGNITUDE, sdgp.FLAG_MASKED)


@pytest.mark.parametrize("layer", [l for l in GROUPED if l.Cin % 64 == 0], ids=[l.name for l in GROUPED if l.Cin % 64 == 0])
def test_grouped_layers_fused(layer):
    import paper_2202_00774_b200 as sdgp
    run(layer, 2, 4, oracle.MAGNITUDE, sdgp.FLAG_FUSED)


def test_fused_refuses_padded_channel_counts():
    import paper_2202_00774_b200 as sdgp
    layer = inputs.ConvLayer("t", 1, 8, 8, 32, 32, 3, 3, 1, 1, 2)
    with pytest.raises(sdgp.SdgpError) as e:
        run(layer, 2, 4, oracle.MAGNITUDE, sdgp.FLAG_FUSED)
    assert e.value.status == 2      # SDGP_ERR_UNSUPPORTED


@pytest.mark.parametrize("B,H,Wd,Cin,Cout,R,S,stride,pad,groups", [
    (5, 14, 14, 160, 160, 3, 3, 1, 1, 10),     # several strips, ragged channel blocks on both sides
    (2, 28, 28, 96, 48, 3, 3, 2, 1, 3),        # 32 input and 16 output channels per group
    (4, 7, 7, 64, 128, 3, 3, 1, 1, 8),         # general kernel (7 x 7 images)
    (3, 16, 16, 40, 80, 1, 1, 1, 0, 1),        # no groups, channel counts that are multiples of 8 only
    (2, 12, 20, 128, 128, 3, 3, 1, 1, 1),      # groups == 1 with aligned channel counts: the ordinary path
])
def test_other_grouped_shapes(B, H, Wd, Cin, Cout, R, S, stride, pad, groups):
    import paper_2202_00774_b200 as sdgp
    layer = inputs.ConvLayer("case", B, H, Wd, Cin, Cout, R, S, stride, pad, groups)
    for flags in (sdgp.FLAG_TWO_PASS, sdgp.FLAG_DENSE):
        run(layer, 2, 4, oracle.MAGNITUDE, flags)


def test_argument_errors():
    import paper_2202_00774_b200 as sdgp
    layer = inputs.ConvLayer("t", 1, 8, 8, 32, 32, 3, 3, 1, 1, 2)
    dO, W = inputs.conv_layer_tensors(layer, seed=1)
    dD = torch.zeros(layer.dD_shape(), dtype=torch.int16, device="cuda")
    ws = torch.empty(1 << 20, dtype=torch.uint8, device="cuda")
    with pytest.raises(sdgp.SdgpError) as e:      # 3 groups do not divide 32 channels
        sdgp.sdgp_dgrad_conv2d_grouped(dev16(dO), dev16(W), dD, 1, 1, 3, 2, 4, sdgp.MAGNITUDE, workspace=ws)
    assert e.value.status == 1
    with pytest.raises(sdgp.SdgpError) as e:      # no workspace
        sdgp.sdgp_dgrad_conv2d_grouped(dev16(dO), dev16(W), dD, 1, 1, 2, 2, 4, sdgp.MAGNITUDE, workspace=None)
    assert e.value.status == 4
    with pytest.raises(sdgp.SdgpError) as e:      # 4 input channels per group: below one 16-byte vector
        sdgp.sdgp_dgrad_conv2d_grouped(dev16(dO), dev16(W[..., :4].copy()), dD, 1, 1, 8, 2, 4, sdgp.MAGNITUDE, workspace=ws)
    assert e.value.status == 2


# The kernel for narrow groups (16 or 32 channels on both sides): widths, partial blocks of 64 channels, lines shorter and longer than
# a round of units, odd and uneven images, filters with fewer and more taps, every group size of the pruning functions
@pytest.mark.parametrize("B,H,Wd,C,R,S,stride,pad,groups,n,m,scheme", [
    (1, 4, 4, 32, 3, 3, 1, 1, 2, 2, 4, oracle.MAGNITUDE),       # one unit, one block that is half empty
    (1, 5, 3, 48, 1, 3, 1, 0, 3, 1, 8, oracle.RESCALED),        # three slices of a block, one row of taps
    (3, 13, 27, 112, 3, 3, 2, 1, 7, 2, 4, oracle.RANDOM),       # four classes of uneven size
    (2, 9, 12, 96, 5, 5, 1, 2, 3, 2, 32, oracle.RESCALED),      # 25 taps of groups of 32 do not fit: the other path
    (2, 10, 7, 64, 3, 3, 1, 2, 4, 2, 16, oracle.RANDOM),        # padding of a whole filter: dL/dO is larger than dD
    (2, 11, 11, 160, 3, 3, 1, 0, 5, 2, 32, oracle.MAGNITUDE),   # no padding: dL/dO is smaller; groups of 32, two blocks and a half
    (1, 3, 260, 32, 3, 3, 1, 1, 2, 2, 4, oracle.MAGNITUDE),     # rows too long for a box: the other path
    (170, 14, 14, 176, 3, 3, 1, 1, 11, 2, 4, oracle.RESCALED),  # four units of every multiprocessor, a last block of 48 channels
])
def test_narrow_groups(B, H, Wd, C, R, S, stride, pad, groups, n, m, scheme):
    import paper_2202_00774_b200 as sdgp
    layer = inputs.ConvLayer("narrow", B, H, Wd, C, C, R, S, stride, pad, groups)
    run(layer, n, m, scheme, sdgp.FLAG_TWO_PASS)


# The last channel block of the strip kernel holds one to four MMAs' channels: every count, in tiles of one strip and of two, and in a last round
# that is dealt out strip by strip (176 images: 88 pair tiles of two strips on 74 pairs)
@pytest.mark.parametrize("B", [3, 176])
@pytest.mark.parametrize("Cout,mode", [(32, "two_pass"), (64, "two_pass"), (96, "two_pass"), (160, "two_pass"), (192, "two_pass"), (64, "fused"), (192, "fused"),
                                       (80, "dense"), (96, "dense"), (112, "dense"), (96, "masked")])
def test_last_channel_block_of_the_strip_kernel(B, Cout, mode):
    import paper_2202_00774_b200 as sdgp
    layer = inputs.ConvLayer("last", B, 16, 16, 64, Cout, 3, 3, 1, 1, 1)
    run(layer, 2, 4, oracle.MAGNITUDE, {"two_pass": sdgp.FLAG_TWO_PASS, "fused": sdgp.FLAG_FUSED, "dense": sdgp.FLAG_DENSE, "masked": sdgp.FLAG_MASKED}[mode])


# Plans and element types of the kernel for narrow groups (test_plan_host.py checks that these layers take it, and how): rings and accumulators
# that are used again, units of one to four accumulators, binary16 under every function
@pytest.mark.parametrize("case", [c for c, _ in plan_cases.NARROW])
def test_narrow_groups_plans(case):
    import paper_2202_00774_b200 as sdgp
    B, H, Wd, C, R, S, stride, pad, groups, n, m, scheme, fp16 = case
    run(inputs.ConvLayer("narrow", B, H, Wd, C, C, R, S, stride, pad, groups), n, m, scheme, sdgp.FLAG_TWO_PASS, dtype=oracle.FP16 if fp16 else oracle.BF16)


@pytest.mark.parametrize("case", [c for c in plan_cases.NARROW_ELSEWHERE if c[0] * c[1] * c[2] * c[3] < 3e6])
def test_narrow_groups_on_the_other_path(case):
    import paper_2202_00774_b200 as sdgp
    B, H, Wd, C, R, S, stride, pad, groups, n, m, scheme = case
    run(inputs.ConvLayer("elsewhere", B, H, Wd, C, C, R, S, stride, pad, groups), n, m, scheme, sdgp.FLAG_TWO_PASS)


@pytest.mark.parametrize("fp16", [False, True])
@pytest.mark.parametrize("case", [c for c, _ in plan_cases.BLOCK_DIAGONAL])
def test_block_diagonal_filters(case, fp16):
    import paper_2202_00774_b200 as sdgp
    B, H, Wd, Cin, Cout, R, S, stride, pad, groups, n, m, scheme = case
    run(inputs.ConvLayer("diagonal", B, H, Wd, Cin, Cout, R, S, stride, pad, groups), n, m, scheme, sdgp.FLAG_TWO_PASS,
        dtype=oracle.FP16 if fp16 else oracle.BF16)


# Infinities and NaN in dL/dO through the narrow-group kernel's own pruning: kept, pruned and rescaled as the oracle does, and felt by their group and
# the pixels under their taps only. (Filters are finite: a pruned position is a zero that meets its filter like any other.)
@pytest.mark.parametrize("fp16", [False, True])
@pytest.mark.parametrize("n,m,scheme", [(2, 4, oracle.MAGNITUDE), (1, 4, oracle.RESCALED), (2, 8, oracle.RESCALED), (2, 32, oracle.RESCALED), (2, 4, oracle.RANDOM)])
@pytest.mark.parametrize("stride,groups", [(1, 6), (2, 3)])
def test_narrow_groups_non_finite_gradients(n, m, scheme, stride, groups, fp16):
    import paper_2202_00774_b200 as sdgp
    dtype = oracle.FP16 if fp16 else oracle.BF16
    layer = inputs.ConvLayer("special", 2, 12, 11, 96, 96, 3, 3, stride, 1, groups)
    dO, W = inputs.conv_layer_tensors(layer, seed=5)
    if fp16:
        dO, W = inputs.bf16_bits_as_f16_bits(dO), inputs.bf16_bits_as_f16_bits(W)
    rng = np.random.Generator(np.random.PCG64(m + n))
    flat = dO.reshape(-1)
    for pattern in (0x7C00, 0xFC00, 0xFE01) if fp16 else (0x7F80, 0xFF80, 0xFFC1):
        flat[rng.integers(0, flat.size, 10)] = pattern
    src = oracle.prune(dO.reshape(-1, 96), n, m, scheme, 3, want=("dense",), dtype=dtype)["dense"].reshape(dO.shape)
    ref = oracle.dgrad_conv2d_grouped(src, W, layer.H, layer.W, groups, stride, 1, dtype=dtype)
    dD = torch.full(layer.dD_shape(), -1, dtype=torch.int16, device="cuda")
    ws = torch.empty(sdgp.sdgp_workspace_size_conv2d_grouped(2, 12, 11, 96, 96, 3, 3, stride, 1, groups, sdgp.FLAG_TWO_PASS), dtype=torch.uint8, device="cuda")
    sdgp.sdgp_dgrad_conv2d_grouped(dev16(dO), dev16(W), dD, stride, 1, groups, n, m, scheme, seed=3, dtype=dtype, workspace=ws)
    assert sdgp.sdgp_last_device_error() == 0
    got = to_f16_f64(dD) if fp16 else to_f64(dD)
    finite = np.isfinite(ref)
    assert (~finite).any() and finite.sum() > finite.size / 2
    assert np.array_equal(np.isnan(got), np.isnan(ref))
    assert np.array_equal(got[np.isinf(ref)], ref[np.isinf(ref)])
    special = magnitudes(src) >= (0x7C00 if fp16 else 0x7F80)
    absdot = oracle.dgrad_conv2d_grouped(np.where(special, 0, magnitudes(src)).astype(np.uint16), magnitudes(W), layer.H, layer.W, groups, stride, 1, dtype=dtype)
    bound = (2.0 ** -10 if fp16 else 2.0 ** -7) * np.abs(ref[finite]) + 2.0 ** -16 * absdot[finite] + (2.0 ** -24 if fp16 else 0.0)  # as in check()
    assert (np.abs(got[finite] - ref[finite]) <= bound).all()


# dD on a 16-byte boundary that is not a 32-byte one (rows leave in halves of a sector), nothing written outside it
@pytest.mark.parametrize("stride,C,groups", [(1, 96, 6), (2, 96, 3), (1, 64, 4)])
def test_narrow_groups_dD_on_a_16_byte_boundary(stride, C, groups):
    import paper_2202_00774_b200 as sdgp
    layer = inputs.ConvLayer("aligned", 3, 15, 10, C, C, 3, 3, stride, 1, groups)
    dO, W = inputs.conv_layer_tensors(layer, seed=4)
    size = int(np.prod(layer.dD_shape()))
    ws = torch.empty(sdgp.sdgp_workspace_size_conv2d_grouped(3, 15, 10, C, C, 3, 3, stride, 1, groups, sdgp.FLAG_TWO_PASS), dtype=torch.uint8, device="cuda")
    around = torch.full((size + 16,), -1, dtype=torch.int16, device="cuda")
    dD = around[8:8 + size].view(layer.dD_shape())
    assert dD.data_ptr() % 32 == 16
    aligned = torch.empty(layer.dD_shape(), dtype=torch.int16, device="cuda")
    for out in (dD, aligned):
        sdgp.sdgp_dgrad_conv2d_grouped(dev16(dO), dev16(W), out, stride, 1, groups, 2, 4, sdgp.MAGNITUDE, workspace=ws)
    assert sdgp.sdgp_last_device_error() == 0
    assert torch.equal(dD, aligned)
    assert bool((around[:8] == -1).all()) and bool((around[8 + size:] == -1).all())
    src = oracle.prune(dO.reshape(-1, C), 2, 4, oracle.MAGNITUDE, 0, want=("dense",))["dense"].reshape(dO.shape)
    check(to_f64(dD), src, W, layer, "16-byte dD")
