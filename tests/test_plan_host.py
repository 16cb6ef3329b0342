"""The choice of kernel as a function of sizes (sdgp_selftest_plan; no GPU): the layers of plan_cases.py take the paths that their GPU tests are for."""
import ctypes

import pytest

import plan_cases

SMS = 148


def plan(B, H, W, Cin, Cout, R, S, stride, pad, groups, n, m, scheme, flags=plan_cases.TWO_PASS):
    from paper_2202_00774_b200 import binding
    out = (ctypes.c_int * 8)()
    assert binding.lib().sdgp_selftest_plan(B, H, W, Cin, Cout, R, S, stride, pad, groups, n, m, scheme, flags, out) == 0
    return list(out)


@pytest.mark.parametrize("case,expected", plan_cases.NARROW)
def test_narrow_groups_take_their_kernel(case, expected):
    B, H, W, C, R, S, stride, pad, groups, n, m, scheme, _ = case
    route, units, tiles, classes, stages, _, _, _ = plan(B, H, W, C, C, R, S, stride, pad, groups, n, m, scheme)
    assert route == 1 and classes == stride * stride
    assert (tiles, -(-units // SMS), stages) == expected


@pytest.mark.parametrize("case", plan_cases.NARROW_ELSEWHERE)
def test_narrow_groups_that_other_kernels_are_faster_on(case):
    B, H, W, C, R, S, stride, pad, groups, n, m, scheme = case
    assert plan(B, H, W, C, C, R, S, stride, pad, groups, n, m, scheme)[0] == 0


@pytest.mark.parametrize("case,route", plan_cases.BLOCK_DIAGONAL)
def test_other_grouped_layers(case, route):
    assert plan(*case)[0] == route


@pytest.mark.parametrize("flags", [plan_cases.TWO_PASS, plan_cases.DENSE])
@pytest.mark.parametrize("case,dealt_out,below", plan_cases.PARITIES)
def test_parities_in_one_launch(case, dealt_out, below, flags):
    B, H, W, Cin, Cout, R, S, pad = case
    route, units, split_from, pairs, bn, nt, images, _ = plan(B, H, W, Cin, Cout, R, S, 2, pad, 1, 2, 4, plan_cases.MAGNITUDE, flags)
    assert route == 2 and pairs == min(units, SMS // 2) and nt in (1, 2) and bn * nt <= 256
    assert (split_from < units) == dealt_out
    rows = 16 // images
    assert ((H + 1) // 2 > H // 2 and (H // 2) % rows == 0) == below


def test_arguments():
    from paper_2202_00774_b200 import binding
    out = (ctypes.c_int * 8)()
    f = binding.lib().sdgp_selftest_plan
    assert f(1, 8, 8, 32, 32, 3, 3, 1, 1, 2, 2, 4, 1, 0, None) == 1
    assert f(1, 8, 8, 32, 32, 3, 3, 3, 1, 2, 2, 4, 1, 0, out) == 1      # stride
    assert f(1, 8, 8, 32, 32, 3, 3, 1, 1, 3, 2, 4, 1, 0, out) == 1      # groups
    assert f(1, 8, 8, 32, 32, 3, 3, 1, 3, 2, 2, 4, 1, 0, out) == 1      # padding
    assert f(1, 8, 8, 32, 32, 3, 3, 1, 1, 2, 2, 4, 1, 1, out) == 0 and list(out) == [0] * 8
