"""AUTO where its kernel goes by the number of points: on both sides of every
bound it runs the family that the bound names (told by the bits), and that
family is right there."""

import numpy as np
import pytest
import torch

import oracle
from paper_2302_08381_gb300 import api
from parity_utils import F64_TOL, assert_grads, assert_values

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _x(n, dtype=torch.float64):
    gen = torch.Generator(device=DEV).manual_seed(n)
    x = torch.randn(n, 3, generator=gen, device=DEV, dtype=torch.float64)
    return (x / x.norm(dim=1, keepdim=True) * (0.8 + 0.4 * torch.rand(n, 1, generator=gen, device=DEV))).to(dtype)


@pytest.mark.parametrize("l_max,normalized,grad,n,degree", [
    (8, False, True, 255, False), (8, False, True, 256, True), (8, False, True, 8192, True),
    (8, False, True, 8193, False), (7, False, True, 12_288, False), (7, False, True, 12_289, True),
    (7, True, True, 10_000, True), (5, False, True, 4096, True), (6, False, True, 4097, False),
    (6, True, True, 8192, True), (5, True, True, 8193, False), (4, True, True, 1000, False),
    (11, True, False, 32_767, False), (13, False, False, 32_768, True), (10, True, False, 40_000, False),
])
def test_fp64_bounds(l_max, normalized, grad, n, degree):
    x = _x(n)
    out = api.spherical_harmonics(x, l_max, normalized, gradients=grad)
    want = api.spherical_harmonics(x, l_max, normalized, gradients=grad,
                                   kernel="degree" if degree else ("point_hc" if grad else "point"))
    out, want = (t if grad else (t,) for t in (out, want))
    assert all(torch.equal(a, b) for a, b in zip(out, want))
    s = np.r_[0:40, n - 41:n]
    p = x.cpu().numpy()[s]
    rv, rg = oracle.spherical_harmonics_grad(p, l_max, normalized)
    assert_values(out[0].cpu().numpy()[s], p, l_max, normalized, F64_TOL, ref=rv)
    if grad:
        assert_grads(out[1].cpu().numpy()[s], p, l_max, normalized, F64_TOL, ref=rg)


@pytest.mark.parametrize("l_max,grad,n,degree", [(3, True, 8191, True), (4, True, 8192, False), (4, False, 100, False),
                                                 (4, True, 65_535, False), (4, True, 65_536, True),
                                                 (2, True, 100, False), (5, True, 9000, True)])
def test_mixed_bounds(l_max, grad, n, degree):
    x = _x(n, torch.float32)
    run = lambda **k: api.spherical_harmonics(x, l_max, True, gradients=grad, qprec="f64", **k)  # noqa: E731
    out, want = run(), run(kernel="degree")
    # the other kernel (POINT_HC in FP64) rounds some of its FP32 results the other way
    out, want = (t if grad else (t,) for t in (out, want))
    same = all(torch.equal(a, b) for a, b in zip(out, want))
    assert same or not degree
    p = x.double().cpu().numpy()
    rv, rg = oracle.spherical_harmonics_grad(p, l_max, True)
    assert_values(out[0].double().cpu().numpy(), p, l_max, True, 2.0 ** -24 + F64_TOL, ref=rv)
    if grad:
        assert_grads(out[1].double().cpu().numpy(), p, l_max, True, 4 * 2.0 ** -24, ref=rg)
