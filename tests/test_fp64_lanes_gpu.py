"""FP64 DEGREE results of a point do not depend on the lanes it is given, and so
neither on the number of points in the call, which AUTO chooses the lanes by."""

import pytest
import torch

from paper_2302_08381_gb300 import _capi as C
from paper_2302_08381_gb300 import api

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("normalized", [False, True])
@pytest.mark.parametrize("l_max", [0, 1, 3, 8, 9, 16, 17, 31, 50])
def test_lanes_and_number_of_points_give_the_same_bits(l_max, normalized):
    gen = torch.Generator(device=DEV).manual_seed(l_max)
    x = torch.randn(40_000 if l_max < 20 else 9_000, 3, generator=gen, device=DEV, dtype=torch.float64)
    x = x / x.norm(dim=1, keepdim=True) * (0.8 + 0.4 * torch.rand(len(x), 1, generator=gen, device=DEV))
    for dtype, kw in ((torch.float64, {}), (torch.float32, {"qprec": "f64"})):
        p = x.to(dtype)
        for grad in (False, True):
            ref = api.spherical_harmonics(p, l_max, normalized, gradients=grad, kernel="degree", **kw)
            for lanes in (0, 1, 2, 4):
                for n in (1, 300, 5000):
                    out = api.spherical_harmonics(p[:n].contiguous(), l_max, normalized, gradients=grad,
                                                  kernel="degree", launch=C.make_launch(0, 0, 0, lanes), **kw)
                    for u, v in zip(out if grad else (out,), ref if grad else (ref,)):
                        assert torch.equal(u, v[:n]), (dtype, grad, lanes, n)
