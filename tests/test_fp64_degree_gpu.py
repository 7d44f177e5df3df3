"""FP64 arithmetic of the DEGREE kernels (degree_f64_kernel) where its integer
products and conversions leave their range: points on the z axis and in the
x-y plane (zero factors), 1e-9 rad from a pole (c_m down to 1e-200, FP32
results that are subnormal or round to zero), at the origin and at very small
and large r; every lanes-per-point split, at degrees around the 16-channel
chunks and at the largest l_max."""

import numpy as np
import pytest
import torch

import oracle
from paper_2302_08381_gb300 import _capi as C
from paper_2302_08381_gb300 import api, inputs
from parity_utils import F64_TOL, assert_grads, assert_values

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _edge_points():
    d = 1e-9
    special = np.array([[0, 0, 1.0], [0, 0, -1.0], [1.0, 0, 0], [0, -1.0, 0], [0.6, 0.8, 0], [d, 0, 1.0],
                        [0, -d, 1.0], [d, d, -1.0], [1e-4, 0, 1.0], [0.6, 0, 0.8], [0, 0.6, -0.8]])
    return np.concatenate([special, inputs.pole_mix_points(37, seed=41).astype(np.float64)])


@pytest.mark.parametrize("lanes", [0, 1, 2, 4])
@pytest.mark.parametrize("l_max", [0, 1, 9, 15, 16, 17, 31, 32, 50])
def test_edge_points_match_oracle(l_max, lanes):
    x = _edge_points()
    for normalized, r in ((True, 1.0), (True, 1e-20), (True, 1e20), (False, 1.0)):
        p = x * r
        t = torch.from_numpy(p).to(DEV)
        v, g = api.spherical_harmonics(t, l_max, normalized, gradients=True, kernel="degree",
                                       launch=C.make_launch(0, 0, 0, lanes))
        rv, rg = oracle.spherical_harmonics_grad(p, l_max, normalized)
        assert_values(v.cpu().numpy(), p, l_max, normalized, F64_TOL, ref=rv)
        assert_grads(g.cpu().numpy(), p, l_max, normalized, F64_TOL, ref=rg)
        v0 = api.spherical_harmonics(t, l_max, normalized, kernel="degree", launch=C.make_launch(0, 0, 0, lanes))
        assert torch.equal(v0, v)


@pytest.mark.parametrize("lanes", [0, 1, 2, 4])
def test_origin_and_largest_degree(lanes):
    t = torch.from_numpy(np.concatenate([np.zeros((1, 3)), _edge_points()])).to(DEV)
    v, g = api.spherical_harmonics(t, 128, True, gradients=True, kernel="degree", launch=C.make_launch(0, 0, 0, lanes))
    ref, gref = api.spherical_harmonics(t, 128, True, gradients=True, kernel="slice")
    assert torch.all(v[0, 1:] == 0) and torch.all(g[0] == 0)
    assert float((v - ref).abs().max()) < 1e-10 and float(((g - gref) / 129.0).abs().max()) < 1e-10


@pytest.mark.parametrize("l_max", [3, 12, 30])
def test_fp32_storage_is_the_rounded_fp64_result(l_max):
    p = np.concatenate([_edge_points(), 1e-13 * _edge_points()]).astype(np.float32)
    for normalized in (False, True):
        launch = C.make_launch(0, 0, 0, 2)
        t = torch.from_numpy(p).to(DEV)
        a = api.spherical_harmonics(t, l_max, normalized, gradients=True, qprec="f64", kernel="degree", launch=launch)
        b = api.spherical_harmonics(t.double(), l_max, normalized, gradients=True, kernel="degree", launch=launch)
        for x32, x64 in zip(a, b):
            assert np.array_equal(x32.cpu().numpy(), x64.cpu().numpy().astype(np.float32))
