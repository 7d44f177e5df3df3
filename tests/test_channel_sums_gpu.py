"""POINT backward and double backward by channel sums: normalized and scaled
points on the axes, next to the poles and at the origin (where A, B, C of
m = 1 and 2 meet c_0, s_0 and vanishing c_m), odd and even row strides."""

import numpy as np
import pytest
import torch

import oracle
from paper_2302_08381_gb300 import api, inputs
from parity_utils import F64_TOL

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("normalized", [False, True])
@pytest.mark.parametrize("l_max", [0, 1, 2, 3, 5, 6, 11, 16])
def test_edge_points_match_oracle(l_max, normalized):
    x = np.concatenate([np.array([[0, 0, 1.0], [0, 0, -2.0], [1.5, 0, 0], [0, -1.0, 0], [0.6, 0.8, 0], [1e-9, 0, 1.0]]),
                        inputs.pole_mix_points(60, seed=51).astype(np.float64) * 1.3])
    K = (l_max + 1) ** 2
    g = inputs.upstream(len(x), K, seed=52).astype(np.float64)
    v = inputs.upstream(len(x), 3, seed=53).astype(np.float64)
    t = [torch.from_numpy(a).to(DEV) for a in (x, g, v)]
    ref = oracle.backward(x, g, l_max, normalized)
    dx = api.backward(t[0], t[1], l_max, normalized, kernel="point").cpu().numpy()
    assert np.max(np.abs(dx - ref)) <= F64_TOL * max(np.max(np.abs(ref)), 1e-3)
    rgg, rgx = oracle.double_backward(x, g, v, l_max, normalized)
    gg, gx = api.double_backward(*t, l_max, normalized, kernel="point")
    floor = 1e-3 * np.max(np.abs(g)) * np.max(np.abs(v))
    assert np.max(np.abs(gg.cpu().numpy() - rgg)) <= F64_TOL * max(np.max(np.abs(rgg)), 1e-3)
    assert np.max(np.abs(gx.cpu().numpy() - rgx)) <= F64_TOL * max(np.max(np.abs(rgx)), floor)


@pytest.mark.parametrize("normalized", [False, True])
def test_origin(normalized):
    x = torch.zeros(40, 3, device=DEV)
    g, v = torch.randn(40, 49, device=DEV), torch.randn(40, 3, device=DEV)
    dx = api.backward(x, g, 6, normalized, kernel="point")
    gg, gx = api.double_backward(x, g, v, 6, normalized, kernel="point")
    if normalized:
        assert not dx.any() and not gg.any() and not gx.any()
    else:  # only the linear harmonics have a gradient there, only the quadratic ones a Hessian
        assert torch.equal(gg[:, 4:], torch.zeros_like(gg[:, 4:])) and torch.isfinite(gx).all() and dx.any()
