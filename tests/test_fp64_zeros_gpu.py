"""FP64 arithmetic of the DEGREE kernels at points with zero coordinates: the
integer products take the zero factors themselves. Bit for bit what the FP64
pipe gives, which runs in tiles that also hold a point out of the integer
products' range."""

import numpy as np
import pytest
import torch

from paper_2302_08381_gb300 import _capi as C
from paper_2302_08381_gb300 import api

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _points(normalized):
    rng = np.random.default_rng(61)
    x = rng.uniform(0.3, 1.4, (211, 3)) * rng.choice([-1.0, 1.0], (211, 3))
    for i, zero in enumerate([(2,), (1,), (0,), (0, 1), (0, 2), (1, 2), ()]):
        x[np.ix_(np.arange(i, len(x), 7), list(zero))] = 0.0
    x[::5] *= np.where(x[::5] == 0, -1.0, 1.0)  # some of the zeros negative
    forced = x.copy()
    out = np.array([[1.0, 0.3, 1e-100], [1e-160, 1e-160, 1.0]]) if normalized else np.array([[1e95, 2e95, 3e95]] * 2)
    forced[3::4] = out[np.arange(len(x[3::4])) % 2]  # a tile holds at least 4 points
    return x, forced, np.arange(len(x)) % 4 != 3


@pytest.mark.parametrize("normalized", [False, True])
@pytest.mark.parametrize("lanes", [0, 1, 2, 4])
@pytest.mark.parametrize("l_max", [0, 1, 8, 17, 33])
def test_zero_coordinates_equal_the_fp64_pipe(l_max, lanes, normalized):
    x, forced, keep = _points(normalized)
    launch = C.make_launch(0, 0, 0, lanes)
    for dtype, kw in ((torch.float64, {}), (torch.float32, {"qprec": "f64"})):
        if dtype == torch.float32 and not normalized:
            continue  # (the forcing points lie beyond FP32)
        for grad in (False, True):
            a, b = (api.spherical_harmonics(torch.from_numpy(p).to(DEV, dtype), l_max, normalized, gradients=grad,
                                            kernel="degree", launch=launch, **kw) for p in (x, forced))
            for u, v in zip(a if grad else (a,), b if grad else (b,)):
                assert torch.isfinite(u[keep]).all()
                assert torch.equal(u[keep], v[keep])
