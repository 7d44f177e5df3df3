"""POINT shapes installed for FP64 requests that AUTO otherwise runs on DEGREE by
the number of points: AUTO runs them, and the autotuner installs none where
DEGREE is faster. Which kernel ran is told by its bits."""

import pytest
import torch

from paper_2302_08381_gb300 import _capi as C
from paper_2302_08381_gb300 import api

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(autouse=True)
def _restore_defaults():
    yield
    C.sphericart_tune_clear()


def _x(n):
    gen = torch.Generator(device=DEV).manual_seed(n)
    return torch.randn(n, 3, generator=gen, device=DEV, dtype=torch.float64)


def _equal(a, b):
    a, b = (t if isinstance(t, tuple) else (t,) for t in (a, b))
    return all(torch.equal(u, v) for u, v in zip(a, b))


@pytest.mark.parametrize("l_max,n,grad", [(8, 20_000, True), (7, 300, True), (5, 1000, True), (12, 33_000, False)])
def test_auto_runs_an_installed_shape(l_max, n, grad):
    x = _x(n)
    point = api.spherical_harmonics(x, l_max, True, gradients=grad, kernel="point_hc" if grad else "point")
    degree = api.spherical_harmonics(x, l_max, True, gradients=grad, kernel="degree")
    assert not _equal(point, degree)
    auto = lambda: api.spherical_harmonics(x, l_max, True, gradients=grad)  # noqa: E731
    assert _equal(auto(), degree)
    C.sphericart_set_launch(l_max, C.SPH_F64, C.SPH_OUT_SAME, int(grad), C.make_launch(16, 1, 4, 0))
    assert _equal(auto(), point)
    C.sphericart_tune_clear()
    assert _equal(auto(), degree)


def test_autotune_keeps_degree_where_it_is_faster():
    x = _x(60_000)
    C.sphericart_set_launch(8, C.SPH_F64, C.SPH_OUT_SAME, 1, C.make_launch(16, 1, 4, 0))
    shape, ms = api.autotune(x, 8, True, reps=1)  # DEGREE takes about 0.6 of the time here
    assert ms > 0 and not any(shape.values())
    assert _equal(api.spherical_harmonics(x, 8, True, gradients=True),
                  api.spherical_harmonics(x, 8, True, gradients=True, kernel="degree"))
    shape, ms = api.autotune(x, 4, True, reps=1)  # (AUTO: POINT)
    assert ms > 0 and shape["points_per_tile"] > 0
