"""POINT shapes installed for FP64 requests that AUTO otherwise runs on DEGREE by
the number of points: AUTO runs them, but not the autotuner's where DEGREE is
faster. Which kernel ran is told by its bits."""

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


def test_autotune_keeps_degree_where_it_is_faster(tmp_path):
    x = _x(60_000)
    auto = lambda: api.spherical_harmonics(x, 8, True, gradients=True)  # noqa: E731
    point, degree = (api.spherical_harmonics(x, 8, True, gradients=True, kernel=k) for k in ("point_hc", "degree"))
    C.sphericart_set_launch(8, C.SPH_F64, C.SPH_OUT_SAME, 1, C.make_launch(16, 1, 4, 0))
    shape, ms = api.autotune(x, 8, True, reps=1)  # DEGREE takes about 0.6 of the time here
    assert ms > 0 and _equal(auto(), degree)
    fam, s = C.sphericart_launch_info(8, C.SPH_F64, C.SPH_OUT_SAME, 1, 0)  # (of calls that name POINT_HC)
    assert fam == C.SPH_KERNEL_POINT_HC and s.points_per_tile == shape["points_per_tile"] > 0
    # a saved table keeps that; one without the last field installs for AUTO
    path = tmp_path / "tune.txt"
    api.save_tuning(str(path))
    C.sphericart_tune_clear()
    assert api.load_tuning(str(path)) == 1 and _equal(auto(), degree)
    line = path.read_text().split()
    assert len(line) == 10 and C.sphericart_tune_import(" ".join(line[:9])) == 1
    assert _equal(auto(), point)
