"""FP64 DEGREE at points with an infinite or NaN coordinate: Qtilde is NaN there,
and every value and derivative that has it, or the bad coordinate, for a factor
is NaN, also where the other factor is zero by its place. The points beside it
are what they are alone."""

import itertools

import numpy as np
import pytest
import torch

from paper_2302_08381_gb300 import _capi as C
from paper_2302_08381_gb300 import api

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _must_be_nan(l_max, bad):
    """[3, K] of the scaled form; `bad`: the coordinates that are not finite."""
    out = np.ones((3, (l_max + 1) ** 2), bool)
    for l in range(l_max + 1):
        for m in range(-l, l + 1):
            k = l * l + l + m
            if m == 0 and l <= 1:  # x, y times a factor that is zero by its place
                out[0, k], out[1, k] = 0 in bad, 1 in bad
            if abs(m) == l and (l <= 1 or bad == {2}):  # zero times c_m, s_m
                out[2, k] = False
    return out


@pytest.mark.parametrize("value", [float("nan"), float("inf"), -float("inf")])
@pytest.mark.parametrize("l_max", [0, 1, 2, 9, 17])
def test_nonfinite_coordinates(l_max, value):
    rng = np.random.default_rng(l_max)
    clean = rng.uniform(0.4, 1.2, (40, 3)) * rng.choice([-1.0, 1.0], (40, 3))
    x, bads = clean.copy(), {}
    for i, bad in enumerate(itertools.chain.from_iterable(itertools.combinations(range(3), r) for r in (1, 2, 3))):
        x[5 * i, list(bad)] = value
        bads[5 * i] = set(bad)
    good = [i for i in range(40) if i not in bads]
    for normalized, lanes, (dtype, kw) in itertools.product(
            (False, True), (0, 1, 2, 4), ((torch.float64, {}), (torch.float32, {"qprec": "f64"}))):
        run = lambda p, **k: api.spherical_harmonics(  # noqa: E731
            torch.from_numpy(p).to(DEV, dtype), l_max, normalized, kernel="degree",
            launch=C.make_launch(0, 0, 0, lanes), **k, **kw)
        v, g = (t.cpu().numpy() for t in run(x, gradients=True))
        cv, cg = (t.cpu().numpy() for t in run(clean, gradients=True))
        assert np.isnan(run(x).cpu().numpy()[list(bads)]).all()
        for i, bad in bads.items():
            assert np.isnan(v[i]).all(), (normalized, lanes, bad)
            need = np.ones_like(g[i], bool) if normalized else _must_be_nan(l_max, bad)
            assert np.isnan(g[i][need]).all(), (normalized, lanes, bad)
        assert np.array_equal(v[good], cv[good]) and np.array_equal(g[good], cg[good])
