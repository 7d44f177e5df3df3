"""Explicit ROW shapes: warps_per_block x blocks_per_sm warps on an SM, in
blocks of as many of them as fit, against the default shape bit for bit, with
one round of tiles, several, and a last one that is spread over the blocks."""

import pytest
import torch

from paper_2302_08381_gb300 import _capi as C
from paper_2302_08381_gb300 import api

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("l_max", [16, 31, 40, 63])
def test_explicit_shapes_equal_the_default(l_max):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    gen = torch.Generator(device=DEV).manual_seed(l_max)
    for n in (1, 4 * sms - 1, 4 * sms * 4 * 3 + 5, 4 * sms * 16 + 4 * sms // 2 + 1):
        x = torch.randn(n, 3, generator=gen, device=DEV)
        g = torch.randn(n, (l_max + 1) ** 2, generator=gen, device=DEV)
        fwd = [api.spherical_harmonics(x, l_max, True, gradients=True, out_dtype=t, kernel="row")
               for t in (None, torch.bfloat16)]
        bwd = api.backward(x, g, l_max, True, kernel="row")
        for W, B in ((1, 1), (2, 1), (1, 3), (2, 2), (2, 32), (1, 0), (0, 2)):
            launch = C.make_launch(0, W, B, 0)
            for t, ref in zip((None, torch.bfloat16), fwd):
                out = api.spherical_harmonics(x, l_max, True, gradients=True, out_dtype=t, kernel="row", launch=launch)
                assert all(torch.equal(a, b) for a, b in zip(out, ref)), (n, W, B, t)
        for W, B in ((1, 1), (8, 1), (3, 2), (8, 32), (8, 0), (0, 2)):
            assert torch.equal(api.backward(x, g, l_max, True, kernel="row", launch=C.make_launch(0, W, B, 0)), bwd)
    assert api.device_status() == 0
