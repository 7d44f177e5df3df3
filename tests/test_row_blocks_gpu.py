"""ROW kernels in blocks of many warps that share one coefficient table: the
default shape (several warps per block once there are more tiles than SMs)
against one-warp blocks, bit for bit, at the smallest and largest l_max of
every channel count, with a ragged last tile."""

import pytest
import torch

from paper_2302_08381_gb300 import _capi as C
from paper_2302_08381_gb300 import api

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _points(n):
    gen = torch.Generator(device=DEV).manual_seed(7)
    return torch.randn(n, 3, generator=gen, device=DEV)


@pytest.mark.parametrize("l_max", [16, 23, 24, 27, 28, 31, 32, 39, 40, 47, 48, 55, 56, 63])
@pytest.mark.parametrize("out_dtype", [torch.float32, torch.bfloat16])
def test_default_blocks_equal_one_warp_blocks(l_max, out_dtype):
    one = C.make_launch(0, 1, 0, 0)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for n in (1, 4 * sms + 3, 4 * sms * 3 + 1, 4 * sms * 20 + 2):
        x = _points(n)
        for grad in (True, False):
            a = api.spherical_harmonics(x, l_max, True, gradients=grad, out_dtype=out_dtype, kernel="row")
            b = api.spherical_harmonics(x, l_max, True, gradients=grad, out_dtype=out_dtype, kernel="row", launch=one)
            for s, t in zip(a if grad else (a,), b if grad else (b,)):
                assert torch.equal(s, t), (l_max, n, grad)
        if out_dtype == torch.float32:
            g = torch.randn(n, (l_max + 1) ** 2, device=DEV)
            assert torch.equal(api.backward(x, g, l_max, True, kernel="row"),
                               api.backward(x, g, l_max, True, kernel="row", launch=one))
    assert api.device_status() == 0
