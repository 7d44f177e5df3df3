"""Forward from host buffers in FP64: the bits of the device path for every
chunking, where AUTO's kernel depends on the number of points and where not."""

import pytest
import torch

from paper_2302_08381_gb300 import api

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("l_max,n", [(5, 3000), (5, 20_000), (6, 9000), (8, 10_000), (8, 20_000), (12, 33_000), (20, 8000)])
@pytest.mark.parametrize("normalized", [False, True])
def test_fp64_chunks_have_the_bits_of_the_whole(l_max, n, normalized):
    x = torch.randn(n, 3, dtype=torch.float64, generator=torch.Generator().manual_seed(l_max)).pin_memory()
    rv, rg = api.spherical_harmonics(x.cuda(), l_max, normalized, gradients=True)
    values = api.spherical_harmonics(x.cuda(), l_max, normalized).cpu()
    for chunk in (0, 224, 4000, 8192, 15_000):
        v, g = api.spherical_harmonics_host(x, l_max, normalized, gradients=True, chunk_points=chunk)
        only = api.spherical_harmonics_host(x, l_max, normalized, chunk_points=chunk)
        torch.cuda.synchronize()
        assert torch.equal(v, rv.cpu()) and torch.equal(g, rg.cpu()), chunk
        assert torch.equal(only, values), chunk
