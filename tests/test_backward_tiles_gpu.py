"""POINT double backward and backward when every warp runs several tiles: the
reuse of the staged buffers (one, two, grad_g in place or apart, rows of one
16-byte unit), for upstream gradients and grad_g on and off 16 bytes."""

import functools

import numpy as np
import pytest
import torch

import oracle
from paper_2302_08381_gb300 import _capi as C
from paper_2302_08381_gb300 import api, inputs

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
TILES = 3  # per warp, the last one ragged


@functools.lru_cache(maxsize=1)
def _case(l_max, normalized, n):
    x = inputs.shell_points(n, 0.7, 3.0, seed=801).astype(np.float32).astype(np.float64)
    g = inputs.upstream(n, (l_max + 1) ** 2, seed=802).astype(np.float32).astype(np.float64)
    v = inputs.upstream(n, 3, seed=803).astype(np.float32).astype(np.float64)
    return x, g, v, oracle.double_backward(x, g, v, l_max, normalized), oracle.backward(x, g, l_max, normalized)


def _at(a, off):
    """The contiguous CUDA copy of `a`, `off` elements past a 16-byte boundary."""
    buf = torch.empty(a.numel() + 4, dtype=a.dtype, device=DEV)
    out = buf[off: off + a.numel()].view(a.shape)
    out.copy_(a)
    return out


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("normalized", [False, True])
@pytest.mark.parametrize("l_max", [0, 1, 3, 4, 6, 7, 8, 10, 11, 12, 16])
def test_many_tiles_per_warp(l_max, normalized, dtype):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = 32 * sms * TILES + 5
    x_np, g_np, v_np, (rgg, rgx), rdx = _case(l_max, normalized, n)
    x, v = (torch.from_numpy(a).to(DEV, dtype) for a in (x_np, v_np))
    code = C.SPH_F32 if dtype == torch.float32 else C.SPH_F64
    launch = C.make_launch(32, 1, 1, 0)  # one warp per SM
    stream = torch.cuda.current_stream().cuda_stream
    tol_g, tol_x = (2e-5, 1e-4) if dtype == torch.float32 else (1e-12, 1e-12)
    floor = 1e-3 * np.max(np.abs(g_np)) * np.max(np.abs(v_np))
    base = None
    for off_g in (0, 1):
        g = _at(torch.from_numpy(g_np).to(dtype), off_g)
        dx = api.backward(x, g, l_max, normalized, kernel="point", launch=launch).double().cpu().numpy()
        assert np.max(np.abs(dx - rdx)) <= tol_g * max(np.max(np.abs(rdx)), 1e-3)
        for off_o in (0, 1):
            for need_g, need_x in ((True, True), (True, False), (False, True)):
                gg = _at(torch.full_like(g, -7.0), off_o) if need_g else None
                gx = torch.full_like(x, -7.0) if need_x else None
                C.sphericart_double_backward(
                    x.data_ptr(), g.data_ptr(), v.data_ptr(), n, l_max, int(normalized), code, C.SPH_KERNEL_POINT,
                    launch, gg.data_ptr() if need_g else None, gx.data_ptr() if need_x else None, stream)
                if base is None:
                    base = (gg.clone(), gx.clone())
                    e = np.max(np.abs(gg.double().cpu().numpy() - rgg)) / max(np.max(np.abs(rgg)), 1e-3)
                    assert e <= tol_g, e
                    e = np.max(np.abs(gx.double().cpu().numpy() - rgx)) / max(np.max(np.abs(rgx)), floor)
                    assert e <= tol_x, e
                assert gg is None or torch.equal(gg, base[0]), (off_g, off_o, need_x)
                assert gx is None or torch.equal(gx, base[1]), (off_g, off_o, need_g)
    assert api.device_status() == 0
