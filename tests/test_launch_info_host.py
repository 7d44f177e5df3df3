"""launch_info reports the shapes that the kernels run, without a GPU."""

import pytest

from paper_2302_08381_gb300 import _capi as C


def test_row_blocks():
    """ROW: as many warps as fit one block per SM (0), its Hessians one or two."""
    for l_max in (17, 40, 63):
        for out in (C.SPH_OUT_SAME, C.SPH_OUT_BF16):
            fam, s = C.sphericart_launch_info(l_max, C.SPH_F32, out, 1, 0)
            assert fam == C.SPH_KERNEL_ROW and (s.warps_per_block, s.lanes_per_point) == (0, 8)
    for l_max, warps in ((17, 1), (39, 1), (40, 2), (63, 2)):
        fam, s = C.sphericart_launch_info(l_max, C.SPH_F32, C.SPH_OUT_SAME, 1, 1)
        assert fam == C.SPH_KERNEL_ROW and (s.warps_per_block, s.lanes_per_point) == (warps, 8)


@pytest.mark.parametrize("l_max,grad,lanes", [(9, 1, 2), (12, 1, 4), (26, 1, 4), (27, 1, 8), (128, 1, 8),
                                              (14, 0, 2), (20, 0, 4), (44, 0, 4), (45, 0, 8)])
def test_fp64_degree_lanes(l_max, grad, lanes):
    fam, s = C.sphericart_launch_info(l_max, C.SPH_F64, C.SPH_OUT_SAME, grad, 0)
    assert fam == C.SPH_KERNEL_DEGREE and s.lanes_per_point == lanes


def test_fp32_degree_lanes():
    fam, s = C.sphericart_launch_info(100, C.SPH_F32, C.SPH_OUT_BF16, 1, 0)
    assert fam == C.SPH_KERNEL_DEGREE and s.lanes_per_point == 4
