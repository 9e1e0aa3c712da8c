"""Rows per segment that the launch planner chooses (152 SMs), where a change of its model had made steps slower: the host runtime
on the stand-in for the CUDA runtime."""
import pytest

import paper_1107_4650_gb300 as D
from tests.test_graph_changes import fake, fake_lib  # noqa: F401


def _rows(field=False, **cfg):
    import numpy as np
    h = D.dirac_create_grid(D.make_config(**cfg))
    try:
        if field:
            D.dirac_set_vector_potential(h, np.zeros((4, 3)))
        return D.dirac_get_info(h)["segment_rows"]
    finally:
        D.dirac_destroy(h)


@pytest.mark.parametrize("n,field,lo,hi", [((2048, 1, 2048), False, 61, 64), ((1024, 1, 1024), True, 16, 17),
                                           ((777, 1, 1000), False, 11, 12), ((1500, 1, 1100), False, 22, 24)])
def test_fp64_second_order_two_points_a_lane(fake, n, field, lo, hi):  # noqa: F811
    assert lo <= _rows(field, n=n, splitting=D.DIRAC_STRANG, points_per_lane=2, steps_per_launch=1) <= hi


@pytest.mark.parametrize("shift,n,lo,hi", [(3, (2048, 1, 2048), 63, 66), (4, (2048, 1, 2048), 63, 66), (3, (1800, 1, 1700), 45, 48),
                                           (4, (1800, 1, 1700), 48, 52)])
def test_fp32_shifts_fill_one_wave(fake, shift, n, lo, hi):  # noqa: F811
    """Two blocks of four warps fit an SM: segments whose warps fill 2 x 152 blocks once."""
    assert lo <= _rows(n=n, precision=D.DIRAC_FP32, char_shift=shift) <= hi


@pytest.mark.parametrize("n,lo,hi", [((1024, 1, 1024), 8, 11), ((520, 1, 384), 2, 3)])
def test_fixed_point_four_points_a_lane(fake, n, lo, hi):  # noqa: F811
    assert lo <= _rows(n=n, precision=D.DIRAC_FX64, points_per_lane=4, steps_per_launch=1) <= hi
