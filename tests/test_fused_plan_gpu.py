"""The 3-D FP32 grids of test_fused_rows_gpu.py take the form with two rows a warp (24-row tiles, 20 of them owned)."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(58, 101, 120), (29, 121, 90), (113, 122, 33)])
def test_two_rows_a_warp_in_use(n):
    import torch

    import paper_1107_4650_gb300 as D
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("the sizes are those of 152 SMs")
    h = D.dirac_create_grid(D.make_config(n, ndim=3, precision=D.DIRAC_FP32))
    try:
        info = D.dirac_get_info(h)
    finally:
        D.dirac_destroy(h)
    segments = -(-n[2] // info["segment_rows"])
    blocks = -(-n[0] // 28) * -(-n[1] // 20) * segments
    assert (info["steps_per_launch"], info["strip_width"], info["launch_warps"]) == (2, 28, 12 * blocks)
