"""Each shape of the tile kernel that the library chooses (152 SMs), at a size that takes it: the library's choice is that shape, and
the steps, launches of its step count and the remainders, have the row kernel's bits."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# precision, second order, uniform field, (nx, nz), (warps, rows a warp, steps a launch)
SHAPES = [
    (0, 0, 0, (57, 41), (8, 1, 2)),
    (0, 0, 0, (128, 128), (12, 1, 2)),
    (0, 0, 0, (449, 200), (16, 1, 2)),
    (0, 0, 0, (149, 530), (20, 1, 1)),
    (0, 0, 0, (520, 384), (20, 1, 2)),
    (0, 0, 0, (301, 257), (24, 1, 2)),
    (0, 0, 1, (128, 128), (8, 1, 1)),
    (0, 0, 1, (200, 150), (12, 1, 1)),
    (0, 0, 1, (884, 67), (16, 1, 1)),
    (0, 1, 0, (57, 41), (8, 1, 1)),
    (0, 1, 0, (128, 128), (12, 1, 1)),
    (0, 1, 0, (700, 500), (16, 1, 1)),
    (0, 1, 0, (520, 384), (20, 1, 1)),
    (0, 1, 0, (301, 257), (24, 1, 1)),
    (0, 1, 1, (57, 41), (8, 1, 1)),
    (0, 1, 1, (128, 128), (12, 1, 1)),
    (0, 1, 1, (301, 257), (16, 1, 1)),
    (1, 0, 0, (200, 150), (8, 4, 4)),
    (1, 0, 0, (128, 128), (16, 1, 4)),
    (1, 0, 1, (128, 128), (8, 4, 2)),
    (1, 1, 0, (200, 150), (8, 4, 2)),
    (1, 1, 0, (128, 128), (16, 1, 2)),
    (1, 1, 1, (301, 257), (8, 4, 1)),
    (1, 1, 1, (128, 128), (16, 1, 1)),
    (2, 0, 0, (128, 128), (12, 1, 2)),
    (2, 0, 0, (700, 500), (16, 1, 2)),
    (2, 0, 0, (520, 384), (20, 1, 2)),
    (2, 0, 0, (301, 257), (24, 1, 2)),
    (2, 1, 0, (57, 41), (8, 1, 1)),
    (2, 1, 0, (128, 128), (12, 1, 1)),
    (2, 1, 0, (162, 350), (20, 1, 1)),
    (2, 1, 0, (301, 257), (24, 1, 1)),
]


@pytest.mark.parametrize("periodic", [0, 1])
@pytest.mark.parametrize("precision,strang,field,n,shape", SHAPES)
def test_shape_in_use_equals_rows(precision, strang, field, n, shape, periodic):
    import torch

    import paper_1107_4650_gb300 as D
    from paper_1107_4650_gb300 import workloads as W
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("the sizes are those of 152 SMs")
    nx, nz = n
    warps, rows, steps = shape
    H = steps * (1 + strang)
    rng = np.random.default_rng(nx + nz)
    psi = W.random_state(nz, 1, nx, nx + nz).astype(np.complex64 if precision == 1 else np.complex128)
    V = rng.uniform(-1, 1, nx) * W.C_AU ** 2
    A = rng.uniform(-1, 1, (8, 3))

    def run(k, p):
        h = D.dirac_create_grid(D.make_config((nx, 1, nz), precision=precision, splitting=strang, boundary=periodic,
                                              steps_per_launch=k, points_per_lane=p, flux_face=nx // 2))
        try:
            D.dirac_set_potential(h, V, D.DIRAC_V_X_ONLY)
            if field:
                D.dirac_set_vector_potential(h, A)
            D.dirac_set_state(h, psi)
            D.dirac_step(h, 2 * steps - 1)
            out = np.empty_like(psi)
            D.dirac_get_state(h, out)
            return out, D.dirac_get_info(h)
        finally:
            D.dirac_destroy(h)

    got, info = run(0, 0)
    tiles = -(-nx // (32 - 2 * H)) * -(-nz // (warps * rows - 2 * H))
    assert (info["steps_per_launch"], info["strip_width"], info["segment_rows"], info["launch_warps"]) == (
        steps, 32 - 2 * H, warps * rows - 2 * H, tiles * warps)
    want, _ = run(1, 2)
    assert np.array_equal(got.view(np.uint8), want.view(np.uint8))
