"""3-D FP32, two steps per fused pass with two rows a warp: the bits of one step per pass, at sizes whose tiles, strips and z
segments end ragged."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("periodic", [0, 1])
@pytest.mark.parametrize("full", [False, True])
@pytest.mark.parametrize("n", [(58, 101, 120), (29, 121, 90), (113, 122, 33)])
def test_two_rows_a_warp(n, full, periodic):
    import paper_1107_4650_gb300 as D
    from paper_1107_4650_gb300 import workloads as W
    nx, ny, nz = n
    psi = W.random_state(nz, ny, nx, sum(n)).astype(np.complex64)
    V = np.random.default_rng(nz).uniform(-1, 1, (nz, ny, nx) if full else nx) * W.C_AU ** 2

    def run(k):
        h = D.dirac_create_grid(D.make_config(n, ndim=3, precision=1, boundary=periodic, steps_per_launch=k, flux_face=nx // 2))
        try:
            D.dirac_set_potential(h, V, D.DIRAC_V_FULL if full else D.DIRAC_V_X_ONLY)
            D.dirac_set_state(h, psi)
            norm = D.dirac_observables(h)["norm"]
            D.dirac_step(h, 5)
            out = np.empty_like(psi)
            D.dirac_get_state(h, out)
            return out, D.dirac_observables(h)["flux_cum"], norm
        finally:
            D.dirac_destroy(h)

    want, fw, norm = run(1)
    got, fg, _ = run(0)
    assert np.array_equal(got.view(np.uint8), want.view(np.uint8))
    # FP32 sums of up to 32 terms and their squares: 40 roundings of 2^-24 a term, whose sizes add up to the norm a step
    assert abs(fw - fg) <= 2 * 40 * 2.0 ** -24 * 5 * norm
