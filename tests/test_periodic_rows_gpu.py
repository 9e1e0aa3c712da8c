"""Periodic 2-D steps through the row ring: rows copied as wrapped pieces, on grids narrower than a warp's strip, just
past its edges and with fewer rows than the halo, against the oracle."""
import numpy as np
import pytest

import oracle
from paper_1107_4650_gb300 import workloads as W

pytestmark = pytest.mark.gpu
DX, C = W.DX_DEFAULT, W.C_AU
SIZES = [(1, 1), (2, 3), (5, 40), (28, 2), (30, 33), (31, 17), (32, 16), (33, 5), (62, 31), (64, 20), (65, 64), (131, 35)]


def _run(D, n, psi, V, steps, **kw):
    h = D.dirac_create_grid(D.make_config((n[0], 1, n[1]), boundary=D.DIRAC_BC_PERIODIC, **kw))
    try:
        D.dirac_set_potential(h, V, D.DIRAC_V_FULL if V.size > n[0] else D.DIRAC_V_X_ONLY)
        (D.dirac_set_state_fx(h, psi, 0) if psi.dtype == np.int64 else D.dirac_set_state(h, psi))
        D.dirac_step(h, steps)
        out = np.empty_like(psi)
        (D.dirac_get_state_fx(h, out) if psi.dtype == np.int64 else D.dirac_get_state(h, out))
        return out
    finally:
        D.dirac_destroy(h)


@pytest.mark.parametrize("strang", [0, 1])
@pytest.mark.parametrize("K,P", [(1, 1), (1, 2), (2, 2)])
@pytest.mark.parametrize("n", SIZES)
def test_periodic_fp64_bits(n, K, P, strang):
    import paper_1107_4650_gb300 as D
    if strang and K == 2:
        pytest.skip("FP64 second order runs one step a launch")
    nx, nz = n
    rng = np.random.default_rng(nx * 100 + nz)
    psi = W.random_state(nz, 1, nx, nx + nz)
    V = rng.uniform(-1, 1, nx if nz % 2 else nx * nz) * C * C
    Vo = V if V.size == nx else V.reshape(nz, 1, nx)
    step = oracle.step_strang2d if strang else (lambda p, *a, **k: oracle.step(p, 2, *a, **k))
    want, _ = step(psi, 1.0, C, DX, 3, V=Vo, periodic=True)
    got = _run(D, n, psi, V, 3, steps_per_launch=K, points_per_lane=P, splitting=strang)
    assert np.array_equal(got, want)


@pytest.mark.parametrize("K,P", [(1, 1), (2, 2), (4, 2)])
@pytest.mark.parametrize("n", SIZES)
def test_periodic_fp32(n, K, P):
    """Four FP32 steps: each rounds every value about nine times (relative 6e-8 each), adding like independent errors
    on a unitary step; 4e-6 is ten times their sum."""
    import paper_1107_4650_gb300 as D
    nx, nz = n
    psi = W.random_state(nz, 1, nx, 3 * nx + nz).astype(np.complex64)
    V = np.random.default_rng(nx).uniform(-1, 1, nx) * C * C
    want, _ = oracle.step(psi.astype(np.complex128), 2, 1.0, C, DX, 4, V=V, periodic=True)
    got = _run(D, n, psi, V, 4, steps_per_launch=K, points_per_lane=P, precision=D.DIRAC_FP32)
    assert np.linalg.norm((got - want).ravel()) <= 4e-6 * np.linalg.norm(want.ravel())


@pytest.mark.parametrize("strang", [0, 1])
@pytest.mark.parametrize("n", SIZES)
def test_periodic_fixed_point_bits(n, strang):
    import paper_1107_4650_gb300 as D
    nx, nz = n
    rng = np.random.default_rng(7 * nx + nz)
    q = rng.integers(-2 ** 50, 2 ** 50, (nz, 1, nx, 4, 2), dtype=np.int64)
    V = rng.uniform(-1, 1, nx) * C * C
    step = oracle.step_strang2d_fx if strang else oracle.step_fx
    want = step(q, 1.0, C, DX, 3, V=V, periodic=True)
    assert np.array_equal(_run(D, n, q, V, 3, precision=D.DIRAC_FX64, splitting=strang), want)
