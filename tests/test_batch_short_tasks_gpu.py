"""Ensembles cut into tasks of a few rows, so that each warp takes many of them and refills its row ring at once after each: the
bits of single grids, stepped by warps that take one task each."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", [1, 8])
@pytest.mark.parametrize("precision,K,P", [(0, 1, 2), (0, 2, 2), (1, 1, 2), (1, 2, 4), (1, 4, 2)])
def test_many_tasks_a_warp(precision, K, P, rows):
    import paper_1107_4650_gb300 as D
    from paper_1107_4650_gb300 import workloads as W
    c, sides, steps = W.C_AU, (1024, 700, 333), 9
    dtype = np.complex64 if precision else np.complex128
    runs = [{"side": s, "face": s // 2, "nsteps": steps, "V0": 1.5 * c * c, "L": 0.005, "p0": 0.5 * c, "width": s / 12 * 10 / 8192,
             "x0": -0.1 * s * 10 / 8192, "absorb": 0, "eta": 0.0} for s in sides]
    psi = [W.random_state(s, 1, s, s).astype(dtype) for s in sides]
    V = [np.random.default_rng(s).uniform(-1, 1, s) * c * c for s in sides]
    cfg = D.dirac_batch_default_config()
    cfg.precision, cfg.steps_per_launch, cfg.points_per_lane, cfg.segment_rows = precision, K, P, rows
    b = D.dirac_batch_create(runs, cfg)
    try:
        for r in range(len(sides)):
            D.dirac_batch_set_state(b, r, psi[r])
            D.dirac_batch_set_potential(b, r, V[r])
        D.dirac_batch_run(b)
        D.dirac_batch_results(b, len(runs))
        got = [np.empty_like(p) for p in psi]
        for r in range(len(sides)):
            D.dirac_batch_get_state(b, r, got[r])
    finally:
        D.dirac_batch_destroy(b)
    for r, s in enumerate(sides):
        h = D.dirac_create_grid(D.make_config((s, 1, s), precision=precision, steps_per_launch=1, points_per_lane=2))
        try:
            D.dirac_set_potential(h, V[r], D.DIRAC_V_X_ONLY)
            D.dirac_set_state(h, psi[r])
            D.dirac_step(h, steps)
            want = np.empty_like(psi[r])
            D.dirac_get_state(h, want)
        finally:
            D.dirac_destroy(h)
        assert np.array_equal(got[r].view(np.uint8), want.view(np.uint8))
