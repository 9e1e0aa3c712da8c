"""A periodic grid's row copy that never completes (DIRAC_INJECT_STALL: its barrier expects 16 bytes more than the wrapped copy
delivers) ends in the kernel's bounded wait and is reported; the process then steps a fresh grid as before."""
import time

import numpy as np
import pytest

import oracle
from paper_1107_4650_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,steps", [(0, 1), (1, 1), (1, 4), (2, 1)])
def test_stalled_wrapped_copy_is_reported(precision, steps, monkeypatch):
    import paper_1107_4650_gb300 as D
    nx, nz = 200, 64
    psi = W.random_state(nz, 1, nx, seed=67)
    own = psi.astype(np.complex64) if precision == 1 else psi
    monkeypatch.setenv("DIRAC_INJECT_STALL", "1")
    h = D.dirac_create_grid(D.make_config((nx, 1, nz), precision=precision, boundary=D.DIRAC_BC_PERIODIC, steps_per_launch=steps,
                                          points_per_lane=2))
    monkeypatch.delenv("DIRAC_INJECT_STALL")
    try:
        D.dirac_set_state(h, own)
        t0 = time.perf_counter()
        D.dirac_step(h, steps)
        with pytest.raises(D.DiracError) as e:
            D.dirac_observables(h)
        assert e.value.status == D.DIRAC_ERR_TIMEOUT
        assert 0.5 < time.perf_counter() - t0 < 20.0
        D.dirac_set_state(h, own)  # clears the report
        D.dirac_observables(h)
    finally:
        D.dirac_destroy(h)
    want, _ = oracle.step(psi, 2, 1.0, W.C_AU, W.DX_DEFAULT, 3, periodic=True)
    h = D.dirac_create_grid(D.make_config((nx, 1, nz), boundary=D.DIRAC_BC_PERIODIC, steps_per_launch=1, points_per_lane=2))
    try:
        D.dirac_set_state(h, psi)
        D.dirac_step(h, 3)
        got = np.empty_like(psi)
        D.dirac_get_state(h, got)
    finally:
        D.dirac_destroy(h)
    assert np.array_equal(got, want)
