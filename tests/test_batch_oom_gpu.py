"""An ensemble whose tuning runs out of memory (an allocation that fails on the host): the plan it had stands, and its runs are
those of an ensemble that was never tuned."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
def test_runs_after_a_failed_autotune(precision, monkeypatch):
    import paper_1107_4650_gb300 as D
    c = 137.0359895
    runs = [{"side": s, "face": s // 2, "nsteps": 23, "V0": 1.5 * c * c, "L": 0.005, "p0": 0.5 * c, "width": s / 12 * 10 / 8192,
             "x0": -0.1 * s * 10 / 8192, "absorb": 0, "eta": 0.0} for s in (200, 130, 64)]

    def run(tune):
        cfg = D.dirac_batch_default_config()
        cfg.precision = precision
        cfg.steps_per_launch, cfg.points_per_lane, cfg.segment_rows = 1, 2, 256  # the least scratch: every other plan needs more
        b = D.dirac_batch_create(runs, cfg)
        try:
            before = D.dirac_batch_get_info(b)
            if tune:
                monkeypatch.setenv("DIRAC_INJECT_OOM", "1")
                with pytest.raises(D.DiracError) as e:
                    D.dirac_batch_autotune(b)
                monkeypatch.delenv("DIRAC_INJECT_OOM")
                assert e.value.status == D.DIRAC_ERR_OOM
            assert D.dirac_batch_get_info(b) == before
            D.dirac_batch_run(b)
            res = D.dirac_batch_results(b, len(runs))
            psi = np.empty((200, 1, 200, 4), dtype=np.complex64 if precision else np.complex128)
            D.dirac_batch_get_state(b, 0, psi)
            return res, psi
        finally:
            D.dirac_batch_destroy(b)

    (want, wpsi), (got, gpsi) = run(False), run(True)
    assert np.array_equal(gpsi.view(np.uint8), wpsi.view(np.uint8))
    for key in want:
        assert np.array_equal(got[key], want[key])
