"""A batch whose runs end one after the other, so that the rows per task change between its launches: each run's state as with
64 rows throughout, bit for bit, and its flux to the rounding of a sum in another order."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("sides,steps", [((8,), (9,)), ((640, 500, 8, 57, 300, 640, 130), (90, 3, 61, 0, 33, 17, 70)),
                                         ((1024,) * 6, (16, 8, 4, 64, 2, 1))])
def test_heights_that_change_give_the_same_runs(sides, steps, precision):
    import paper_1107_4650_gb300 as D
    rng = np.random.default_rng(len(sides))
    c = 137.0359895
    runs = [{"side": s, "face": max(1, s // 2 + 3) if s > 8 else 4, "nsteps": n, "V0": rng.uniform(0.5, 3) * c * c, "L": 0.005,
             "p0": rng.uniform(0.2, 1) * c, "width": max(1.0, s / 12) * 10 / 8192, "x0": -0.1 * s * 10 / 8192, "absorb": 0, "eta": 0.0}
            for s, n in zip(sides, steps)]

    def run(rows):
        cfg = D.dirac_batch_default_config()
        cfg.precision = precision
        cfg.segment_rows = rows
        b = D.dirac_batch_create(runs, cfg)
        try:
            D.dirac_batch_run(b)
            res = D.dirac_batch_results(b, len(runs))
            out = []
            for r, s in enumerate(sides):
                psi = np.empty((s, 1, s, 4), dtype=np.complex64 if precision else np.complex128)
                D.dirac_batch_get_state(b, r, psi)
                out.append(psi)
        finally:
            D.dirac_batch_destroy(b)
        return res, out

    want, wpsi = run(64)
    got, gpsi = run(0)
    for a, b in zip(gpsi, wpsi):
        assert np.array_equal(a.view(np.uint8), b.view(np.uint8))
    # a step's flux is a sum of at most side + 32 terms whose sizes add up to the norm at most, 2^-53 a term, on both sides
    tol = [2.0 ** -53 * 2 * (s + 32 + n) * max(n, 1) * max(w, 1.0) for s, n, w in zip(sides, steps, want["norm0"])]
    assert np.all(np.abs(np.asarray(got["flux"]) - np.asarray(want["flux"])) <= tol)
    assert np.array_equal(got["norm0"], want["norm0"])
