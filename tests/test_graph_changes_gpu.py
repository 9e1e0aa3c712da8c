"""Steps replayed from graphs after a change of what the graphs hold: the bits and the flux of the same calls without graphs."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _run(change, graphs, psi, **cfg):
    import paper_1107_4650_gb300 as D
    h = D.dirac_create_grid(D.make_config(psi.shape[2::-1], use_graphs=graphs, flux_face=psi.shape[2] // 2, **cfg))
    try:
        D.dirac_set_state(h, psi)
        change(D, h)
        out = np.empty_like(psi)
        D.dirac_get_state(h, out)
        return out, D.dirac_observables(h)["flux_cum"]
    finally:
        D.dirac_destroy(h)


def _same_with_and_without(change, psi, **cfg):
    (a, fa), (b, fb) = _run(change, 1, psi, **cfg), _run(change, 0, psi, **cfg)
    assert np.array_equal(a.view(np.uint8), b.view(np.uint8))
    assert fa == fb  # the parts and the order of their sum are the same


@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("n", [(96, 1, 80), (20, 12, 16)])
def test_potential_of_another_kind(n, precision):
    from paper_1107_4650_gb300 import workloads as W
    psi = W.random_state(n[2], n[1], n[0], 3).astype(np.complex64 if precision == 1 else np.complex128)
    V = np.random.default_rng(5).uniform(-1, 1, n[::-1]) * W.C_AU ** 2

    def change(D, h):
        for kind in (D.DIRAC_V_FULL, D.DIRAC_V_X_ONLY, D.DIRAC_V_NONE, D.DIRAC_V_FULL):
            D.dirac_set_potential(h, None if kind == D.DIRAC_V_NONE else V if kind == D.DIRAC_V_FULL else V[0, 0], kind)
            D.dirac_step(h, 32 * D.dirac_get_info(h)["steps_per_launch"])

    _same_with_and_without(change, psi, ndim=3 if n[1] > 1 else 2, precision=precision)


@pytest.mark.parametrize("splitting", [0, 1])
@pytest.mark.parametrize("n", [(96, 1, 80), (20, 12, 16)])
def test_fixed_point_state_of_another_norm(n, splitting):
    from paper_1107_4650_gb300 import workloads as W
    psi = W.random_state(n[2], n[1], n[0], 3)

    def change(D, h):
        steps = 32 * D.dirac_get_info(h)["steps_per_launch"]
        D.dirac_step(h, steps)
        D.dirac_set_state(h, psi * 37.0)
        D.dirac_step(h, steps)

    _same_with_and_without(change, psi, ndim=3 if n[1] > 1 else 2, precision=2, splitting=splitting)
