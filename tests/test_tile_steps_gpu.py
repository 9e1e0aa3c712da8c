"""Small 2-D grids: several steps of a tile per launch give the row kernel's state bit for bit and its face flux to the
rounding of a sum in another order."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# one cell, one row, one column, tiles cut at either end, one tile more than a row of them, sizes that take each shape
SIZES = [(1, 1), (40, 1), (1, 40), (5, 3), (24, 24), (25, 9), (30, 14), (57, 41), (128, 128), (200, 150), (301, 257), (520, 384),
         (700, 500)]


@pytest.mark.parametrize("periodic", [0, 1])
@pytest.mark.parametrize("precision,strang", [(0, 0), (0, 1), (1, 0), (1, 1), (2, 0), (2, 1)])
@pytest.mark.parametrize("n", SIZES)
def test_tiles_equal_rows(n, precision, strang, periodic):
    import paper_1107_4650_gb300 as D
    from paper_1107_4650_gb300 import workloads as W
    nx, nz = n
    rng = np.random.default_rng(nx + nz)
    psi = W.random_state(nz, 1, nx, nx + 3 * nz)
    psi = psi.astype(np.complex64) if precision == 1 else psi
    full = (nx + nz) % 2 == 0
    V = rng.uniform(-1, 1, (nz, 1, nx) if full else nx) * W.C_AU ** 2
    steps = 15  # launches of every length: 15 = 3 x 4 + 2 + 1 = 7 x 2 + 1

    def run(k, p):
        h = D.dirac_create_grid(D.make_config((nx, 1, nz), precision=precision, splitting=strang, boundary=periodic,
                                              steps_per_launch=k, points_per_lane=p, flux_face=nx // 2 if nx > 1 else -1))
        try:
            D.dirac_set_potential(h, V, D.DIRAC_V_FULL if full else D.DIRAC_V_X_ONLY)
            D.dirac_set_state(h, psi)
            before = D.dirac_observables(h)["norm"]
            D.dirac_step(h, steps)
            out = np.empty(psi.shape, dtype=psi.dtype)
            D.dirac_get_state(h, out)
            obs = D.dirac_observables(h)
            info = D.dirac_get_info(h)
        finally:
            D.dirac_destroy(h)
        return out, obs, info, before

    want, owant, _, norm = run(1, 1)
    got, ogot, info, _ = run(0, 0)
    # steps_per_launch and points_per_lane as reported are a pair that a configuration takes
    again, _, _, _ = run(info["steps_per_launch"], info["points_per_lane"])
    assert np.array_equal(got.view(np.uint8), want.view(np.uint8))
    assert np.array_equal(again.view(np.uint8), want.view(np.uint8))
    # per sweep a sum of at most nz + 1 terms whose sizes add up to the norm at most; 2^-53 a term, both sides
    sweeps = steps * (1 + strang)
    tol = 2.0 ** -53 * 2 * (nz + 2 + sweeps) * sweeps * max(norm, 1.0)
    key = [k for k in ogot if "flux" in k][0]
    assert abs(ogot[key] - owant[key]) <= tol, (ogot[key], owant[key], tol)


@pytest.mark.parametrize("periodic", [0, 1])
@pytest.mark.parametrize("precision,strang", [(0, 0), (0, 1), (1, 0), (1, 1)])
@pytest.mark.parametrize("n,full", [((5, 3), False), ((28, 12), False), ((57, 41), False), ((57, 41), True), ((200, 150), False),
                                    ((301, 257), False), ((520, 384), False)])
def test_tiles_in_a_field_equal_rows(n, full, precision, strang, periodic):
    import paper_1107_4650_gb300 as D
    from paper_1107_4650_gb300 import workloads as W
    nx, nz = n
    rng = np.random.default_rng(nx + nz)
    psi = W.random_state(nz, 1, nx, nx + 3 * nz).astype(np.complex64 if precision else np.complex128)
    V = rng.uniform(-1, 1, (nz, 1, nx) if full else nx) * W.C_AU ** 2
    A = rng.uniform(-1, 1, (9, 3))  # another matrix each step

    def run(k, p):
        h = D.dirac_create_grid(D.make_config((nx, 1, nz), precision=precision, splitting=strang, boundary=periodic,
                                              steps_per_launch=k, points_per_lane=p))
        try:
            D.dirac_set_vector_potential(h, A)
            D.dirac_set_potential(h, V, D.DIRAC_V_FULL if full else D.DIRAC_V_X_ONLY)
            D.dirac_set_state(h, psi)
            D.dirac_step(h, 4)
            D.dirac_step(h, 5)
            out = np.empty_like(psi)
            D.dirac_get_state(h, out)
            return out
        finally:
            D.dirac_destroy(h)

    assert np.array_equal(run(0, 0).view(np.uint8), run(1, 2).view(np.uint8))


def test_tiles_inside_a_callers_capture():
    """A copy and the steps captured in a caller's graph and replayed: the same state as the calls made directly."""
    import torch

    import paper_1107_4650_gb300 as D
    from paper_1107_4650_gb300 import workloads as W
    nx, nz = 96, 80
    psi = torch.from_numpy(W.random_state(nz, 1, nx, 4)).cuda()
    stream = torch.cuda.Stream()
    h = D.dirac_create_grid(D.make_config((nx, 1, nz), stream=stream.cuda_stream, flux_face=50))
    try:
        with torch.cuda.stream(stream):
            stream.wait_stream(torch.cuda.default_stream())
            D.dirac_set_state(h, psi)
            D.dirac_step(h, 8)
            D.dirac_step(h, 8)
            want = torch.empty_like(psi)
            D.dirac_get_state(h, want)
            D.dirac_set_state(h, psi)
            src = torch.zeros(1024, device="cuda")
            dst = torch.ones(1024, device="cuda")
            stream.synchronize()
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=stream):
                dst.copy_(src)
                D.dirac_step(h, 8)
            g.replay()  # eight steps are an even number of launches: the state is back in the buffer it started in
            g.replay()
            got = torch.empty_like(psi)
            D.dirac_get_state(h, got)
            stream.synchronize()
        assert torch.equal(torch.view_as_real(got), torch.view_as_real(want))
    finally:
        D.dirac_destroy(h)
