"""Stores of whole 32-byte pieces and, for caller-owned buffers that lie 16 bytes past such a boundary, of 16-byte ones:
the same bits, on grids whose strips end ragged, both boundaries, every storage type."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("periodic", [0, 1])
@pytest.mark.parametrize("precision,K,strang", [(0, 1, 0), (0, 1, 1), (1, 1, 0), (1, 2, 0), (1, 4, 0), (1, 2, 1), (2, 1, 0), (2, 1, 1)])
@pytest.mark.parametrize("n", [(28, 1, 5), (61, 1, 40), (130, 1, 67), (45, 9, 11)])
def test_caller_buffers_off_the_32_byte_boundary(n, precision, K, strang, periodic):
    import torch

    import paper_1107_4650_gb300 as D
    from paper_1107_4650_gb300 import workloads as W
    nx, ny, nz = n
    ndim = 3 if ny > 1 else 2
    if ndim == 3:
        K = 0
    cells = nx * ny * nz
    kind = {0: torch.float64, 1: torch.float32, 2: torch.int64}[precision]
    elem = 4 if precision == 1 else 8
    psi = torch.from_numpy(W.random_state(nz, ny, nx, nx + nz)).cuda()
    psi = psi.to(torch.complex64) if precision == 1 else psi
    V = np.random.default_rng(nz).uniform(-1, 1, nx) * W.C_AU ** 2

    def run(shift):
        pads = [torch.zeros(8 * cells + 64, dtype=kind, device="cuda") for _ in range(2)]
        bufs = [p[shift // elem:] for p in pads]
        assert all(b.data_ptr() % 32 == shift % 32 for b in bufs)
        h = D.dirac_create_grid(D.make_config(n, ndim=ndim, precision=precision, boundary=periodic, steps_per_launch=K,
                                              splitting=strang, ext_state=[b.data_ptr() for b in bufs]))
        try:
            D.dirac_set_potential(h, V, D.DIRAC_V_X_ONLY)
            D.dirac_set_state(h, psi)
            D.dirac_step(h, 5)
            out = torch.empty_like(psi)
            D.dirac_get_state(h, out)
            torch.cuda.synchronize()
            guard = [p[:shift // elem].abs().sum().item() + p[shift // elem + 8 * cells:].abs().sum().item() for p in pads]
        finally:
            D.dirac_destroy(h)
        assert guard == [0, 0]
        return out

    a, b = run(0), run(16)
    assert torch.equal(torch.view_as_real(a), torch.view_as_real(b))
