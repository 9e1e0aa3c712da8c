"""Training batches at the edges of the kernels' tiles (128 samples of a product, 64 of a K stage, 32 and 16 of the layer
kernels, 256 of the batch sums) and on buffers that grow from call to call, against the CPU network."""
import numpy as np
import pytest

from oracle import mlp as M

pytestmark = pytest.mark.gpu
LO, HI = np.array([0.5, 0.2, 40.0]), np.array([3.0, 1.0, 150.0])


def _data(B, seed):
    rng = np.random.default_rng(seed)
    return LO + (HI - LO) * rng.uniform(0, 1, (B, 3)), rng.uniform(0, 1, B)


@pytest.mark.parametrize("B", [1, 2, 15, 16, 17, 31, 33, 63, 65, 127, 128, 129, 255, 256, 257, 513, 1000])
def test_gradient_at_the_tiles_edges(B):
    """Tolerance of the gradient test at 64 and 300 samples: BF16 operands differ from the oracle's where a rounding
    point falls the other way, a few 1e-3 of a block's norm."""
    import paper_1107_4650_gb300 as D
    q, t = _data(B, B)
    h = D.dirac_surrogate_create(LO, HI, seed=7, max_batch=1024)
    try:
        loss, g = D.dirac_surrogate_gradient(h, q, t)
        p = D.dirac_surrogate_get_params(h).astype(np.float64)
        y = D.dirac_surrogate_predict(h, q)
    finally:
        D.dirac_surrogate_destroy(h)
    _, want = M.loss_and_grad(p, 2.0 * (q - LO) / (HI - LO) - 1.0, t, round_bf16=True)
    # the loss is the sequential sum of the FP32 squared errors of the predictions, exactly
    d = (y.astype(np.float32) - t.astype(np.float32)).astype(np.float32)
    total = 0.0
    for v in (d * d).astype(np.float32):
        total += float(v)
    assert loss == total / B
    gb, wb = M.unpack(g), M.unpack(want)
    for name in gb:
        assert np.linalg.norm(gb[name] - wb[name]) <= 2e-2 * np.linalg.norm(wb[name]) + 1e-30, name


def test_growing_and_shrinking_batches_leave_nothing_behind():
    """A small batch after a large one (whose rows still lie in the buffers), and training after either, give what a
    fresh network gives, bit for bit."""
    import paper_1107_4650_gb300 as D
    h = D.dirac_surrogate_create(LO, HI, seed=9, max_batch=1024)
    try:
        p0 = D.dirac_surrogate_get_params(h)
        for B in (40, 1000, 130, 7, 700):
            q, t = _data(B, B)
            got = D.dirac_surrogate_gradient(h, q, t)
            f = D.dirac_surrogate_create(LO, HI, seed=9, max_batch=1024)
            want = D.dirac_surrogate_gradient(f, q, t)
            D.dirac_surrogate_destroy(f)
            assert got[0] == want[0] and np.array_equal(got[1], want[1])
            D.dirac_surrogate_set_params(h, p0)
            f = D.dirac_surrogate_create(LO, HI, seed=9, max_batch=1024)
            D.dirac_surrogate_set_params(f, p0)
            lf = D.dirac_surrogate_train(f, q, t, 2, max(1, B // 3), 1e-3)
            pf = D.dirac_surrogate_get_params(f)
            D.dirac_surrogate_destroy(f)
            lh = D.dirac_surrogate_train(h, q, t, 2, max(1, B // 3), 1e-3)
            assert lh == lf and np.array_equal(D.dirac_surrogate_get_params(h), pf)
            D.dirac_surrogate_set_params(h, p0)
    finally:
        D.dirac_surrogate_destroy(h)


@pytest.mark.parametrize("n", [1, 31, 32, 33, 127, 129, 4863, 4864, 4865, 6000])
def test_small_and_large_calls_predict_the_same_bits(n):
    """Calls of up to 32 queries for each of 152 SMs run on 32-query tiles and pinned buffers, larger ones on 128-query
    tiles and device buffers: a query's prediction does not depend on which, nor on its neighbours."""
    import paper_1107_4650_gb300 as D
    q, _ = _data(6000, 3)
    h = D.dirac_surrogate_create(LO, HI, seed=11, max_batch=8192)
    try:
        whole = D.dirac_surrogate_predict(h, q)
        assert np.array_equal(D.dirac_surrogate_predict(h, q[:n]), whole[:n])
        assert np.array_equal(D.dirac_surrogate_predict(h, q[6000 - n:]), whole[6000 - n:])
    finally:
        D.dirac_surrogate_destroy(h)
