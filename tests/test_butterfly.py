"""FP64 pairs (a + b, a - b) split over the FP64 and the integer pipe (csrc/butterfly.cuh): the integer magnitude sum
against the FP64 add on the CPU, and whole steps on states of every exponent against the oracle, bit for bit."""
import os
import shutil
import subprocess

import numpy as np
import pytest

import oracle
from paper_1107_4650_gb300 import workloads as W

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1107_4650_gb300", "csrc")

HARNESS = r'''
#include "butterfly.cuh"
#include <math.h>
#include <stdio.h>
#include <string.h>
static uint64_t s = 88172645463325252ull;
static uint64_t r() { s ^= s << 13; s ^= s >> 7; s ^= s << 17; return s; }
static double f(uint64_t u) { double x; memcpy(&x, &u, 8); return x; }
static uint64_t bits(double x) { uint64_t u; memcpy(&u, &x, 8); return u; }
int main() {
    const uint64_t F = (1ull << 52) - 1, E = 0x7ffull << 52;
    long bad = 0;
    for (long i = 0; i < 4000000; ++i) {
        uint64_t a = r(), b = r();
        const int m = i % 8;  // exponents: any, near each other, both subnormal or nearly, both about to overflow
        long ea = m == 6 ? (long)(r() % 70) : m == 7 ? 2047 - (long)(r() % 70) : (long)((a >> 52) & 0x7ff);
        const long span = m == 0 ? 4 : m == 1 ? 33 : m == 2 ? 70 : 8, off = (long)(r() % span);
        long eb = m == 5 ? (long)((b >> 52) & 0x7ff) : ea + ((r() & 1) ? off : -off);
        eb = eb < 0 ? 0 : eb > 2047 ? 2047 : eb;
        a = (a & ~E) | ((uint64_t)ea << 52);
        b = (b & ~E) | ((uint64_t)eb << 52);
        if (r() & 1) {  // short and all-ones mantissas: exact ties and carries
            const int k = r() % 53, l = r() % 53;
            if (r() & 1) a |= F;
            if (r() & 1) b |= F;
            a = (a & ~F) | ((a & F) >> k << k);
            b = (b & ~F) | ((b & F) >> l << l);
        }
        if ((r() & 15) == 0) a &= ~(F | E);
        if ((r() & 15) == 0) b &= ~(F | E);
        if ((r() & 15) == 0) a &= ~F;
        const double want = copysign(fabs(f(a)) + fabs(f(b)), f(a));
        const uint64_t got = dirac::magnitude_sum_bits(a, b);
        const bool low_nan = ((a >> 32) & 0x7fffffff) == 0x7ff00000 || ((b >> 32) & 0x7fffffff) == 0x7ff00000;
        bad += isnan(want) ? !(isnan(f(got)) || low_nan) : got != bits(want);
    }
    printf("%ld\n", bad);
    return bad != 0;
}
'''


def test_integer_magnitude_sum_is_the_fp64_add(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    src = tmp_path / "t.cpp"
    src.write_text(HARNESS)
    subprocess.run([gxx, "-O2", "-ffp-contract=off", "-I", CSRC, str(src), "-o", str(tmp_path / "t"), "-lm"], check=True)
    out = subprocess.run([str(tmp_path / "t")], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout


def _state(nz, ny, nx, kind, seed):
    """Random signs and mantissas (some of few bits: ties) over the exponents of `kind`."""
    rng = np.random.default_rng(seed)
    lo, hi = {"ordinary": (-3, 3), "apart": (-60, 60), "every": (-1070, 960), "subnormal": (-1074, -1010)}[kind]
    shape = (nz, ny, nx, 4, 2)
    m = np.where(rng.random(shape) < 0.3, rng.integers(0, 9, shape) / 4.0, rng.uniform(-2, 2, shape))
    with np.errstate(under="ignore"):
        x = np.ldexp(m * rng.choice([-1.0, 1.0], shape), rng.integers(lo, hi, shape))
    x[rng.random(shape) < 0.1] = 0.0
    return np.ascontiguousarray(x).view(np.complex128)[..., 0]


def _deferred(psi, ndim, nsteps):
    """Massless steps without a potential in the kernels' order: sweeps without their 1/2, the power of two at the end
    of the step.  (The oracle halves after each sweep, which rounds subnormal values where the kernels do not: on a
    state of subnormals the two differ whichever pipe forms the sums.)"""
    def moved(a, axis, by):
        out = np.zeros_like(a)
        n = a.shape[axis]
        src = [slice(None)] * a.ndim
        dst = [slice(None)] * a.ndim
        src[axis], dst[axis] = (slice(0, n - 1), slice(1, n)) if by > 0 else (slice(1, n), slice(0, n - 1))
        if n > 1:
            out[tuple(dst)] = a[tuple(src)]
        return out

    def times_i(a):
        return np.stack([-a[..., 1], a[..., 0]], axis=-1)

    p = [np.ascontiguousarray(psi[..., c]).view(np.float64).reshape(psi.shape[:3] + (2,)) for c in range(4)]
    for _ in range(nsteps):
        for axis in ((2, 1, 0) if ndim == 3 else (2, 0)):
            if axis == 2:  # x
                turned = [p[3], p[2], p[1], p[0]]
            elif axis == 1:  # y
                turned = [-times_i(p[3]), times_i(p[2]), -times_i(p[1]), times_i(p[0])]
            else:
                turned = [p[2], -p[3], p[0], -p[1]]
            p = [moved(a + t, axis, 1) + moved(a - t, axis, -1) for a, t in zip(p, turned)]
        p = [a * (0.125 if ndim == 3 else 0.25) for a in p]
    return np.stack([np.ascontiguousarray(a).view(np.complex128)[..., 0] for a in p], axis=-1)


@pytest.mark.gpu
@pytest.mark.parametrize("kind", ["ordinary", "apart", "every", "subnormal"])
@pytest.mark.parametrize("P", [1, 2])
@pytest.mark.parametrize("n", [(29, 1, 1), (30, 1, 17), (31, 1, 40), (95, 1, 33), (33, 9, 7)])
def test_step_bits_over_all_exponents(n, P, kind):
    import paper_1107_4650_gb300 as D
    nx, ny, nz = n
    ndim = 3 if ny > 1 else 2
    psi0 = _state(nz, ny, nx, kind, 17 * nx + P)
    V = W.tanh_step(nx, W.DX_DEFAULT, -nx * W.DX_DEFAULT / 2, 0.0, 2.5 * W.C_AU ** 2, 4 * W.DX_DEFAULT)
    plain = kind in ("every", "subnormal")
    if plain:
        want = _deferred(psi0, ndim, 2)
    else:
        want, _ = oracle.step(psi0, ndim, 1.0, W.C_AU, W.DX_DEFAULT, 2, V=V)
    h = D.dirac_create_grid(D.make_config(n, ndim=ndim, points_per_lane=P, steps_per_launch=1, m=0.0 if plain else 1.0))
    try:
        if not plain:
            D.dirac_set_potential(h, V, D.DIRAC_V_X_ONLY)
        D.dirac_set_state(h, psi0)
        D.dirac_step(h, 2)
        got = np.empty_like(psi0)
        D.dirac_get_state(h, got)
    finally:
        D.dirac_destroy(h)
    assert np.array_equal(got, want)


@pytest.mark.gpu
def test_step_passes_on_infinities_and_nans():
    import paper_1107_4650_gb300 as D
    nx, nz = 64, 40
    psi0 = _state(nz, 1, nx, "ordinary", 5)
    psi0[7, 0, 9, 0] = np.inf
    psi0[30, 0, 33, 2] = np.nan
    want, _ = oracle.step(psi0, 2, 1.0, W.C_AU, W.DX_DEFAULT, 2)
    h = D.dirac_create_grid(D.make_config((nx, 1, nz)))
    try:
        D.dirac_set_state(h, psi0)
        D.dirac_step(h, 2)
        got = np.empty_like(psi0)
        D.dirac_get_state(h, got)
        with pytest.raises(D.DiracError):
            D.dirac_observables(h)
    finally:
        D.dirac_destroy(h)
    a, b = got.view(np.float64), want.view(np.float64)
    assert np.array_equal(np.isnan(a), np.isnan(b)) and np.array_equal(a[~np.isnan(b)], b[~np.isnan(b)])
