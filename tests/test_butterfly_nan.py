"""NaNs through the integer magnitude sum (csrc/butterfly.cuh): whichever words hold the payload, and whatever the other operand
is, the sum is a NaN, as the FP64 add's is."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1107_4650_gb300", "csrc")

HARNESS = r'''
#include "butterfly.cuh"
#include <initializer_list>
#include <stdio.h>
int main() {
    const uint64_t E = 0x7ffull << 52, S = 1ull << 63;
    const uint64_t payload[] = {1, 2, 0x80000000ull, 0xffffffffull, 1ull << 32, 1ull << 51, (1ull << 52) - 1, (1ull << 51) | 1};
    const uint64_t other[] = {E, 0, 1, 0x3ff0000000000000ull, 0x7fefffffffffffffull, 0x7fe0000000000000ull, E | 1, E | 0xffffffffull,
                              E | (1ull << 51), E | (1ull << 32)};
    int bad = 0;
    for (uint64_t p : payload)
        for (uint64_t o : other)
            for (int s = 0; s < 4; ++s) {
                const uint64_t a = (E | p) | (s & 1 ? S : 0), b = o | (s & 2 ? S : 0);
                for (uint64_t r : {dirac::magnitude_sum_bits(a, b), dirac::magnitude_sum_bits(b, a)}) bad += (r & ~S) <= E;
            }
    const uint64_t inf[] = {0, 1, 0x3ff0000000000000ull, 0x7fefffffffffffffull, E};
    for (uint64_t o : inf)
        bad += dirac::magnitude_sum_bits(E, o) != E || dirac::magnitude_sum_bits(o, E) != E || dirac::magnitude_sum_bits(S | E, o) != (S | E);
    printf("%d\n", bad);
    return bad != 0;
}
'''


def test_nan_payloads_in_either_word(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    src = tmp_path / "t.cpp"
    src.write_text(HARNESS)
    subprocess.run([gxx, "-O2", "-I", CSRC, str(src), "-o", str(tmp_path / "t")], check=True)
    out = subprocess.run([str(tmp_path / "t")], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout


@pytest.mark.gpu
def test_step_on_an_infinity_beside_such_a_nan():
    """The device's form of the same comparison: an infinity added to a NaN of the smallest payload, in either order, leaves NaNs
    where the oracle's additions do."""
    import numpy as np

    import oracle
    import paper_1107_4650_gb300 as D
    from paper_1107_4650_gb300 import workloads as W
    nx, nz = 64, 40
    psi = W.random_state(nz, 1, nx, 8)
    nan = np.array([0x7ff0000000000001], dtype=np.uint64).view(np.float64)[0]
    for z, a, b in ((10, np.inf, nan), (25, nan, np.inf)):  # components 1 and 4 meet in the x sweep
        v = psi[z, 0, 20].view(np.float64)
        v[0], v[6] = a, b
    want, _ = oracle.step(psi, 2, 1.0, W.C_AU, W.DX_DEFAULT, 1)
    for k, p in ((0, 0), (1, 1)):
        h = D.dirac_create_grid(D.make_config((nx, 1, nz), steps_per_launch=k, points_per_lane=p))
        try:
            D.dirac_set_state(h, psi)
            D.dirac_step(h, 1)
            got = np.empty_like(psi)
            D.dirac_get_state(h, got)
        finally:
            D.dirac_destroy(h)
        g, w = got.view(np.float64), want.view(np.float64)
        assert np.array_equal(np.isnan(g), np.isnan(w)) and np.array_equal(g[~np.isnan(w)], w[~np.isnan(w)])
