"""What a grid's replayed graphs hold (flux scratch, plan, kind of table, fixed-point scale) has changed between two calls of
dirac_step: the host runtime on a stand-in for the CUDA runtime and the launchers (fake_cuda.cpp), no GPU.  The launches with
use_graphs are those without, and none touches freed memory."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

import paper_1107_4650_gb300 as D
from paper_1107_4650_gb300 import build as B
from paper_1107_4650_gb300 import workloads as W

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def fake_lib(tmp_path_factory):
    gxx, cuda = shutil.which("g++"), os.path.join(os.path.dirname(os.path.dirname(B._nvcc())), "include")
    if gxx is None or not os.path.exists(os.path.join(cuda, "cuda_runtime.h")):
        pytest.skip("no g++ or no CUDA headers")
    lib = str(tmp_path_factory.mktemp("fake") / "libfake.so")
    # (bound to its own stand-ins whatever runtime the process has loaded)
    subprocess.run([gxx, "-std=c++17", "-O1", "-fPIC", "-shared", "-Wl,-Bsymbolic", "-fopenmp", "-I", cuda, "-I", B.CSRC, "-x", "c++",
                    os.path.join(B.CSRC, "dirac_api.cu"), os.path.join(HERE, "fake_cuda.cpp"), "-o", lib], check=True)
    return lib


@pytest.fixture
def fake(fake_lib, monkeypatch):
    monkeypatch.setattr(D, "_lib", None)
    lib = D.load_library(fake_lib)
    lib.fake_log.restype = ctypes.c_char_p
    lib.fake_limit.argtypes = [ctypes.c_size_t]
    lib.fake_limit(2 ** 64 - 1)
    lib.fake_reset()
    return lib


def _launches(lib, change, graphs, **cfg):
    """The launches of `change` (a function of the handle) on a fresh grid, and how many of them touched freed memory."""
    lib.fake_reset()
    h = D.dirac_create_grid(D.make_config(use_graphs=graphs, **cfg))
    try:
        change(h)
    finally:
        D.dirac_destroy(h)
    return lib.fake_log().decode().splitlines(), lib.fake_violations()


def _same_with_and_without(lib, change, **cfg):
    want, bad = _launches(lib, change, 0, **cfg)
    assert bad == 0
    got, bad = _launches(lib, change, 1, **cfg)
    assert bad == 0
    assert got == want


@pytest.mark.parametrize("splitting", [0, 1])
@pytest.mark.parametrize("precision,n", [(0, (96, 1, 80)), (1, (300, 1, 200)), (2, (40, 1, 33)), (0, (20, 12, 16)), (1, (20, 12, 16)),
                                         (2, (20, 12, 16))])
def test_potential_of_another_kind(fake, precision, n, splitting):
    V = np.zeros(n[::-1])

    def change(h):
        for kind in (D.DIRAC_V_FULL, D.DIRAC_V_X_ONLY, D.DIRAC_V_NONE, D.DIRAC_V_FULL):
            D.dirac_set_potential(h, None if kind == D.DIRAC_V_NONE else V if kind == D.DIRAC_V_FULL else V[0, 0], kind)
            D.dirac_step(h, 32 * D.dirac_get_info(h)["steps_per_launch"])  # one graph

    _same_with_and_without(fake, change, n=n, ndim=3 if n[1] > 1 else 2, precision=precision, splitting=splitting,
                           flux_face=n[0] // 2)


@pytest.mark.parametrize("splitting", [0, 1])
@pytest.mark.parametrize("n,points", [((40, 1, 33), 0), ((2000, 1, 1500), 0), ((20, 12, 16), 0), ((20, 12, 16), 1)])
def test_fixed_point_state_of_another_scale(fake, n, points, splitting):
    q = np.zeros(n[::-1] + (4, 2), dtype=np.int64)
    psi = np.zeros(n[::-1] + (4,), dtype=np.complex128)

    def change(h):
        for shift in (50, 43, None, 50):
            D.dirac_set_state(h, psi) if shift is None else D.dirac_set_state_fx(h, q, shift)
            D.dirac_step(h, 32 * D.dirac_get_info(h)["steps_per_launch"])

    _same_with_and_without(fake, change, n=n, ndim=3 if n[1] > 1 else 2, precision=2, splitting=splitting, points_per_lane=points,
                           flux_face=n[0] // 2)


@pytest.mark.parametrize("precision,n,what", [(1, (2048, 1, 2048), "scratch"), (0, (1536, 1, 1536), "scratch"), (0, (40, 1, 40), "field"),
                                              (1, (24, 24, 24), "field"), (1, (2048, 1, 2048), "table"), (0, (40, 1, 40), "table")])
def test_steps_after_a_failed_allocation(fake, precision, n, what):
    """A call that runs out of memory leaves a grid whose next steps touch nothing that was freed."""
    def change(h):
        steps = 32 * D.dirac_get_info(h)["steps_per_launch"]
        if what == "field":
            D.dirac_set_vector_potential(h, np.zeros((2 * steps, 3)))
        D.dirac_step(h, steps)
        fake.fake_limit(96 * 600 if what == "scratch" else 0)  # (room for the field's table alone)
        with pytest.raises(D.DiracError) as e:
            if what == "table":
                D.dirac_set_potential(h, np.zeros(n[::-1]), D.DIRAC_V_FULL)
            else:
                D.dirac_set_vector_potential(h, np.zeros((600 if what == "scratch" else 5 * steps, 3)))
        assert e.value.status == D.DIRAC_ERR_OOM
        fake.fake_limit(2 ** 64 - 1)
        D.dirac_step(h, steps)

    for graphs in (0, 1):
        log, bad = _launches(fake, change, graphs, n=n, ndim=3 if n[1] > 1 else 2, precision=precision, flux_face=n[0] // 2)
        assert bad == 0, [l for l in log if "freed" in l][:2]
