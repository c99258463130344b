"""CPU tests of the cooperative launch's way out where fewer CTAs fit than the
device holds (gf_coop.h), with a fake of the launch that refuses."""
import ctypes as C
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
REFUSED = 720


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("coop") / "libcoop.so")
    src = os.path.join(ROOT, "tests", "coop", "coop_shim.cpp")
    r = subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I",
                        os.path.join(ROOT, "paper_2212_09005_gb300", "csrc"), "-o", out, src],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    lib = C.CDLL(out)

    def call(grid, fits, error=0):
        tried, err, recorded = (C.c_int * 64)(), C.c_int(), C.c_int()
        n = lib.coop_run(grid, fits, error, tried, C.byref(err), C.byref(recorded))
        return list(tried[:n]), err.value, recorded.value

    return call


@pytest.mark.parametrize("grid,fits,tried", [(608, 608, [608]), (608, 607, [608, 304]), (608, 32, [608, 304, 152, 76, 38, 19]),
                                             (7, 1, [7, 3, 1]), (1, 1, [1]), (2, 1, [2, 1])])
def test_smaller_grids_until_one_fits(run, grid, fits, tried):
    assert run(grid, fits) == (tried, 0, 0)


def test_what_no_grid_mends_is_reported(run):
    assert run(5, 0) == ([5, 2, 1], REFUSED, REFUSED)
    assert run(608, 608, error=98) == ([608], 98, 98)


def test_every_cooperative_launch_has_the_way_out():
    csrc = os.path.join(ROOT, "paper_2212_09005_gb300", "csrc")
    launches = coop = 0
    for name in os.listdir(csrc):
        with open(os.path.join(csrc, name)) as f:
            text = f.read()
        launches += text.count("cudaLaunchCooperativeKernel(")
        if not name.endswith(".h"):
            coop += text.count("coop_launch(")
    assert launches == coop > 0
