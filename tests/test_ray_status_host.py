"""Status word of the scalar update (csrc/ray.cuh, host build): converged where
the iteration met its tolerance or nothing flows, the cap bit where it did not,
and neither beside a trial strain that is not finite."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

import synth

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = os.path.join(ROOT, "tests", "native", "ray_status_check.cpp")
CONVERGED, NONFINITE, CAP = 1 << 16, 1 << 17, 1 << 18
FLAGS = 0xF << 16


@pytest.fixture(scope="module")
def word(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("ray_status") / "s.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-fPIC", "-shared",
                    "-I/usr/local/cuda/include", SRC, "-o", out], check=True)
    lib = ctypes.CDLL(out)
    lib.ray_status_word.restype = ctypes.c_uint32
    dp = ctypes.POINTER(ctypes.c_double)

    def call(mode, eps, shift=0.0, prm=synth.MATRIX_16):
        p, e, sig = np.array(prm, dtype=float), np.array(eps, dtype=float), np.empty(6)
        w = lib.ray_status_word(mode, p.ctypes.data_as(dp), e.ctypes.data_as(dp), ctypes.c_double(0.01),
                                ctypes.c_double(shift), sig.ctypes.data_as(dp))
        return w & FLAGS, sig
    return call


EPS = [0.01, -0.003, 0.001, 0.002, 0.0, -0.004]


@pytest.mark.parametrize("mode", [0, 1, 2])
def test_status(word, mode):
    w, sig = word(mode, EPS)
    assert w == CONVERGED
    assert word(mode, [0.0] * 6)[0] == CONVERGED
    for bad in (np.nan, np.inf):
        assert word(mode, [bad, 0, 0, 0, 0, 0])[0] == NONFINITE
        assert word(mode, [0, 0, 0, 0, bad, 0])[0] == NONFINITE
    # a start at theta = 1: more evaluations, the same root
    w, other = word(mode, EPS, -40.0)
    assert w == CONVERGED and np.allclose(other, sig, rtol=1e-14 if mode < 2 else 1e-6)
    # a start many orders below the root: the evaluations run out
    assert word(mode, EPS, 10.0)[0] == CAP


@pytest.mark.parametrize("mode", [0, 1])
def test_square_out_of_range(word, mode):
    """A finite trial strain whose square leaves the FP64 range is not solved, and says so."""
    assert word(mode, [1e160, 0, 0, 0, 0, 0])[0] == NONFINITE
