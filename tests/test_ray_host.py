"""The scalar equation of a proportional law (csrc/ray.cuh) against the general
AD-driven Newton solver on the same potentials (host build of the device
headers): sigma, z, tangent and the status flags over exponents, step sizes and
magnitudes of the trial strain, and the degenerate states."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

import synth

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = os.path.join(ROOT, "tests", "native", "ray_check.cpp")
_dp = ctypes.POINTER(ctypes.c_double)


@pytest.fixture(scope="module")
def rlib(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("ray") / "ray.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-fPIC", "-shared",
                    "-I/usr/local/cuda/include", SRC, "-o", out], check=True)
    return ctypes.CDLL(out)


def update(lib, general, mode, prm, eps, zn, h):
    n = eps.shape[0]
    prm = np.array(prm)
    sig, z, tan = np.empty((n, 6)), np.empty((n, 6)), np.empty((n, 21))
    st = np.empty(n, dtype=np.int32)
    lib.ray_update(general, mode, prm.ctypes.data_as(_dp), ctypes.c_int64(n), eps.ctypes.data_as(_dp),
                   zn.ctypes.data_as(_dp), ctypes.c_double(h), sig.ctypes.data_as(_dp), z.ctypes.data_as(_dp),
                   tan.ctypes.data_as(_dp), st.ctypes.data_as(ctypes.POINTER(ctypes.c_int32)))
    return sig, z, tan, st


# Both solvers are converged to rounding.  FP64 and FP32-bulk: the general solver forms the stress from eps - y
# (absolute rounding of a few 2^-53 of the strain, against a deviatoric part that may be a hundredth of it) and the
# FP32-bulk one carries 2^-45; FP32: the general solver's rescaled constant and eps - y carry some 2^-20.
BOUND = {0: 1e-12, 1: 1e-10, 2: 5e-5}


@pytest.mark.parametrize("mode", [0, 1, 2])
@pytest.mark.parametrize("n_exp", [0.5, 1.0, 2.0, 5.0, 20.0])
def test_ray_equals_the_general_solver(rlib, mode, n_exp):
    prm = synth.MATRIX_16[:4] + (n_exp,)
    for h, amp in ((1e-4, 1.0), (1e-2, 1.0), (1.0, 1.0), (1e-2, 1e-3)):
        eps, zn = synth.material_batch(300, seed=int(n_exp * 10) + mode)
        eps, zn = eps * amp, zn * amp
        a, b = (update(rlib, g, mode, prm, eps, zn, h) for g in (0, 1))
        for x, y in zip(a[:3], b[:3]):
            scale = np.abs(y).max(1)
            assert (np.abs(x - y).max(1) / scale).max() < BOUND[mode], (h, amp)
        assert np.all((a[3] >> 16) & 0xF == 1), "converged, no other flag"
        if mode < 2:  # (the general FP32 Newton reports the iteration cap where its steps stay above 1e-6)
            assert np.all((b[3] >> 16) & 0xF == 1)


@pytest.mark.parametrize("mode", [0, 1, 2])
def test_degenerate_states(rlib, mode):
    """No deviatoric trial strain, one far below the resolution, and non-finite input."""
    eps = np.zeros((4, 6))
    eps[1, :3] = 0.0078125          # hydrostatic, exactly
    eps[2, 0] = 1e-30
    eps[3, 3] = np.nan
    zn = np.zeros((4, 6))
    sig, z, tan, st = update(rlib, 0, mode, synth.MATRIX_16, eps, zn, 0.01)
    assert np.array_equal(z[:2], zn[:2]) and np.array_equal(sig[0], np.zeros(6))
    assert np.all((st[:3] >> 16) & 0xF == 1) and np.all(st[:2] & 0xFFFF == 0)
    assert (st[3] >> 17) & 1
    assert np.all(np.isfinite(tan[:3]))


def ode(lib, general, pair, prm, eps_n, eps, zn, h, rtol, atol, cap):
    n = eps.shape[0]
    prm = np.array(prm)
    sig, z, st = np.empty((n, 6)), np.empty((n, 6)), np.empty(n, dtype=np.int32)
    d = ctypes.c_double
    lib.ray_ode(general, pair, prm.ctypes.data_as(_dp), ctypes.c_int64(n), eps_n.ctypes.data_as(_dp),
                eps.ctypes.data_as(_dp), zn.ctypes.data_as(_dp), d(h), d(rtol), d(atol), cap, sig.ctypes.data_as(_dp),
                z.ctypes.data_as(_dp), st.ctypes.data_as(ctypes.POINTER(ctypes.c_int32)))
    return sig, z, st


@pytest.mark.parametrize("pair", [0, 1])
@pytest.mark.parametrize("n_exp", [1.0, 2.0, 3.0, 4.5, 5.0, 9.0, 25.0])
def test_explicit_pairs_equal_the_general_state(rlib, pair, n_exp):
    """Same substeps (accepted and rejected) and, where they are the same, sigma
    and z to rounding: integer, half-integer and real powers, a cap that cuts
    the integration short, and a zero error scale (atol = 0, zero shears)."""
    prm = synth.MATRIX_16[:4] + (n_exp,)
    eps_n, eps, zn = synth.ode23_batch(200, seed=int(10 * n_exp) + pair)
    zero = np.zeros_like(eps)
    zero[:, 0] = eps[:, 0]
    for args in ((eps_n, eps, zn, 0.1, 1e-3, 1e-6, 100000), (eps_n, eps, zn, 0.1, 1e-5, 1e-9, 7),
                 (np.zeros_like(eps), zero, np.zeros_like(eps), 0.05, 1e-3, 0.0, 100000)):
        a, b = (ode(rlib, g, pair, prm, *args) for g in (0, 1))
        same = a[2] == b[2]
        # a borderline accept or reject may flip between the two roundings (n = 1: its error estimate cancels)
        assert same.mean() > (0.9 if n_exp == 1.0 else 0.99)
        for x, y in zip(a[:2], b[:2]):
            scale = np.abs(y).max()
            assert np.abs(x - y)[same].max() < 1e-10 * scale
