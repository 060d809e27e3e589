"""Rounding of the FP32 scalar update (csrc/ray.cuh, host build): its 2-norm
error against the FP64 update of the same FP32 inputs is no larger than the
general FP32 solver's, in the stress and in the internal variables, on the
material batch, and with a hydrostatic strain many times the deviatoric one
(whose rounding must not reach z: bound 2^-24, one rounding of z)."""
import numpy as np
import pytest

import synth
from test_ray_host import rlib, update  # noqa: F401  (rlib is a fixture)


def errors(lib, general, prm, eps, zn, h):
    exact = update(lib, 0, 0, prm, eps, zn, h)
    got = update(lib, general, 2, prm, eps, zn, h)
    return [np.linalg.norm(a - b) / np.linalg.norm(b) for a, b in zip(got[:2], exact[:2])]


@pytest.mark.parametrize("n_exp", [1.0, 2.0, 3.0, 5.0, 10.0, 20.0])
@pytest.mark.parametrize("h", [1e-3, 1e-2, 1e-1])
def test_no_larger_than_the_general_solver(rlib, n_exp, h):  # noqa: F811
    prm = synth.MATRIX_16[:4] + (n_exp,)
    eps, zn = (a.astype(np.float32).astype(np.float64) for a in synth.material_batch(20000, seed=int(n_exp)))
    for a, b in zip(errors(rlib, 0, prm, eps, zn, h), errors(rlib, 1, prm, eps, zn, h)):
        assert a <= b


@pytest.mark.parametrize("n_exp", [1.0, 3.0, 10.0])
def test_hydrostatic_strain_does_not_reach_z(rlib, n_exp):  # noqa: F811
    prm = synth.MATRIX_16[:4] + (n_exp,)
    eps, zn = synth.material_batch(20000, seed=77)
    eps = zn + 0.05 * eps
    eps[:, :3] += 0.01
    eps, zn = (a.astype(np.float32).astype(np.float64) for a in (eps, zn))
    assert errors(rlib, 0, prm, eps, zn, 0.1)[1] < 2.0 ** -24
