"""The explicit ODE pairs of the Norton law (csrc/ode_ray.cuh, host build) in
units and at exponents where a power of the shear modulus alone leaves the
FP64 range, against the AD state of the same potentials: converged with the
same substeps, and within the error control of each other (10 (rtol |sigma| +
atol), the criterion of the other ODE tests).  Not to rounding: the AD state's
error estimate is a difference of two stresses, whose cancellation moves its
substep sizes (n = 60: 5e-8 of the stress from a 40-digit integration, where
this state is within 2e-9)."""
import numpy as np
import pytest

import synth
from test_ray_host import ode, rlib  # noqa: F401  (rlib is a fixture)


@pytest.mark.parametrize("pair", [0, 1])
@pytest.mark.parametrize("prm", [(70e9, 0.3, 1e8, 1.0, 30.0), (210e9, 0.3, 2e8, 1.0, 28.0),
                                 (200e3, 0.3, 100.0, 1.0, 60.0), (70.0, 0.3, 0.1, 1.0, 120.0)])
def test_units_and_high_exponents(rlib, pair, prm):  # noqa: F811
    eps_n, eps, zn = synth.ode23_batch(200, seed=int(prm[4]) + pair)
    rtol, atol = 1e-3, 1e-5 * prm[2]
    a, b = (ode(rlib, g, pair, prm, eps_n, eps, zn, 0.1, rtol, atol, 20000) for g in (0, 1))
    assert np.all((b[2] >> 16) & 7 == 1) and np.all((a[2] >> 16) & 7 == 1), "converged, no other flag"
    assert (a[2] == b[2]).mean() > 0.99
    assert np.all(np.abs(a[0] - b[0]) <= 10 * (rtol * np.abs(b[0]).max(1, keepdims=True) + atol))
    assert np.all(np.abs(a[1] - b[1]).max(1) <= 10 * (rtol * np.abs(b[0]).max(1) + atol) / (prm[0] / 2.6))
