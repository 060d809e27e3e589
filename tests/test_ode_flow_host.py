"""Internal variables of the explicit ODE pairs in the elastic deviatoric strain
(csrc/ode_ray.cuh, host build) against the AD state: flows many orders below the
strain, hydrostatic strains (no flow at all) and non-finite input."""
import numpy as np
import pytest

import synth
from test_ray_host import ode, rlib  # noqa: F401  (rlib is a fixture)

PRM = synth.MATRIX_16[:4]


# One substep (a second one starts at a size that the AD state's cancelling stress difference sets, and the
# flow of a single voxel with two differed by 3e-12): the flow's relative rounding is some n 2^-52.
@pytest.mark.parametrize("pair", [0, 1])
@pytest.mark.parametrize("n_exp", [1.0, 2.0, 4.5, 5.0])
@pytest.mark.parametrize("scale", [1e-3, 1e-5, 1e-7])
def test_small_flows(rlib, pair, n_exp, scale):  # noqa: F811
    _, eps, _ = synth.ode23_batch(200, seed=9)
    zero = np.zeros_like(eps)
    # h: the n = 1 flow is a fixed fraction of the strain whatever its size, keep it small too
    h = 1e-8 if n_exp == 1.0 else 0.1
    a, b = (ode(rlib, g, pair, PRM + (n_exp,), zero, eps * scale, zero, h, 1e-3, 1e-20, 1000) for g in (0, 1))
    assert (a[2] == b[2]).mean() > 0.99 and np.all((a[2] >> 16) & 7 == 1)
    assert np.all(np.abs(b[1]).max(1) > 0)
    one = (a[2] == b[2]) & (a[2] & 0xFFFF == 1) & ((a[2] >> 20) & 0x7FF == 0)
    assert np.all(np.abs(a[1] - b[1]).max(1)[one] <= 1e-12 * np.abs(b[1]).max(1)[one])


@pytest.mark.parametrize("pair", [0, 1])
@pytest.mark.parametrize("n_exp", [1.0, 5.0])
def test_hydrostatic_strains_do_not_flow(rlib, pair, n_exp):  # noqa: F811
    p = np.random.default_rng(5).uniform(-0.01, 0.01, 50)
    eps = np.zeros((50, 6))
    eps[:, :3] = p[:, None]
    a = ode(rlib, 0, pair, PRM + (n_exp,), 0.3 * eps, eps, np.zeros_like(eps), 0.1, 1e-3, 1e-6, 1000)
    assert np.array_equal(a[1], np.zeros_like(eps)) and np.all((a[2] >> 16) & 7 == 1)


@pytest.mark.parametrize("pair", [0, 1])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_non_finite_input(rlib, pair, bad):  # noqa: F811
    """One non-finite entry in eps_n, eps or z_n: the status words and where the results are finite."""
    base = synth.ode23_batch(18, seed=3)
    args = [x.copy() for x in base]
    for k in range(18):
        args[k // 6][k, k % 6] = bad
    a, b = (ode(rlib, g, pair, PRM + (5.0,), *args, 0.1, 1e-3, 1e-6, 40) for g in (0, 1))
    assert np.array_equal(a[2], b[2])
    if np.isnan(bad):
        assert np.array_equal(np.isfinite(a[0]), np.isfinite(b[0]))
        assert np.array_equal(np.isfinite(a[1]), np.isfinite(b[1]))
