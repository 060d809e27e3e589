"""The scalar update (csrc/ray.cuh, host build) at Norton exponents far below
one, rates and step sizes of any unit: the constant of the scalar equation
leaves the FP64 range there (n = 0.03 and edot0 h of 1e-6 against strains of
1e-2) and belongs to a scaled trial strain.  Against the radial return in
extended precision."""
import numpy as np
import pytest

import synth
from test_ray_host import rlib, update  # noqa: F401  (rlib is a fixture)


def radial_return(prm, eps, zn, h):
    E, nu, s0, e0, n = (np.longdouble(v) for v in prm)
    mu, kappa = E / (2 * (1 + nu)), E / (3 * (1 - 2 * nu))
    dev = eps.astype(np.longdouble) - zn
    z = zn.astype(np.longdouble)
    z[:, 2] = -z[:, 0] - z[:, 1]
    dev[:, 2] = eps[:, 2].astype(np.longdouble) - z[:, 2]
    tr = eps[:, :3].astype(np.longdouble).sum(1)
    dev[:, :3] -= tr[:, None] / 3
    norm2 = (dev[:, :3] ** 2).sum(1) + (dev[:, 3:] ** 2).sum(1) / 2
    trial, c = 2 * mu * np.sqrt(np.longdouble(1.5) * norm2), 3 * mu * np.longdouble(h) * e0
    # s0 x + c x^n = trial, Newton in ln x from above
    u = np.minimum(np.log(trial / s0), np.log(trial / c) / n)
    for _ in range(80):
        a, b = s0 * np.exp(u), c * np.exp(n * u)
        u = u - (a + b - trial) / (a + n * b)
    a, b = s0 * np.exp(u), c * np.exp(n * u)
    w = np.array([2, 2, 2, 1, 1, 1], dtype=np.longdouble) * mu
    sig = w * (a / (a + b))[:, None] * dev
    sig[:, :3] += kappa * tr[:, None]
    return sig.astype(np.float64), (z + (b / (a + b))[:, None] * dev).astype(np.float64)


# FP64 and the FP32-bulk mode (2^-45): sigma against its largest entry, which the hydrostatic part sets; FP32: 2^-24
# through the power's argument, the stress and the sums
BOUND = {0: 1e-12, 1: 1e-11, 2: 1e-5}


@pytest.mark.parametrize("mode", [0, 1, 2])
@pytest.mark.parametrize("n_exp", [0.003, 0.01, 0.03, 0.05, 0.1])
def test_small_exponents(rlib, mode, n_exp):  # noqa: F811
    base_eps, base_zn = synth.material_batch(40, seed=11)
    for edot0 in (1.0, 1e-3, 1e-9, 1e4):
        for h in (1e-6, 1e-3, 0.1, 1e5):
            for amp in (1.0, 1e-3):
                prm = (70.0, 0.3, 0.1, edot0, n_exp)
                eps, zn = (a * amp for a in (base_eps, base_zn))
                if mode == 2:
                    eps, zn = (a.astype(np.float32).astype(np.float64) for a in (eps, zn))
                got = update(rlib, 0, mode, prm, eps, zn, h)
                assert np.all((got[3] >> 16) & 0xF == 1)
                for a, b in zip(got[:2], radial_return(prm, eps, zn, h)):
                    assert np.all(np.abs(a - b).max(1) <= BOUND[mode] * np.abs(b).max(1)), (edot0, h, amp)
