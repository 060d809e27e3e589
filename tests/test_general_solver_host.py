"""The general implicit-Euler path (csrc/solver.cuh, csrc/voxel.cuh: segment
search, AD-driven Newton, tangent from the AD blocks) against the FP64 oracle.
The shipped laws take the scalar equation on the GPU, so the general path is
instantiated on the host only, on the Norton potentials without the declaration
that selects the scalar one; here it is held to the oracle by itself, and not only
to the scalar update that it is compared with elsewhere."""
import numpy as np
import pytest

import oracle as O
import synth
from test_host_solver import _trial_cases
from test_ray_host import rlib, update  # noqa: F401  (rlib is a fixture)


@pytest.mark.parametrize("mode", [0, 1])
def test_general_solver_matches_oracle(rlib, mode):  # noqa: F811
    eps, zn = synth.material_batch(3000, seed=5)
    iu = np.triu_indices(6)
    for h in (1e-3, 1e-2, 1e-1):
        sig, z, tan, st = update(rlib, 1, mode, synth.MATRIX_16, eps, zn, h)
        s2, z2, C2 = O.update(O.KIND_NORTON, synth.MATRIX_16, eps, zn, h, tangent=True)
        assert np.all((st >> 16) & 0xF == 1) and np.all((st >> 8) & 0xFF >= 1), "converged by Newton steps"
        assert (np.abs(sig - s2).max(1) / np.abs(s2).max(1)).max() < 1e-11
        assert (np.abs(z - z2).max(1) / np.abs(z2).max(1)).max() < 1e-11
        assert (np.abs(tan - C2[:, iu[0], iu[1]]).max(1) / np.abs(C2).max((1, 2))).max() < 1e-11


@pytest.mark.parametrize("case", ["hydrostatic", "tiny_deviatoric", "unloading"])
@pytest.mark.parametrize("mode", [0, 1])
def test_general_solver_small_trial_states(rlib, case, mode):  # noqa: F811
    """Deviatoric trial strains from 1e-25 to 1e-1, alone, on a hydrostatic strain, or on an accumulated viscous
    strain: converged, sigma to 1e-10, z to 1e-10 of the flow and the rounding of the inputs."""
    rng = np.random.default_rng(40 + ["hydrostatic", "tiny_deviatoric", "unloading"].index(case) * 2 + mode)
    eps, zn = _trial_cases(case, 300, rng)
    for n_exp in (1.0, 2.0, 5.0, 10.0, 20.0):
        prm = synth.MATRIX_16[:4] + (n_exp,)
        for h in (1e-4, 1e-2, 1.0):
            sig, z, _, st = update(rlib, 1, mode, prm, eps, zn, h)
            s2, z2 = O.update(O.KIND_NORTON, prm, eps, zn, h)
            assert np.all((st >> 16) & 0xF == 1)
            assert (np.abs(sig - s2).max(1) / np.abs(s2).max(1)).max() < 1e-10
            bound = 1e-10 * np.abs(z2 - zn).max(1) + 2e-15 * (np.abs(eps).max(1) + np.abs(zn).max(1))
            assert np.all(np.abs(z - z2).max(1) <= bound)
