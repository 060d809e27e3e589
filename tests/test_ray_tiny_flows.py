"""Flows many orders below the trial strain in the FP32-bulk update (csrc/ray.cuh):
the double-float root takes them at its own accuracy (host build), and at about the
cost of any other flow (GPU)."""
import numpy as np
import pytest

import synth
from test_ray_host import rlib, update  # noqa: F401  (rlib is a fixture)
from test_ray_small_exponents import radial_return


# theta^(1/n) is the power's result (2^-45) times rounded factors: some n 2^-43 of the flow
@pytest.mark.parametrize("n_exp", [3.0, 10.0, 20.0, 50.0])
@pytest.mark.parametrize("amp", [1e-1, 1e-2, 1e-3])
def test_accuracy_of_tiny_flows(rlib, n_exp, amp):  # noqa: F811
    prm = synth.MATRIX_16[:4] + (n_exp,)
    eps, _ = synth.material_batch(300, seed=8)
    eps, zn = eps * amp, np.zeros_like(eps)
    sig, z, _, st = update(rlib, 0, 1, prm, eps, zn, 0.01)
    s2, z2 = radial_return(prm, eps, zn, 0.01)
    assert np.all((st >> 16) & 0xF == 1) and np.all((st >> 20) & 0xF >= 1), "solved by the correction"
    assert np.all(np.abs(z - z2).max(1) <= n_exp * 2.0 ** -43 * np.abs(z2).max(1))
    assert np.all(np.abs(sig - s2).max(1) <= 1e-12 * np.abs(s2).max(1))


@pytest.mark.gpu
def test_nearly_elastic_voxels_cost_no_more(gsm):
    """Strains of 2e-5 at n = 20 (flows below 2^-100 of them) against the flowing batch: below twice its time (three
    times by the FP64 root)."""
    import torch
    n = 1 << 22
    g = torch.Generator(device="cuda").manual_seed(5)
    eps = (torch.rand((6, n), generator=g, device="cuda", dtype=torch.float64) * 2 - 1) * 0.02
    zn, sig, z = torch.zeros_like(eps), torch.empty_like(eps), torch.empty_like(eps)
    mat = gsm.norton(*synth.MATRIX_16[:4], 20.0, precision=gsm.GSM_FP32_FP64FIX)

    def best(e):
        times = []
        for _ in range(5):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            gsm.gsm_update(mat, e, zn, 0.01, sig, z)
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b))
        return min(times[1:])

    flowing = best(eps)
    assert best(eps * 1e-3) < 2.0 * flowing
