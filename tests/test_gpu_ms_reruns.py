"""A basic-scheme context keeps nothing of a run for the next: FP32-bulk runs
repeated on one context, after a run that ended non-finite, and resumed, bit
for bit as on a context of their own (own transforms and cuFFT grid sizes)."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

E2 = synth.ramp(2, [0.002, 0, 0, 0.001, 0, 0])
H2 = [0.1, 0.1]


def context(gsm, N):
    import torch
    phase = torch.from_numpy(synth.sphere_phase(N, 0.2)).cuda()
    laws = [gsm.norton(*synth.MATRIX_16, precision=gsm.GSM_FP32_FP64FIX), gsm.elastic(*synth.INCLUSION_16)]
    return gsm.ms_create(phase, laws, gsm.MS_PREC_FP32_BULK)


def run(gsm, ctx, N, E, h, forced, **kw):
    import torch
    eps = kw.pop("eps", torch.empty((6, N ** 3), dtype=torch.float64, device="cuda"))
    z = kw.pop("z", torch.empty_like(eps))
    out = gsm.ms_run(ctx, E, h, tol=1e-12, forced_iters=forced, eps=eps, z=z, switch_tol=1e-12, **kw)
    return out["Sigma"], eps.cpu().numpy().copy(), z.cpu().numpy().copy()


@pytest.mark.parametrize("N", [16, 14])
@pytest.mark.parametrize("between", [None, 0.05, 1e30, np.nan])
def test_repeated_runs_are_the_same_run(gsm, N, between):
    ref = run(gsm, context(gsm, N), N, E2, H2, [9, 9])
    assert all(np.all(np.isfinite(a)) for a in ref)
    ctx = context(gsm, N)
    if between is None:
        run(gsm, ctx, N, E2, H2, [9, 9])
    else:  # another load: larger, beyond the FP32 range of the spectra, not a number
        run(gsm, ctx, N, [[between, 0, 0, 0, 0, 0]], [0.1], [5], check=False)
    again = run(gsm, ctx, N, E2, H2, [9, 9])
    for a, b in zip(ref, again):
        assert np.array_equal(a, b)


def test_resumed_run_continues_the_run(gsm):
    """N a power of two: the export of the strain (N^3 eps / N^3) is exact."""
    import torch
    N = 16
    ref = run(gsm, context(gsm, N), N, E2, H2, [9, 9])
    eps = torch.empty((6, N ** 3), dtype=torch.float64, device="cuda")
    z = torch.empty_like(eps)
    run(gsm, context(gsm, N), N, E2[:1], H2[:1], [9], eps=eps, z=z)
    two = run(gsm, context(gsm, N), N, E2[1:], H2[1:], [9], eps=eps, z=z, resume=True, E_prev=E2[0])
    assert np.array_equal(two[0][-1], ref[0][-1])
    for a, b in zip(ref[1:], two[1:]):
        assert np.array_equal(a, b)
