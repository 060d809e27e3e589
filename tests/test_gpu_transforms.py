"""The library's own transforms with the fused Green pass (every grid size that
has them, and grid sizes that take the library transform): a few iterations of
an elastic two-phase grid against the same iterations with torch's FFT in FP64."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

OWN = [8, 12, 16, 20, 24, 32, 36, 40, 48, 60, 64, 72, 80, 96, 100, 120, 128, 144, 150, 160, 180, 192, 240, 256]
LAWS = [(70.0, 0.3), (140.0, 0.2)]
E0 = [0.002, -0.001, 0.0005, 0.001, -0.0015, 0.003]


def reference(phase, n_iter):
    """Strain of the n_iter-th evaluation and its mean stress, FP64 torch."""
    import torch
    N = phase.shape[0]
    lm = [(E * nu / ((1 + nu) * (1 - 2 * nu)), E / (2 * (1 + nu))) for E, nu in LAWS]
    lam = torch.tensor([a for a, _ in lm], dtype=torch.float64, device="cuda")[phase.long()]
    mu = torch.tensor([b for _, b in lm], dtype=torch.float64, device="cuda")[phase.long()]
    lam0, mu0 = (0.5 * (min(v) + max(v)) for v in zip(*lm))
    f = torch.fft.fftfreq(N, d=1.0 / N, device="cuda", dtype=torch.float64).round()
    k = [f[:, None, None], f[None, :, None], torch.arange(N // 2 + 1, device="cuda", dtype=torch.float64)[None, None]]
    some = sum((c != 0).int() for c in k)
    edge = sum((c.abs() == N // 2).int() for c in k) > 0 if N % 2 == 0 else torch.zeros_like(some, dtype=torch.bool)
    keep = (~((some == 0) | (edge & (some >= 2)))).double()
    k2 = (k[0] ** 2 + k[1] ** 2 + k[2] ** 2).clamp(min=1.0)
    eps = torch.tensor(E0, dtype=torch.float64, device="cuda")[:, None, None, None].expand(6, N, N, N).clone()
    for it in range(n_iter):
        s = mu * eps
        s[:3] = 2 * mu * eps[:3] + lam * eps[:3].sum(0)
        if it == n_iter - 1:
            return eps, s.mean(dim=(1, 2, 3))
        h = [torch.fft.rfftn(s[c]) for c in range(6)]
        q = [(h[a] * k[0] + h[b] * k[1] + h[c] * k[2]) * keep for a, b, c in ((0, 5, 4), (5, 1, 3), (4, 3, 2))]
        kq = (k[0] * q[0] + k[1] * q[1] + k[2] * q[2]) * (lam0 + mu0) / (mu0 * (lam0 + 2 * mu0)) / k2 ** 2
        for c, (i, j) in enumerate(((0, 0), (1, 1), (2, 2), (1, 2), (0, 2), (0, 1))):
            d = (k[j] * q[i] + k[i] * q[j]) / (2 * mu0 * k2) - kq * k[i] * k[j]
            eps[c] -= torch.fft.irfftn(d, s=(N, N, N)) * (1.0 if c < 3 else 2.0)


def fields(gsm, N, precision, n_iter):
    import torch
    g = torch.Generator(device="cuda").manual_seed(N)
    phase = (torch.rand((N, N, N), generator=g, device="cuda") < 0.3).to(torch.uint8)
    laws = [gsm.elastic(*p) for p in LAWS]
    ctx = gsm.ms_create(phase, laws, precision)
    eps = torch.empty((6, N ** 3), dtype=torch.float64, device="cuda")
    out = gsm.ms_run(ctx, [E0], [0.1], tol=1e-14, forced_iters=[n_iter], eps=eps, z=torch.empty_like(eps),
                     switch_tol=1e-14)
    # an FP32-bulk step ends with an FP64 evaluation at the strain of its last FP32 one
    ref, mean = reference(phase, n_iter - 1 if precision == gsm.MS_PREC_FP32_BULK else n_iter)
    return eps.reshape(6, N, N, N), out["Sigma"][0], ref, mean.cpu().numpy()


# FP64: a transform's rounding is below log2(N^3) 2^-53 of its largest values (24 x 1.1e-16 at 256), four of them;
# FP32 bulk (the strain of the last evaluation comes from FP32 passes): the same in 2^-24.
@pytest.mark.parametrize("N", OWN + [9, 14, 22, 34])
@pytest.mark.parametrize("precision,bound", [(0, 2e-14), (1, 1e-5)])
def test_iterations_match_torch(gsm, N, precision, bound):
    eps, Sigma, ref, mean = fields(gsm, N, precision, 4)
    scale = float(ref.abs().max())
    assert float((eps - ref).abs().max()) < bound * scale
    assert np.max(np.abs(Sigma - mean)) < bound * np.max(np.abs(mean))
