"""The voxel schedule of the ODE update without tangent: every voxel of ragged
batches is taken once, whatever its block, and a flow confined to one part of
the field is shared by all blocks."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def fields(*arrays):
    import torch
    return [torch.from_numpy(np.ascontiguousarray(a.T)).cuda() for a in arrays]


def test_ragged_batches(gsm):
    """A voxel's result does not depend on the batch: the first n voxels alone, bit for bit, nothing beyond them."""
    import torch
    N = 70003
    eps_n, eps, zn = fields(*synth.ode23_batch(N, seed=4))
    mat = gsm.norton(*synth.MATRIX_16)
    ref = [torch.empty_like(eps) for _ in range(2)]
    gsm.gsm_update_ode23(mat, eps_n, eps, zn, 0.1, *ref)
    for n in (1, 7, 8, 9, 127, 128, 129, 1031, 58367, 58368, 58369, N - 1):  # 58368 = 152 x 3 x 128
        out = [torch.full_like(eps, -7.0) for _ in range(2)]
        gsm.gsm_update_ode23(mat, eps_n, eps, zn, 0.1, *out, n_vox=n)
        for a, b in zip(out, ref):
            assert torch.equal(a[:, :n], b[:, :n]) and torch.all(a[:, n:] == -7.0)


@pytest.mark.parametrize("method", ["ode23", "ode12"])
def test_confined_flow_is_shared_by_all_blocks(gsm, method):
    """2 % of 2^20 voxels flow: in one run of the field they take no longer than twice what they take in random order
    (one contiguous range a block: about six times)."""
    import torch
    N, k = 1 << 20, 20000
    eps_n, eps, zn = synth.ode23_batch(k, seed=6)
    batch = [np.zeros((N, 6)) for _ in range(3)]
    for b, a in zip(batch, (eps_n, eps, zn)):
        b[:k] = a
    clustered = fields(*batch)
    order = torch.randperm(N, generator=torch.Generator().manual_seed(1)).cuda()
    shuffled = [a[:, order].contiguous() for a in clustered]
    mat = gsm.norton(*synth.MATRIX_16)
    sig, z = torch.empty_like(clustered[0]), torch.empty_like(clustered[0])

    def best(args):
        times = []
        for _ in range(4):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            gsm.gsm_update_ode23(mat, *args, 0.1, sig, z, method=method)
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b))
        return min(times[1:])

    assert best(clustered) < 2.0 * best(shuffled)
