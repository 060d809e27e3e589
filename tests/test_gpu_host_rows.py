"""gsm_update_host without a chunk size, rows off 32-byte boundaries: the route
(the kernel on the host memory, or staged copies) follows the lengths on both
sides of its lines, the results are the device update's bit for bit, and it is
not slower than staging by hand."""
import pytest

import synth

pytestmark = pytest.mark.gpu


def arrays(gsm, n, precision, tangent):
    import torch
    dt = torch.float32 if precision == 2 else torch.float64
    g = torch.Generator(device="cuda").manual_seed(n)
    eps = (torch.rand((6, n), generator=g, device="cuda", dtype=dt) * 2 - 1) * 0.02
    y = (torch.rand((5, n), generator=g, device="cuda", dtype=dt) * 2 - 1) * 0.005
    zn = torch.stack([y[0], y[1], -y[0] - y[1], y[2], y[3], y[4]])
    dev = [eps, zn, torch.empty_like(eps), torch.empty_like(eps),
           torch.empty((21, n), dtype=dt, device="cuda") if tangent else None]
    host = [torch.empty(a.shape, dtype=dt).pin_memory() if a is not None else None for a in dev]
    host[0].copy_(eps)
    host[1].copy_(zn)
    torch.cuda.synchronize()
    return gsm.norton(*synth.MATRIX_16, precision=precision), dev, host


def call(f, mat, a, **kw):
    f(mat, a[0], a[1], 0.01, a[2], a[3], a[4], **kw)


# (precision, tangent, voxels): each side of each line of the rule, and rows at 32-byte boundaries beyond it
@pytest.mark.parametrize("precision,tangent,n", [
    (2, True, (1 << 19) - 1), (2, True, (1 << 19) + 5), (2, True, (1 << 19) + 8), (2, True, (1 << 21) + 3),
    (2, False, (1 << 22) - 1), (2, False, (1 << 22) + 9), (0, True, (1 << 21) - 1), (0, True, (1 << 21) + 7),
    (1, False, (1 << 21) + 7)])
def test_same_results_on_either_route(gsm, precision, tangent, n):
    import torch
    mat, dev, host = arrays(gsm, n, precision, tangent)
    call(gsm.gsm_update, mat, dev)
    call(gsm.gsm_update_host, mat, host)
    torch.cuda.synchronize()
    for a, b in zip(dev[2:], host[2:]):
        assert a is None or torch.equal(a.cpu(), b)


def test_under_capture(gsm):
    """A captured call keeps the one kernel on the host memory."""
    import torch
    n = (1 << 19) + 5
    mat, dev, host = arrays(gsm, n, 2, True)
    call(gsm.gsm_update, mat, dev)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        call(gsm.gsm_update_host, mat, host)
    graph.replay()
    torch.cuda.synchronize()
    for a, b in zip(dev[2:], host[2:]):
        assert torch.equal(a.cpu(), b)


def test_long_odd_rows_are_not_slower_than_staged(gsm):
    import torch
    mat, _, host = arrays(gsm, (1 << 22) + 9, 2, True)

    times = {0: [], 1 << 19: []}
    for _ in range(10):  # in turn: the link's rate drifts by some percent
        for chunk, out in times.items():
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            call(gsm.gsm_update_host, mat, host, chunk=chunk)
            b.record()
            torch.cuda.synchronize()
            out.append(a.elapsed_time(b))
    direct, staged = (min(t[1:]) for t in times.values())
    assert direct < 1.15 * staged  # (1.3 times by the kernel on the host memory)
