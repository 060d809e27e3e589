"""The basic scheme on a non-blocking stream: planning a grid size's own
transforms (their twiddle tables) uses the caller's stream only, so a new grid
size admitted while the legacy default stream is busy neither waits for it nor
depends on it."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def test_planning_leaves_the_default_stream_alone(gsm):
    import torch
    side = torch.cuda.Stream()
    laws = [gsm.norton(*synth.MATRIX_16, precision=gsm.GSM_FP32_FP64FIX), gsm.elastic(*synth.INCLUSION_16)]
    E = synth.ramp(1, [0.001, 0, 0, 0, 0, 0])

    def server():
        sv = gsm.Server(1 << 30, 4, stream=side)
        return sv, sv.submit(synth.sphere_phase(16, 0.2), laws, E, [0.1], tol=1e-4)

    def finish(sv, jid):
        while sum(sv.tick()[:2]):
            pass
        return sv.fetch(jid)["Sigma"]

    ref = finish(*server())  # every kernel of the path is loaded now
    sv, jid = server()
    torch.cuda.synchronize()
    busy = torch.cuda.Event()
    torch.cuda._sleep(2_000_000_000)  # about a second of the legacy default stream
    busy.record()
    sv.tick()
    assert not busy.query()
    assert np.array_equal(finish(sv, jid), ref)
