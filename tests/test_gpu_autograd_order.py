"""density_energy on a stream that is not the handle's: the same bits with
work of several milliseconds ahead of the positions on the caller's stream and
ahead of the gather on the handle's."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

CYCLES = 20_000_000   # about 10 ms


@pytest.mark.parametrize("mode", ["gather", "adjoint"])
@pytest.mark.parametrize("own", [False, True])
def test_late_positions_and_a_busy_handle(mode, own):
    import torch
    from paper_1312_4587_gb300 import fftpl as F
    from paper_1312_4587_gb300.autograd import density_energy
    inst = synth.make_instance("medium")
    x = torch.from_numpy(inst.x).cuda()
    y = torch.from_numpy(inst.y).cuda()
    hs = torch.cuda.Stream() if own else torch.cuda.default_stream()
    torch.cuda.synchronize()

    def go(p, slow):
        if slow:
            torch.cuda._sleep(CYCLES)
        xs = torch.zeros_like(x).copy_(x).requires_grad_(True)
        ys = torch.zeros_like(y).copy_(y).requires_grad_(True)
        N = density_energy(xs, ys, p, mode)
        loss = N * 0.3
        if slow:
            with torch.cuda.stream(hs):
                torch.cuda._sleep(CYCLES)
        loss.backward()
        gx, gy = xs.grad * 1.0, ys.grad * 1.0   # on the caller's stream
        torch.cuda.current_stream().synchronize()
        return N.item(), gx.cpu().numpy(), gy.cpu().numpy()

    with torch.cuda.stream(hs):
        with F.Problem(inst, deterministic=1) as p:
            ref = go(p, False)
            torch.cuda.synchronize()
            with torch.cuda.stream(torch.cuda.Stream()):
                got = go(p, True)
            torch.cuda.synchronize()
    assert got[0] == ref[0]
    assert np.array_equal(got[1], ref[1]) and np.array_equal(got[2], ref[2])
