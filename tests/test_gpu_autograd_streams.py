"""density_energy where its device-side path may not be taken: on another
stream than the handle's, with a batch of incoming gradients, and where the
gradient is itself differentiated by the incoming one.  The handle
is deterministic, so every way has to give the same bits."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def F():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_1312_4587_gb300 import fftpl
    fftpl.lib()
    return fftpl


def forward_backward(p, x, y, mode):
    from paper_1312_4587_gb300.autograd import density_energy
    x = x.detach().clone().requires_grad_(True)
    y = y.detach().clone().requires_grad_(True)
    N = density_energy(x, y, p, mode)
    (N * 0.3).backward()
    return N.item(), x.grad.cpu().numpy(), y.grad.cpu().numpy()


@pytest.mark.parametrize("mode", ["gather", "adjoint"])
def test_other_stream_same_bits(F, mode):
    import torch
    inst = synth.make_instance("medium")
    x = torch.from_numpy(inst.x).cuda()
    y = torch.from_numpy(inst.y).cuda()
    with F.Problem(inst, deterministic=1) as p:
        ref = forward_backward(p, x, y, mode)
        torch.cuda.synchronize()
        with torch.cuda.stream(torch.cuda.Stream()):
            got = forward_backward(p, x, y, mode)
            torch.cuda.synchronize()
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(side):
        with F.Problem(inst, deterministic=1) as p:
            own = forward_backward(p, x, y, mode)
            torch.cuda.synchronize()
    for r in (got, own):
        assert r[0] == ref[0]
        assert np.array_equal(r[1], ref[1]) and np.array_equal(r[2], ref[2])


def test_batched_gradients(F):
    import torch
    from paper_1312_4587_gb300.autograd import density_energy
    inst = synth.make_instance("medium")
    x = torch.from_numpy(inst.x).cuda().requires_grad_(True)
    y = torch.from_numpy(inst.y).cuda().requires_grad_(True)
    w = torch.tensor([1.0, -2.5, 0.25], dtype=torch.float64, device="cuda")
    with F.Problem(inst, deterministic=1) as p:
        N = density_energy(x, y, p)
        gx, gy = torch.autograd.grad(N, (x, y), grad_outputs=w, is_grads_batched=True,
                                     retain_graph=True)
        for k in range(3):
            hx, hy = torch.autograd.grad(N, (x, y), grad_outputs=w[k], retain_graph=True)
            assert torch.equal(gx[k], hx) and torch.equal(gy[k], hy)


def test_gradient_differentiable_by_the_incoming_one(F):
    # d/dw sum(w dN/dx) = sum(dN/dx)
    import torch
    from paper_1312_4587_gb300.autograd import density_energy
    inst = synth.make_instance("medium")
    x = torch.from_numpy(inst.x).cuda().requires_grad_(True)
    y = torch.from_numpy(inst.y).cuda()
    w = torch.tensor(0.3, dtype=torch.float64, device="cuda", requires_grad=True)
    with F.Problem(inst, deterministic=1) as p:
        N = density_energy(x, y, p)
        gx, = torch.autograd.grad(N, x, grad_outputs=w, create_graph=True)
        one, = torch.autograd.grad(N, x, retain_graph=True)
        plain, = torch.autograd.grad(N, x, grad_outputs=w.detach())
        assert torch.equal(gx, plain)
        v = one.sign()
        dw, = torch.autograd.grad((gx * v).sum(), w)
        ref = one.double().abs().sum().item()
        # a float32 sum of m terms
        assert abs(dw.item() - ref) <= 2.0 ** -24 * x.numel() * ref
