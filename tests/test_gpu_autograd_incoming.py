"""Incoming gradients that the device-side gather cannot take as they lie in
memory: one that carries a forward-mode tangent, one whose memory holds its
negative."""
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def case():
    import torch
    inst = synth.make_instance("medium")
    return (inst, torch.from_numpy(inst.x).cuda().requires_grad_(True),
            torch.from_numpy(inst.y).cuda().requires_grad_(True))


def test_forward_mode_tangent_of_the_incoming_gradient(case):
    # the gradient is linear in the incoming one: its tangent is the gradient
    # for the tangent
    import torch
    import torch.autograd.forward_ad as fw
    from paper_1312_4587_gb300 import fftpl as F
    from paper_1312_4587_gb300.autograd import density_energy
    inst, x, y = case
    w = torch.tensor(0.3, dtype=torch.float64, device="cuda")
    t = torch.tensor(-2.0, dtype=torch.float64, device="cuda")
    with F.Problem(inst, deterministic=1) as p:
        N = density_energy(x, y, p)
        ref = torch.autograd.grad(N, (x, y), grad_outputs=w, retain_graph=True)
        tan = torch.autograd.grad(N, (x, y), grad_outputs=t, retain_graph=True)
        with fw.dual_level():
            got = torch.autograd.grad(N, (x, y), grad_outputs=fw.make_dual(w, t))
            for g, r, d in zip(got, ref, tan):
                u = fw.unpack_dual(g)
                assert torch.equal(u.primal, r)
                assert u.tangent is not None
                assert torch.equal(u.tangent, d)


def test_incoming_gradient_with_the_negative_bit(case):
    # the imaginary part of a conjugate is a view that stands for the negative
    # of what lies in memory
    import torch
    from paper_1312_4587_gb300 import fftpl as F
    from paper_1312_4587_gb300.autograd import density_energy
    inst, x, y = case
    w = torch.tensor([0.5, 0.3], dtype=torch.float64, device="cuda")
    neg = torch.view_as_complex(w).conj().imag
    assert neg.is_neg() and neg.item() == -0.3
    with F.Problem(inst, deterministic=1) as p:
        N = density_energy(x, y, p)
        got = torch.autograd.grad(N, (x, y), grad_outputs=neg, retain_graph=True)
        ref = torch.autograd.grad(N, (x, y), grad_outputs=neg.clone().resolve_neg())
        for g, r in zip(got, ref):
            assert torch.equal(g, r)
