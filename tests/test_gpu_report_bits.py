"""Deterministic mode: fftpl_eval_host reports the same bits through pinned
buffers (kernels over the host link), through pageable ones (copies) and as
fftpl_eval, one block of cells, more than the cell kernels' grid takes at once,
and between."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name", ["tiny", "medium", "precision_sub", "large", "diff"])
def test_host_routes_report_the_same_bits(name):
    import torch
    from paper_1312_4587_gb300 import fftpl as F
    inst = synth.make_instance(name)
    m = inst.m_mov
    x, y = torch.from_numpy(inst.x), torch.from_numpy(inst.y)
    with F.Problem(inst, deterministic=1) as p:
        g = [torch.empty(m, device="cuda") for _ in range(4)]
        dev = F.fftpl_eval(p.h, x.cuda(), y.cuda(), inst.gamma, *g)
        pin = [torch.empty(m).pin_memory() for _ in range(4)]
        pinned = F.fftpl_eval_host(p.h, x.pin_memory(), y.pin_memory(), inst.gamma, *pin)
        page = [np.empty(m, np.float32) for _ in range(4)]
        paged = F.fftpl_eval_host(p.h, inst.x.copy(), inst.y.copy(), inst.gamma, *page)
    assert pinned == paged == dev
    for a, b, c in zip(g, pin, page):
        assert np.array_equal(a.cpu().numpy(), c) and np.array_equal(b.numpy(), c)
