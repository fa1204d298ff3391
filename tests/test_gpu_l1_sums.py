"""The gradients' L1 norms where a few terms are large and the many others just
below half a unit in the last place of one of them: a float32 chain over the
cells of a thread drops the small ones.

Two-pin nets: pins far apart (many gamma) pull their cells with exactly 1, pins
a distance d << gamma apart with about d / gamma.  The limit of the relative error:
one rounding of a cell's |g_x| + |g_y|, five of a warp's tree and one of a
thread's total, 2^-24 each."""
import types

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

U = 2.0 ** -24
BIG = 3 * 256 * 152            # cells of the large nets, numbered first
M = 20 * BIG


def pairs(x, y):
    """Two-pin nets of cells (2 k, 2 k + 1)."""
    m, L = x.size, 64.0
    return types.SimpleNamespace(
        region=(-L / 2, -L / 2, L / 2, L / 2), n=64, target_density=1.0, gamma=0.5, m_mov=m,
        m_fix=0, w=np.full(m, 1.0 / 64, np.float32), h=np.full(m, 1.0 / 64, np.float32),
        fix_x=np.zeros(0, np.float32), fix_y=np.zeros(0, np.float32),
        net_ptr=np.arange(0, m + 1, 2, dtype=np.int32), pin_cell=np.arange(m, dtype=np.int32),
        pin_dx=np.zeros(m, np.float32), pin_dy=np.zeros(m, np.float32), x=x, y=y)


@pytest.fixture(scope="module")
def inst():
    import torch
    from paper_1312_4587_gb300 import fftpl as F
    # the distance whose gradient comes nearest to 2^-24 from below
    d = (np.arange(1, 65) / 32 * U).astype(np.float32)
    few = pairs(np.stack([np.zeros(64, np.float32), d], 1).ravel(), np.zeros(128, np.float32))
    with F.Problem(few) as p:
        gx, gy = torch.empty(128, device="cuda"), torch.empty(128, device="cuda")
        F.fftpl_wa(p.h, torch.from_numpy(few.x).cuda(), torch.from_numpy(few.y).cuda(), few.gamma,
                   gx, gy)
    pull = gx.abs().cpu().numpy()[1::2]
    best = np.where(pull < U, pull, 0).argmax()
    assert pull[best] > 0.6 * U
    x = np.zeros(M, np.float32)
    y = np.linspace(-30, 30, M // 2).astype(np.float32).repeat(2)
    x[0:BIG:2] = -30.0
    x[1:BIG:2] = 30.0
    x[BIG + 1::2] = d[best]
    return pairs(x, y)


def l1(gx, gy):
    return float(gx.double().abs().sum() + gy.double().abs().sum())


@pytest.mark.parametrize("det", [0, 1])
def test_l1_norms(inst, det):
    import torch
    from paper_1312_4587_gb300 import fftpl as F
    x, y = torch.from_numpy(inst.x), torch.from_numpy(inst.y)
    xd, yd = x.cuda(), y.cuda()
    with F.Problem(inst, deterministic=det) as p:
        def near(value, gx, gy):
            ref = l1(gx, gy)
            assert abs(value - ref) <= 7 * U * ref

        g = [torch.empty(M, device="cuda") for _ in range(4)]
        rep = F.fftpl_eval(p.h, xd, yd, inst.gamma, *g)
        assert g[2][0].abs() == 1 and 0.6 * U < g[2][BIG].abs() < U
        near(rep["gN_l1"], g[0], g[1])
        near(rep["gW_l1"], g[2], g[3])
        pin = [torch.empty(M).pin_memory() for _ in range(4)]
        rep = F.fftpl_eval_host(p.h, x.pin_memory(), y.pin_memory(), inst.gamma, *pin)
        near(rep["gN_l1"], pin[0], pin[1])
        near(rep["gW_l1"], pin[2], pin[3])
        F.fftpl_density(p.h, xd, yd, g[0], g[1])
        near(F.fftpl_report(p.h)["gN_l1"], g[0], g[1])
        F.fftpl_wa(p.h, xd, yd, inst.gamma, g[2], g[3])
        near(F.fftpl_report(p.h)["gW_l1"], g[2], g[3])


def test_first_lambda(inst):
    # lambda_0 = ||grad W~||_1 / ||grad N||_1 of the loop's own cell kernel
    import torch
    from paper_1312_4587_gb300 import fftpl as F
    xd, yd = torch.from_numpy(inst.x).cuda(), torch.from_numpy(inst.y).cuda()
    with F.Problem(inst, deterministic=1, gamma_fixed=inst.gamma) as p:
        g = [torch.empty(M, device="cuda") for _ in range(4)]
        F.fftpl_eval(p.h, xd, yd, inst.gamma, *g)
        F.fftpl_place_init(p.h, xd, yd)
        lam = F.fftpl_step(p.h, 1)[0][0]["lam"]
    ref = l1(g[2], g[3]) / l1(g[0], g[1])
    assert abs(lam - ref) <= 14 * U * ref
