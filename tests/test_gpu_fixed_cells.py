"""The fixed cells' map at the edges of the rasteriser's rules: one cell, as
many as blocks and one more, several rounds of a block's threads, spans of 16
and 17 bins, macros side by side in the list, cells beyond the region."""
import types

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def instance(m_fix, n, seed):
    rng = np.random.default_rng(seed)
    L = float(2 * n)
    w = rng.choice([0.5, 2.0, 7.0, 8.0], m_fix).astype(np.float32)
    h = rng.choice([0.5, 2.0, 6.0, 8.0], m_fix).astype(np.float32)
    w[:5] = h[:5] = L / 4
    x = rng.uniform(-4, L + 4, m_fix).astype(np.float32)
    y = rng.uniform(-4, L + 4, m_fix).astype(np.float32)
    x[::3] = 2.0 * np.rint(x[::3] / 2)     # edges on bin edges: spans of 4 x 4 bins and more
    y[::3] = 2.0 * np.rint(y[::3] / 2)
    one = np.ones(1, np.float32)
    return types.SimpleNamespace(
        region=(0.0, 0.0, L, L), n=n, target_density=1.0, gamma=1.0, m_mov=1, m_fix=m_fix,
        w=np.concatenate([one, w]), h=np.concatenate([one, h]), fix_x=x, fix_y=y,
        net_ptr=np.zeros(1, np.int32), pin_cell=np.zeros(0, np.int32),
        pin_dx=np.zeros(0, np.float32), pin_dy=np.zeros(0, np.float32), x=one * -9, y=one * -9)


@pytest.mark.parametrize("m_fix", [1, 127, 2432, 2433, 5000, 2432 * 128 + 1])
def test_macro_map(m_fix):
    import torch
    from paper_1312_4587_gb300 import fftpl as F
    inst = instance(m_fix, 64, m_fix)
    q = oracle.overlap_map_q(inst.region, inst.n, inst.fix_x, inst.fix_y, inst.w[1:], inst.h[1:])
    q += oracle.overlap_map_q(inst.region, inst.n, inst.x, inst.y, inst.w[:1], inst.h[:1])
    with F.Problem(inst, deterministic=1) as p:
        F.fftpl_density(p.h, torch.from_numpy(inst.x).cuda(), torch.from_numpy(inst.y).cuda())
        got = F.fftpl_fields(p.h, p.n)["rho"].cpu().numpy()
    # units of 2^-32, exactly summed, to float32 and over A_b = 4
    assert np.array_equal(got, q.astype(np.float32) * np.float32(2.0 ** -34))
