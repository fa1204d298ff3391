"""What a handle lays out at creation, against the oracle: the order of cells
and nets at the edges of the sort's tiles (2048 keys, 256 a warp), and the map
of the fixed cells.  W within 1e-6 and grad W within 1e-5 (float32 terms, FP64
sums); the density within 1e-6 (float32 overlap areas)."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def F():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_1312_4587_gb300 import fftpl
    fftpl.lib()
    return fftpl


def rel(a, b):
    a = np.asarray(a, np.float64).ravel(); b = np.asarray(b, np.float64).ravel()
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


def run(F, inst, **opts):
    import torch
    xy = [torch.from_numpy(np.ascontiguousarray(v, np.float32)).cuda() for v in (inst.x, inst.y)]
    with F.Problem(inst, **opts) as p:
        g = [torch.empty_like(xy[0]) for _ in range(4)]
        rep = F.fftpl_eval(p.h, *xy, inst.gamma, *g)
        rho = F.fftpl_fields(p.h, inst.n)["rho"].cpu().numpy()
    return rep, [v.cpu().numpy() for v in g], rho


@pytest.mark.parametrize("det", [0, 1])
@pytest.mark.parametrize("m,E", [(1, 1), (33, 255), (2047, 257), (2048, 2049), (2049, 2047),
                                 (300, 70000)])
def test_net_order(F, m, E, det):
    """Degrees 0 (an empty net) to 70, most of them 2 or 3; far more cells
    than the nets reach, or far fewer."""
    rng = np.random.default_rng(m + E)
    base = synth.make_instance("tiny")
    L = base.region[2]
    deg = np.where(rng.random(E) < 0.9, rng.integers(0, 4, E), rng.integers(4, 71, E))
    deg[0] = 2
    P = int(deg.sum())
    nf = 3
    inst = synth.Instance(
        name="order", region=base.region, n=base.n, target_density=1.0, gamma=base.gamma,
        m_mov=m, m_fix=nf, w=np.full(m + nf, 1.5, np.float32), h=np.full(m + nf, 1.0, np.float32),
        fix_x=rng.uniform(0, L, nf).astype(np.float32),
        fix_y=rng.uniform(0, L, nf).astype(np.float32),
        net_ptr=np.concatenate([[0], np.cumsum(deg)]).astype(np.int32),
        pin_cell=rng.integers(0, m + nf, P).astype(np.int32),
        pin_dx=rng.uniform(-0.4, 0.4, P).astype(np.float32),
        pin_dy=rng.uniform(-0.4, 0.4, P).astype(np.float32),
        x=rng.uniform(0, L, m).astype(np.float32), y=rng.uniform(0, L, m).astype(np.float32))
    ref = oracle.wa(inst.net_ptr, inst.pin_cell, inst.pin_dx, inst.pin_dy, m, inst.x, inst.y,
                    inst.gamma, inst.fix_x, inst.fix_y)
    rep, g, _ = run(F, inst, deterministic=det)
    assert abs(rep["W"] - ref["W"]) <= 1e-6 * abs(ref["W"])
    assert abs(rep["hpwl"] - ref["hpwl"]) <= 1e-6 * abs(ref["hpwl"])
    want = np.concatenate([ref["gcx"], ref["gcy"]])
    if np.any(want):
        assert rel(np.concatenate(g[2:]), want) < 1e-5


@pytest.mark.parametrize("det", [0, 1])
@pytest.mark.parametrize("place", ["bin", "edge", "outside", "whole", "overlapping"])
def test_fixed_map(F, place, det):
    base = synth.make_instance("tiny")
    L, wb = base.region[2], base.region[2] / base.n
    x, y, w, h = {
        "bin": ([2.5 * wb], [3.5 * wb], [wb], [wb]),
        "edge": ([0.0, L], [L / 3, L], [7.3 * wb, 2.2 * wb], [0.4 * wb, 3.1 * wb]),
        "outside": ([-5 * wb, L + 9 * wb], [L / 2, L / 2], [2 * wb, wb], [wb, wb]),
        "whole": ([L / 2], [L / 2], [1.5 * L], [2.0 * L]),
        "overlapping": ([L / 2, L / 2 + 3.3 * wb], [L / 2, L / 2], [21.7 * wb, 8 * wb],
                        [11.1 * wb, 30.2 * wb]),
    }[place]
    f32 = lambda v: np.asarray(v, np.float32)
    d = dict(base.__dict__)
    m = base.m_mov
    d.update(m_fix=len(x), fix_x=f32(x), fix_y=f32(y), target_density=0.8,
             w=np.concatenate([base.w[:m], f32(w)]), h=np.concatenate([base.h[:m], f32(h)]))
    inst = synth.Instance(**d)
    want, _, _ = oracle.density(inst.region, inst.n, 0.8, inst.x, inst.y, inst.w[:m], inst.h[:m],
                                inst.fix_x, inst.fix_y, inst.w[m:], inst.h[m:])
    _, _, rho = run(F, inst, deterministic=det)
    assert rel(rho, want) < 1e-6
