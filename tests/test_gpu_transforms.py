"""The transform passes at every grid size they are built for, in FP64: up to
n = 1024 a random map on a region with different side lengths against the
oracle's explicit sums, at 2048 and 4096 the density map of a placement
against FP64 cosine and sine transforms.

Bound: four one-dimensional passes of log2 n butterfly levels, each rounding
with a relative root-mean-square error of at most 2^-24, add up in quadrature
to sqrt(4 log2 n) 2^-24; four times that covers the twiddles, the packing and
the divide."""
import math

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def F():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_1312_4587_gb300 import fftpl
    fftpl.lib()
    return fftpl


def bound(n):
    return 4.0 * math.sqrt(4.0 * math.log2(n)) * 2.0 ** -24


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a, np.float64) - b) / np.linalg.norm(b))


@pytest.mark.parametrize("n", [16, 32, 64, 128, 256, 512, 1024])
def test_solve_every_size(F, n):
    import torch
    rng = np.random.default_rng(n)
    rho = rng.uniform(0.0, 2.0, (n, n)).astype(np.float32)
    Lx, Ly = 3.0 * n, 2.0 * n
    out = [torch.empty(n, n, device="cuda") for _ in range(3)]
    N = F.fftpl_solve_noalloc(torch.from_numpy(rho).cuda(), n, Lx, Ly, *out, want_N=True)
    _, psi, ex, ey = oracle.solve(rho.astype(np.float64), Lx, Ly)
    for got, want, key in zip(out, (psi, ex, ey), ("psi", "ex", "ey")):
        assert rel(got.cpu().numpy(), want) < bound(n), key
    want = oracle.energy(rho, psi, (Lx / n) * (Ly / n))
    assert abs(N - want) < bound(n) * abs(want)


def solve_fft(rho, L):
    """psi, E_x, E_y of a square region's map by FP64 DCT / DST."""
    from scipy import fft
    n = rho.shape[0]
    a = fft.dctn(rho, type=2, workers=-1) / (4.0 * n * n)
    a[1:, :] *= 2
    a[:, 1:] *= 2
    w = np.pi * np.arange(n) / L
    d = w[:, None] ** 2 + w[None, :] ** 2
    d[0, 0] = 1.0
    a[0, 0] = 0.0
    a /= d

    def cos_sum(c, axis):
        c = np.moveaxis(c, axis, -1) * 0.5
        c[..., 0] *= 2
        return np.moveaxis(fft.dct(c, type=3, workers=-1), -1, axis)

    def sin_sum(c, axis):
        c = np.moveaxis(c, axis, -1) * (0.5 * w)
        c = np.concatenate([c[..., 1:], np.zeros_like(c[..., :1])], axis=-1)
        return np.moveaxis(fft.dst(c, type=3, workers=-1), -1, axis)

    p = cos_sum(a, 0)
    return cos_sum(p, 1), sin_sum(p, 1), cos_sum(sin_sum(a, 0), 1)


@pytest.mark.parametrize("n", [2048, 4096])
def test_density_solve_largest_sizes(F, n):
    import torch

    import synth
    base = synth.make_instance("medium")
    rng = np.random.default_rng(n)
    m = 60000
    L = float(n)
    w = rng.integers(1, 40, m).astype(np.float32)
    inst = synth.Instance(**dict(
        base.__dict__, n=n, region=(0.0, 0.0, L, L), m_mov=m, m_fix=0, w=w,
        h=np.ones(m, np.float32), fix_x=np.zeros(0, np.float32), fix_y=np.zeros(0, np.float32),
        net_ptr=np.zeros(1, np.int32), pin_cell=np.zeros(0, np.int32),
        pin_dx=np.zeros(0, np.float32), pin_dy=np.zeros(0, np.float32),
        x=rng.normal(0.5 * L, 0.1 * L, m).astype(np.float32),
        y=rng.normal(0.5 * L, 0.1 * L, m).astype(np.float32)))
    with F.Problem(inst) as p:
        F.fftpl_density(p.h, torch.from_numpy(inst.x).cuda(), torch.from_numpy(inst.y).cuda())
        f = {k: v.cpu().numpy() for k, v in F.fftpl_fields(p.h, n).items()}
        F.fftpl_check(p.h)
    want = solve_fft(f["rho"].astype(np.float64), L)
    for key, ref in zip(("psi", "ex", "ey"), want):
        assert rel(f[key], ref) < bound(n), key
