"""What a user of this framework has it do, as cases that can be timed.

A case is one call (or one short run of calls) through the public Python
binding on a seeded synthetic placement instance whose distributions are those
of the repository's own generator: cells one row high with lognormal widths,
60 % two-pin nets, 25 % of degree 3-4, 15 % of degree 5-50, nets local in a
random cell permutation, macros over 12 % of the region.  `spread` says where
a placement run stands: "start" is the Gaussian cluster every run begins
from, "late" the nearly uniform spread of its last iterations, where nets are
short and neighbours in the netlist lie close together.
"""
import math
import types

import numpy as np
import torch

from paper_1312_4587_gb300 import autograd, serve
from paper_1312_4587_gb300 import fftpl as F

REPORT = ("N", "W", "hpwl", "tau", "gN_l1", "gW_l1", "charge", "mov_area")
PINS_PER_NET = 3.545    # mean degree of the net distribution


def _case(name, kind, m, n, wb, nets=1.05, macros=0, rho=0.9, spread="start", **more):
    return dict(name=name, kind=kind, m=m, n=n, wb=wb, nets=int(round(nets * m)), macros=macros,
                rho=rho, spread=spread, **more)


def listed():
    return [
        # The smallest instance of the repository: a user's own optimiser on a
        # block of 1,000 cells reads f and its gradient; latency is all.
        _case("eval_tiny", "eval", 1000, 64, 2.0, 1.2, 0, 1.0, graphs=1),
        # A small block with ragged sizes and the default options (no graph),
        # late in its run.
        _case("eval_medium", "eval", 6001, 128, 1.5, 1.05, 5, spread="late"),
        # Reproducible runs with the model variants: deterministic mode,
        # log-sum-exp wirelength, Helmholtz smoothing.
        _case("eval_sub_variants", "eval", 34375, 256, 1.5, 1.045, 3, spread="late",
              graphs=1, det=1, lse=1, eps_modes=2.0),
        # An ADAPTEC1-sized circuit in the middle of its run.
        _case("eval_large", "eval", 210000, 512, 2.0, 1.0476, 40, spread="late", graphs=1),
        # The headline: a BIGBLUE4-sized circuit at the start of its run.
        _case("eval_precision", "eval", 2200000, 2048, 1.5, 1.04545, 150, graphs=1),
        # The same evaluation for a placer whose data live in pinned host memory.
        _case("host_precision", "eval_host", 2200000, 2048, 1.5, 1.04545, 150,
              spread="late", graphs=1),
        # The density energy as a torch loss term: forward and backward.
        _case("autograd_diff", "autograd", 500000, 1024, 1.5, 1.048, 0, 1.0, mode="gather"),
        # The largest grid, for a caller that brings its own wirelength term.
        _case("density_max", "density", 5000000, 4096, 1.5, 0.0, 200, spread="late"),
        # The solve on its own, on a caller's density map.
        _case("solve_map", "solve", 0, 512, 2.0),
        # A placement run's first iterations (Nesterov) at ADAPTEC1 size.
        _case("place_large", "place", 210000, 512, 2.0, 1.0476, 40, graphs=1, iters=12),
        # The tensor-core solve path at the headline's grid.
        _case("density_tc", "density", 1100000, 2048, 1.5, 0.0, 75, path="tc"),
        # Jobs that arrive together at the placement server.
        _case("serve_mix", "serve", 40000, 0, 0.0, macros=4, spread="start", jobs=12,
              iters=10),
    ]


def _grid(m, macro_frac, rng=None):
    """Bins per side 2^ceil(log2 sqrt m) and the bin width (a multiple of 0.5)
    that keeps the movable area at or below 70 % of the free area."""
    n = min(4096, 1 << max(4, math.ceil(math.log2(math.sqrt(m)))))
    if rng is not None and n < 2048 and rng.random() < 0.25:
        n *= 2
    wb = 0.5
    while m * 2.4 > 0.7 * (wb * n) ** 2 * (1.0 - macro_frac):
        wb += 0.5
    return n, wb


def draw(rng):
    """One more case: any entry point, cell counts log-uniform over its range."""
    kind = rng.choices(("eval", "density", "autograd", "wa", "place", "eval_host", "solve",
                        "tc", "serve"), (40, 10, 10, 10, 12, 5, 5, 4, 4))[0]
    if kind == "solve":
        return {"kind": "solve", "m": 0, "n": 2 ** rng.randint(5, 10), "nets": 0, "macros": 0,
                "wb": rng.choice((1.0, 1.5, 2.0)), "rho": 1.0,
                "spread": rng.choice(("start", "late"))}
    lo, hi = {"place": (1000, 220000), "serve": (5000, 60000), "tc": (20000, 1000000)}.get(
        kind, (1000, 2000000))
    m = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    macros = rng.choice((0, max(1, m // 5500)))
    macros = min(macros, 150)
    n, wb = _grid(m, 0.12, rng)
    c = dict(kind=kind, m=m, n=n, wb=wb, nets=int(m * rng.uniform(0.9, 1.2)), macros=macros,
             rho=rng.choice((0.9, 1.0)), spread=rng.choice(("start", "late")))
    if kind in ("eval", "place", "wa"):
        c["graphs"] = rng.choice((0, 1, 1))
        c["lse"] = 1 if rng.random() < 0.2 else 0
        c["det"] = 1 if rng.random() < 0.2 else 0
        c["eps_modes"] = 2.0 if rng.random() < 0.15 else 0.0
    if kind == "autograd":
        c["mode"] = rng.choice(("gather", "gather", "adjoint"))
    if kind == "density":
        c["det"] = 1 if rng.random() < 0.2 else 0
    if kind == "place":
        c["iters"] = rng.randint(4, 12)
        c["cg"] = 1 if rng.random() < 0.3 else 0
    if kind == "tc":
        c["kind"] = "density"
        c["path"] = rng.choice(("tc", "tc", "radix"))
        c["n"] = max(256, n)
        c["wb"] = wb * n / c["n"]
    if kind == "serve":
        c.update(n=0, wb=0.0, jobs=rng.randint(3, 10), iters=rng.randint(4, 10))
    return c


# ------------------------------------------------------------------ inputs

def _macros(rs, L, k):
    """k rectangles with integer corners in slots of their own over 12 % of R."""
    if k == 0:
        z = np.zeros(0, np.float32)
        return z, z, z, z
    g = math.ceil(math.sqrt(2 * k))
    slot = rs.permutation(g * g)[:k]
    asp = np.exp(rs.uniform(math.log(0.5), math.log(2.0), k))
    area = 0.12 * L * L / k
    w = np.clip(np.rint(np.sqrt(area * asp)), 1, L / g - 1)
    h = np.clip(np.rint(area / w), 1, L / g - 1)
    lx = np.floor(slot % g * (L / g) + rs.uniform(0, 1, k) * (L / g - w))
    ly = np.floor(slot // g * (L / g) + rs.uniform(0, 1, k) * (L / g - h))
    return tuple(a.astype(np.float32) for a in (lx + 0.5 * w, ly + 0.5 * h, w, h))


def _rand(gen, size):
    return torch.rand(size, generator=gen, device="cuda", dtype=torch.float64)


def _instance(m, n, wb, nets, macros, rho, spread, seed):
    """A seeded instance with the fields fftpl.Problem takes (host arrays)
    and start positions x, y (CUDA tensors)."""
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    rs = np.random.RandomState(int(seed) % (1 << 31))
    L = wb * n
    w = torch.randn(m, generator=gen, device="cuda", dtype=torch.float64) * 0.6 + math.log(2.0)
    w = torch.exp(w).round().clamp(1, min(40.0, L / 4)).float()
    h = torch.ones(m, device="cuda")
    fx, fy, fw, fh = _macros(rs, L, macros)
    perm = torch.randperm(m, generator=gen, device="cuda")
    # nets: degree, then pins at distinct offsets around an anchor in perm
    u = _rand(gen, nets)
    ds = torch.arange(5, 51, device="cuda", dtype=torch.float64)
    cdf = torch.cumsum(ds ** -2.5, 0)
    big = 5 + torch.searchsorted(cdf / cdf[-1], _rand(gen, nets)).clamp(max=45)
    mid = 3 + (_rand(gen, nets) < 0.5).long()
    deg = torch.where(u < 0.6, torch.full_like(mid, 2), torch.where(u < 0.85, mid, big))
    ptr = torch.zeros(nets + 1, dtype=torch.int64, device="cuda")
    ptr[1:] = torch.cumsum(deg, 0)
    P = int(ptr[-1])
    net = torch.repeat_interleave(torch.arange(nets, device="cuda"), deg)
    dn = deg[net]
    gap = 1 + (_rand(gen, P) * (128 // dn).double()).long()
    run = torch.cumsum(gap, 0)
    first = run[ptr[:-1]] if nets else run
    off = run - first[net]
    span = off[ptr[1:] - 1] if nets else off
    anchor = (_rand(gen, nets) * m).long()
    cell = perm[(anchor[net] + off - span[net] // 2) % m] if P else net
    dx = ((_rand(gen, P) - 0.5) * w[cell]).float()
    dy = ((_rand(gen, P) - 0.5) * h[cell]).float()
    if macros and nets:
        # about 1 % of the nets end on a macro pin
        sel = torch.nonzero(_rand(gen, nets) < 0.01).squeeze(1)
        last = ptr[sel + 1] - 1
        k = (_rand(gen, sel.numel()) * macros).long()
        cell[last] = m + k
        dx[last] = ((_rand(gen, sel.numel()) - 0.5) * torch.from_numpy(fw).cuda()[k]).float()
        dy[last] = ((_rand(gen, sel.numel()) - 0.5) * torch.from_numpy(fh).cuda()[k]).float()
    if spread == "start":
        x = torch.randn(m, generator=gen, device="cuda", dtype=torch.float64) * 0.1 * L + 0.5 * L
        y = torch.randn(m, generator=gen, device="cuda", dtype=torch.float64) * 0.1 * L + 0.5 * L
    else:
        # 64 cells that are neighbours in the netlist share a square tile
        side = math.ceil(math.sqrt(max(1, math.ceil(m / 64))))
        t = torch.empty(m, dtype=torch.int64, device="cuda")
        t[perm] = torch.arange(m, device="cuda") // 64
        row = t // side
        col = torch.where(row % 2 == 0, t % side, side - 1 - t % side)
        x = (col + _rand(gen, m)) * (L / side)
        y = (row + _rand(gen, m)) * (L / side)
    x = torch.minimum(torch.maximum(x.float(), 0.5 * w), L - 0.5 * w)
    y = torch.minimum(torch.maximum(y.float(), 0.5 * h), L - 0.5 * h)
    return types.SimpleNamespace(
        region=(0.0, 0.0, L, L), n=n, target_density=rho, gamma=0.5 * wb, m_mov=m,
        m_fix=macros, w=np.concatenate([w.cpu().numpy(), fw]),
        h=np.concatenate([h.cpu().numpy(), fh]), fix_x=fx, fix_y=fy,
        net_ptr=ptr.to(torch.int32).cpu().numpy(), pin_cell=cell.to(torch.int32).cpu().numpy(),
        pin_dx=dx.cpu().numpy(), pin_dy=dy.cpu().numpy(), x=x, y=y)


def _of(case, seed):
    return _instance(case["m"], case["n"], case["wb"], case["nets"], case["macros"], case["rho"],
                     case["spread"], seed)


def _options(case):
    """Handle options; eps_modes: the Helmholtz eps as a multiple of the
    lowest mode's (pi / L)^2."""
    o = dict(use_graphs=case.get("graphs", 0), deterministic=case.get("det", 0),
             wirelength=F.FFTPL_WL_LSE if case.get("lse") else F.FFTPL_WL_WA,
             optimizer=F.FFTPL_OPT_CG if case.get("cg") else F.FFTPL_OPT_NESTEROV)
    o["helmholtz_eps"] = _eps(case)
    o["solve_path"] = {"tc": F.FFTPL_SOLVE_TC_BF16X3, "radix": F.FFTPL_SOLVE_TC_RADIX}.get(
        case.get("path"), F.FFTPL_SOLVE_FFT)
    return o


def _dw_ref(m):
    """Small circuits scale the paper's reference HPWL change."""
    return 3.5e5 * min(1.0, m / 210000)


def _eps(case):
    k = case.get("eps_modes", 0.0)
    return float(k * (math.pi / (case["wb"] * case["n"])) ** 2) if k else 0.0


def _jobs(case, seed):
    """The jobs of one serving pass: cell counts spread over 1/8 .. 2 times m."""
    rs = np.random.RandomState(int(seed) % (1 << 31))
    jobs = []
    for k in range(case["jobs"]):
        m = int(case["m"] * 2.0 ** (-3.0 + 4.0 * (k + 0.5) / case["jobs"]))
        n, wb = _grid(m, 0.12)
        j = _instance(m, n, wb, int(1.05 * m), max(1, m // 5500) if case["macros"] else 0,
                      case["rho"], case["spread"], int(rs.randint(1 << 30)))
        j.x, j.y = j.x.cpu().numpy(), j.y.cpu().numpy()
        jobs.append(j)
    return jobs


def _density_map(case, seed):
    """A density map: a spread-out cluster plus the noise of single cells."""
    n = case["n"]
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    k = torch.linspace(-1, 1, n, device="cuda")
    s = 0.1 if case["spread"] == "start" else 2.0
    blob = torch.exp(-(k[:, None] ** 2 + k[None, :] ** 2) / s)
    return (blob * 2.0 * torch.rand((n, n), generator=gen, device="cuda")).contiguous()


def prepare(case, seed):
    kind = case["kind"]
    s = types.SimpleNamespace(case=case, kind=kind)
    if kind == "serve":
        s.jobs = _jobs(case, seed)
        return s
    if kind == "solve":
        s.rho, s.n, s.L = _density_map(case, seed), case["n"], case["wb"] * case["n"]
        s.out = [torch.empty_like(s.rho) for _ in range(3)]
        return s
    inst = _of(case, seed)
    s.gamma, s.x, s.y = inst.gamma, inst.x, inst.y
    if kind == "eval_host":
        s.x, s.y = s.x.cpu().pin_memory(), s.y.cpu().pin_memory()
        s.g = [torch.empty(case["m"], pin_memory=True) for _ in range(4)]
    else:
        s.g = [torch.empty_like(s.x) for _ in range(4)]
    if kind == "place":
        s.prob = F.Problem(inst, dw_ref=_dw_ref(case["m"]), **_options(case))
    else:
        s.prob = F.Problem(inst, **_options(case))
    if kind == "autograd":
        s.x.requires_grad_(True)
        s.y.requires_grad_(True)
    return s


def _scalars(rep):
    return {k: np.float32(rep[k]) for k in REPORT}


def run(s):
    kind = s.kind
    if kind in ("eval", "eval_host"):
        call = F.fftpl_eval if kind == "eval" else F.fftpl_eval_host
        rep = call(s.prob.h, s.x, s.y, s.gamma, *s.g)
        return {"gNx": s.g[0], "gNy": s.g[1], "gWx": s.g[2], "gWy": s.g[3], **_scalars(rep)}
    if kind == "density":
        N = F.fftpl_density(s.prob.h, s.x, s.y, s.g[0], s.g[1])
        return {"gNx": s.g[0], "gNy": s.g[1], "N": np.float32(N)}
    if kind == "wa":
        W = F.fftpl_wa(s.prob.h, s.x, s.y, s.gamma, s.g[2], s.g[3])
        return {"gWx": s.g[2], "gWy": s.g[3], "W": np.float32(W)}
    if kind == "autograd":
        s.x.grad = s.y.grad = None
        loss = autograd.density_energy(s.x, s.y, s.prob, s.case["mode"]).float()
        loss.backward()
        return {"gNx": s.x.grad, "gNy": s.y.grad, "N": loss.detach()}
    if kind == "solve":
        F.fftpl_solve_noalloc(s.rho, s.n, s.L, s.L, *s.out)
        return {"psi": s.out[0], "ex": s.out[1], "ey": s.out[2]}
    if kind == "place":
        F.fftpl_place_init(s.prob.h, s.x, s.y)
        rows, ran = F.fftpl_step(s.prob.h, s.case["iters"])
        F.fftpl_place_positions(s.prob.h, s.g[0], s.g[1])
        rec = np.array([[r["hpwl"], r["N"], r["tau"]] for r in rows], np.float32)
        return {"x": s.g[0], "y": s.g[1], "hpwl": rec[:, 0], "N": rec[:, 1], "tau": rec[:, 2],
                "ran": ran}
    with serve.Server(max_active=8, iters_per_tick=5) as srv:
        ids = [srv.submit(j, s.case["iters"], dw_ref=_dw_ref(j.m_mov)) for j in s.jobs]
        srv.drain()
        out = {}
        for k, i in enumerate(ids):
            _, out["x%d" % k], out["y%d" % k] = srv.job(i)
    return out


# -------------------------------------------------------------------- work

def _transforms(n):
    """Four real two-dimensional transforms of n x n."""
    return 4 * 2.5 * n * n * 2 * math.log2(n)


def work(case):
    kind, m, n = case["kind"], case["m"], case["n"]
    P = PINS_PER_NET * case["nets"]
    if kind == "serve":
        tot = {"bytes": 0.0, "flops": 0.0}
        for k in range(case["jobs"]):
            jm = int(case["m"] * 2.0 ** (-3.0 + 4.0 * (k + 0.5) / case["jobs"]))
            jn, jwb = _grid(jm, 0.12)
            w = work(dict(case, kind="place", m=jm, n=jn, wb=jwb, nets=int(1.05 * jm)))
            tot = {q: tot[q] + w[q] for q in tot}
        return tot
    if kind == "solve":
        return {"bytes": 16.0 * n * n, "flops": _transforms(n)}
    dens = {"bytes": 24.0 * m + 4.0 * n * n, "flops": _transforms(n) + 60.0 * m}
    wl = {"bytes": 12.0 * P + 4.0 * case["nets"] + 16.0 * m, "flops": 60.0 * P}
    if kind in ("density", "autograd"):
        return dens
    if kind == "wa":
        return wl
    # positions are read once for both terms
    both = {"bytes": dens["bytes"] + wl["bytes"] - 8.0 * m, "flops": dens["flops"] + wl["flops"]}
    if kind == "place":
        # the loop keeps five vectors of 2 m between iterations
        evals = case["iters"] * (2 if case.get("cg") else 1)
        return {"bytes": evals * (both["bytes"] + 40.0 * m), "flops": evals * both["flops"]}
    return both


# ---------------------------------------------------- the same in 64 bits

def _axis_overlap(lo, hi, n, wb):
    """[k][n] overlap lengths of the intervals [lo, hi] with the bins."""
    e = torch.arange(n + 1, device="cuda", dtype=torch.float64) * wb
    a = torch.maximum(lo[:, None], e[None, :-1])
    b = torch.minimum(hi[:, None], e[None, 1:])
    return (b - a).clamp(min=0)


def _pairs(x, y, w, h, n, wb):
    """For every offset (dj, di) inside the largest span: flat bin numbers and
    overlap areas of all cells.  Edges are float32, as the library defines them."""
    xl, xh = (x - 0.5 * w).double(), (x + 0.5 * w).double()
    yl, yh = (y - 0.5 * h).double(), (y + 0.5 * h).double()
    i0 = torch.floor(xl / wb).long().clamp(0, n - 1)
    j0 = torch.floor(yl / wb).long().clamp(0, n - 1)
    ni = int((torch.floor(xh / wb).long().clamp(0, n - 1) - i0).max()) + 1
    nj = int((torch.floor(yh / wb).long().clamp(0, n - 1) - j0).max()) + 1
    for dj in range(nj):
        j = (j0 + dj).clamp(max=n - 1)
        oy = (torch.minimum(yh, (j + 1) * wb) - torch.maximum(yl, j * wb)).clamp(min=0)
        oy = torch.where(j0 + dj < n, oy, torch.zeros_like(oy))
        for di in range(ni):
            i = (i0 + di).clamp(max=n - 1)
            ox = (torch.minimum(xh, (i + 1) * wb) - torch.maximum(xl, i * wb)).clamp(min=0)
            ox = torch.where(i0 + di < n, ox, torch.zeros_like(ox))
            yield j * n + i, ox * oy


def _dct(a):
    """sum_x a[.., x] cos(pi u (2x+1) / 2n) for all u."""
    n = a.shape[-1]
    z = torch.fft.fft(a.to(torch.complex128), n=2 * n)[..., :n]
    return (z * _phase(n).conj()).real


def _phase(n):
    t = torch.arange(n, device="cuda", dtype=torch.float64) * (math.pi / (2 * n))
    return torch.complex(torch.cos(t), torch.sin(t))


def _sums(c):
    """(sum_u c[.., u] cos(pi u (2x+1) / 2n), the same with sin) for all x."""
    n = c.shape[-1]
    z = torch.fft.ifft(c * _phase(n), n=2 * n)[..., :n] * (2 * n)
    return z.real, z.imag


def _solve64(rho, L, eps):
    """psi, E_x, E_y of a density map by the cosine series."""
    n = rho.shape[0]
    a = _dct(_dct(rho).T.contiguous()).T / (n * n)
    a[1:, :] *= 2
    a[:, 1:] *= 2
    wv = torch.arange(n, device="cuda", dtype=torch.float64) * (math.pi / L)
    d = wv[:, None] ** 2 + wv[None, :] ** 2 + eps
    if eps == 0.0:
        d[0, 0] = 1.0
        a[0, 0] = 0.0
    c = a / d
    p, _ = _sums(c.T.contiguous())                       # along y: [u][y]
    _, r = _sums((c * wv[:, None]).T.contiguous())
    p, r = p.T.contiguous(), r.T.contiguous()
    return _sums(p)[0], _sums(p * wv[None, :])[1], _sums(r)[0]


def _density64(case, inst, adjoint=False):
    m, n, wb = inst.m_mov, inst.n, case["wb"]
    x, y = inst.x, inst.y
    w, h = (torch.from_numpy(a[:m]).cuda() for a in (inst.w, inst.h))
    D = torch.zeros(n * n, device="cuda", dtype=torch.float64)
    for b, ov in _pairs(x, y, w, h, n, wb):
        D.index_add_(0, b, ov)
    D = D.view(n, n)
    Fx = torch.zeros_like(D)
    if inst.m_fix:
        fx, fy = torch.from_numpy(inst.fix_x).cuda(), torch.from_numpy(inst.fix_y).cuda()
        fw, fh = (torch.from_numpy(a[m:]).cuda() for a in (inst.w, inst.h))
        Fx = _axis_overlap((fy - 0.5 * fh).double(), (fy + 0.5 * fh).double(), n, wb).T @ \
            _axis_overlap((fx - 0.5 * fw).double(), (fx + 0.5 * fw).double(), n, wb)
    A = wb * wb
    rho = (D + case["rho"] * Fx) / A
    psi, ex, ey = _solve64(rho, wb * n, _eps(case))
    area = float((w.double() * h.double()).sum())
    out = {"N": 0.5 * A * float((rho * psi).sum()), "charge": float(rho.sum()) * A,
           "tau": float((D - case["rho"] * (A - Fx)).clamp(min=0).sum()) / area,
           "mov_area": area}
    if adjoint:
        gx, gy = _adjoint64(psi, x, y, w, h, n, wb)
    else:
        gx, gy = torch.zeros_like(x).double(), torch.zeros_like(y).double()
        for b, ov in _pairs(x, y, w, h, n, wb):
            gx -= ov * ex.reshape(-1)[b]
            gy -= ov * ey.reshape(-1)[b]
    out.update(gNx=gx, gNy=gy, gN_l1=float(gx.abs().sum() + gy.abs().sum()))
    return out


def _adjoint64(psi, x, y, w, h, n, wb):
    """The exact derivative of the binned energy: psi at the bin of the upper
    edge less psi at the bin of the lower edge, times the other axis' overlap."""
    res = []
    for a, aw, b, bw, at in ((x, w, y, h, lambda k, j: psi[j, k]),
                             (y, h, x, w, lambda k, j: psi[k, j])):
        lo, hi = (a - 0.5 * aw).double(), (a + 0.5 * aw).double()
        bl, bh = (b - 0.5 * bw).double(), (b + 0.5 * bw).double()
        kl, kh = torch.floor(lo / wb).long(), torch.floor(hi / wb).long()
        j0 = torch.floor(bl / wb).long().clamp(0, n - 1)
        span = int((torch.floor(bh / wb).long().clamp(0, n - 1) - j0).max()) + 1
        g = torch.zeros_like(lo)
        for dj in range(span):
            j = (j0 + dj).clamp(max=n - 1)
            ov = (torch.minimum(bh, (j + 1) * wb) - torch.maximum(bl, j * wb)).clamp(min=0)
            ov = torch.where(j0 + dj < n, ov, torch.zeros_like(ov))
            up = torch.where((kh >= 0) & (kh < n), at(kh.clamp(0, n - 1), j), 0.0)
            dn = torch.where((kl >= 0) & (kl < n), at(kl.clamp(0, n - 1), j), 0.0)
            g += ov * (up - dn)
        res.append(g)
    return res


def _wire64(case, inst):
    m = inst.m_mov
    g = float(np.float32(inst.gamma))
    ptr = torch.from_numpy(inst.net_ptr).cuda().long()
    deg = ptr[1:] - ptr[:-1]
    E = deg.numel()
    net = torch.repeat_interleave(torch.arange(E, device="cuda"), deg)
    cell = torch.from_numpy(inst.pin_cell).cuda().long()
    out, W, hp, l1 = {}, 0.0, 0.0, 0.0
    for key, pos, fix, off in (("gWx", inst.x, inst.fix_x, inst.pin_dx),
                               ("gWy", inst.y, inst.fix_y, inst.pin_dy)):
        c = torch.cat([pos, torch.from_numpy(fix).cuda()])
        p = (c[cell] + torch.from_numpy(off).cuda()).double()    # fl32(centre + offset)
        M = torch.full((E,), -math.inf, device="cuda", dtype=torch.float64)
        M = M.scatter_reduce(0, net, p, "amax")
        mu = torch.full((E,), math.inf, device="cuda", dtype=torch.float64)
        mu = mu.scatter_reduce(0, net, p, "amin")
        tp, tm = p - M[net], p - mu[net]
        ap, am = torch.exp(tp / g), torch.exp(-tm / g)

        def seg(v):
            return torch.zeros(E, device="cuda", dtype=torch.float64).index_add_(0, net, v)
        Sp, Sm = seg(ap), seg(am)
        hp += float((M - mu).sum())
        if case.get("lse"):
            W += float((M - mu).sum() + g * (torch.log(Sp) + torch.log(Sm)).sum())
            gp = ap / Sp[net] - am / Sm[net]
        else:
            Tp, Tm = seg(tp * ap) / Sp, seg(tm * am) / Sm
            W += float((M - mu + Tp - Tm).sum())
            gp = ap / Sp[net] * (1 + (tp - Tp[net]) / g) - am / Sm[net] * (1 - (tm - Tm[net]) / g)
        mov = cell < m
        out[key] = torch.zeros(m, device="cuda", dtype=torch.float64).index_add_(
            0, cell[mov], gp[mov])
        l1 += float(out[key].abs().sum())
    out.update(W=W, hpwl=hp, gW_l1=l1)
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind in ("place", "serve"):
        return None     # a loop of many steps: rounding travels through all of them
    if kind == "solve":
        psi, ex, ey = _solve64(_density_map(case, seed).double(), case["wb"] * case["n"], 0.0)
        return {"psi": psi, "ex": ex, "ey": ey}
    inst = _of(case, seed)
    if kind == "wa":
        o = _wire64(case, inst)
        return {k: o[k] for k in ("gWx", "gWy", "W")}
    o = _density64(case, inst, case.get("mode") == "adjoint")
    if kind in ("density", "autograd"):
        return {k: o[k] for k in ("gNx", "gNy", "N")}
    o.update(_wire64(case, inst))
    return {k: o[k] for k in ("gNx", "gNy", "gWx", "gWy") + REPORT}
