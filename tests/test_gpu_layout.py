"""The order of cells and nets that creation sorts on the device, exactly, against
a stable sort on the host: cells by (label, distance, index), nets by (degree
descending, lowest cell number, index); sizes around the sort's tiles (2048
keys) and above 65,536 key values (three passes of eight bits).  Handles made
again get the same layout."""
import types

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

INF = 0x7FFFFFFF
SEED_STRIDE, ROUNDS, MAX_DEGREE = 64, 6, 64   # of the label rounds
BIG_MIN, BIG_MAX = 7, 64                      # degrees with several lanes per net


def instance(m, E, seed):
    rng = np.random.default_rng(seed)
    deg = np.where(rng.random(E) < 0.9, rng.integers(0, 4, E), rng.integers(4, 71, E))
    deg[0] = 2
    P, nf = int(deg.sum()), 3
    # most nets local, so that labels travel; a part of the cells unreached
    first = np.repeat(rng.integers(0, m, E), deg)
    pc = np.minimum(first + rng.integers(0, 40, P), m + nf - 1)
    pc[rng.random(P) < 0.02] = m
    return types.SimpleNamespace(
        region=(0.0, 0.0, 128.0, 128.0), n=64, target_density=1.0, m_mov=m, m_fix=nf,
        w=np.full(m + nf, 1.5, np.float32), h=np.ones(m + nf, np.float32),
        fix_x=np.full(nf, 9, np.float32), fix_y=np.full(nf, 9, np.float32),
        net_ptr=np.concatenate([[0], np.cumsum(deg)]).astype(np.int32),
        pin_cell=pc.astype(np.int32), pin_dx=np.zeros(P, np.float32),
        pin_dy=np.zeros(P, np.float32))


def lanes(d):
    if not BIG_MIN <= d <= BIG_MAX:
        return 1
    return 2 if d <= 8 else 4 if d <= 16 else 8 if d <= 32 else 16


def expected(inst):
    m, ptr, pc = inst.m_mov, inst.net_ptr, inst.pin_cell
    E = ptr.size - 1
    deg = np.diff(ptr)
    net = np.repeat(np.arange(E), deg)
    mov = pc < m
    lab = np.where(np.arange(m) % SEED_STRIDE == 0, np.arange(m), INF)
    dist = np.where(lab < INF, 0, INF)
    use = mov & ((deg >= 2) & (deg <= MAX_DEGREE))[net]
    for r in range(ROUNDS):
        nl = np.full(E, INF)
        np.minimum.at(nl, net[use], lab[pc[use]])
        new = lab.copy()
        np.minimum.at(new, pc[use], nl[net[use]])
        dist[new < lab] = r + 1
        lab = new
    order = np.lexsort((np.arange(m), dist, lab))
    rank = np.empty(m, np.int32)
    rank[order] = np.arange(m)
    key = np.full(E, m)
    np.minimum.at(key, net[mov], rank[pc[mov]])
    slot, pins = 0, []
    for d in range(int(deg.max()), 1, -1):
        nets = np.flatnonzero(deg == d)
        nets = nets[np.argsort(key[nets], kind="stable")]
        L = lanes(d)
        G, rows = 32 // L, -(-d // L)
        slabs = -(-nets.size // G)
        block = np.full(slabs * rows * 32, -1, np.int32)
        j, k = np.meshgrid(np.arange(nets.size), np.arange(d), indexing="ij")
        c = pc[ptr[nets][:, None] + np.arange(d)]
        at = (j // G) * 32 * rows + (j % G) * L + 32 * (k // L) + k % L
        block[at] = np.where(c < m, rank[np.minimum(c, m - 1)], -1)
        pins.append(block)
    return rank, np.concatenate(pins)


@pytest.mark.parametrize("m,E", [(1, 1), (255, 300), (2047, 2049), (2049, 2047), (6001, 6145),
                                 (70001, 40000), (30000, 140000)])
def test_layout(m, E):
    from paper_1312_4587_gb300 import fftpl as F
    inst = instance(m, E, m + E)
    rank, pins = expected(inst)
    for _ in range(3):
        with F.Problem(inst) as p:
            got_rank, got_pins = F.fftpl_debug_layout(p.h, m)
        assert np.array_equal(got_rank, rank)
        assert np.array_equal(got_pins, pins)
