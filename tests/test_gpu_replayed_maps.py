"""Maps formed on demand after a caller's own graph has evaluated again: the
handle does not see a replay, so what it formed before must not be given out as
current."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def maps(F, p):
    return [t.clone() for t in F.fftpl_fields(p.h, p.n).values()]


@pytest.mark.parametrize("path", ["FFT", "TC_BF16X3", "TC_RADIX"])
def test_maps_after_a_replay(path):
    import torch
    from paper_1312_4587_gb300 import fftpl as F
    inst = synth.make_instance("precision_sub")
    rng = np.random.default_rng(3)
    opts = dict(deterministic=1, solve_path=getattr(F, "FFTPL_SOLVE_" + path))
    xs = [torch.from_numpy(inst.x).cuda(),
          torch.from_numpy(rng.permutation(inst.x)).cuda()]
    y = torch.from_numpy(inst.y).cuda()
    ref = []
    with F.Problem(inst, **opts) as p:
        for x in xs:
            F.fftpl_density(p.h, x, y, sync=False)
            g = [torch.empty_like(x) for _ in range(2)]
            F.fftpl_gather(p.h, x, y, *g, mode=1)
            ref.append(maps(F, p) + g)
        torch.cuda.synchronize()
    side = torch.cuda.Stream()
    x = xs[0].clone()
    torch.cuda.synchronize()
    with torch.cuda.stream(side):
        with F.Problem(inst, **opts) as p:
            F.fftpl_density(p.h, x, y, sync=False)
            maps(F, p)
            side.synchronize()
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=side):
                F.fftpl_density(p.h, x, y, sync=False)
            for k in (0, 1):
                x.copy_(xs[k])
                graph.replay()
                g = [torch.empty_like(x) for _ in range(2)]
                F.fftpl_gather(p.h, x, y, *g, mode=1)
                for got, want in zip(maps(F, p) + g, ref[k]):
                    assert torch.equal(got, want)
            side.synchronize()
