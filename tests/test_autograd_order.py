"""density_energy on a stream that is not the handle's: the order of the
handle's work and the caller's, with the library replaced by a record of its
calls (no GPU)."""
import types

import pytest
import torch

from paper_1312_4587_gb300 import autograd as A

HANDLE, CALLER = 7, 9


@pytest.fixture
def calls(monkeypatch):
    log = []

    def energy(h, x, y, sync=True):
        log.append("energy")
        return 2.0

    def gather(h, x, y, gx, gy, mode=0):
        log.append("gather")
        gx.copy_(x)
        gy.copy_(y)

    monkeypatch.setattr(A.F, "fftpl_energy", energy)
    monkeypatch.setattr(A.F, "fftpl_gather", gather)
    for name in ("fftpl_order_after", "fftpl_order_before"):
        monkeypatch.setattr(A.F, name, lambda h, s, name=name: log.append((name, s)),
                            raising=False)
    monkeypatch.setattr(torch.cuda, "current_stream",
                        lambda device=None: types.SimpleNamespace(cuda_stream=CALLER))
    return log


def test_other_stream_is_ordered_both_ways(calls):
    p = types.SimpleNamespace(h=None, stream=HANDLE)
    x = torch.tensor([1.0, 2.0], requires_grad=True)
    y = torch.tensor([3.0, 4.0], requires_grad=True)
    after, before = ("fftpl_order_after", CALLER), ("fftpl_order_before", CALLER)
    N = A.density_energy(x, y, p)
    # the handle reads x and y after the caller's stream has written them
    assert calls == [after, "energy"]
    del calls[:]
    (3.0 * N).backward()
    # it gathers after the incoming gradient; the caller's stream then waits
    assert calls == [after, "gather", before]
    assert torch.equal(x.grad, 3.0 * x.detach()) and torch.equal(y.grad, 3.0 * y.detach())


def test_other_stream_recomputes_in_order(calls):
    p = types.SimpleNamespace(h=None, stream=HANDLE)
    x = torch.tensor([1.0, 2.0], requires_grad=True)
    y = torch.tensor([3.0, 4.0])
    N = A.density_energy(x, y, p)
    A.density_energy(x, y, p)   # the maps belong to this one now
    del calls[:]
    N.backward()
    assert calls == [("fftpl_order_after", CALLER), "energy", "gather",
                     ("fftpl_order_before", CALLER)]
