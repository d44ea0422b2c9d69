"""Handles of captured steps: their launches have no event to ask, so they are
destroyed outright, outside the capture; and none is asked for during one."""
import gc

import pytest

from test_retire import Event, destroyed, handle  # noqa: F401  (destroyed is the fixture)

import paper_2604_22242_gb300 as fx


def test_during_a_capture_nothing_is_asked_or_destroyed(destroyed, monkeypatch):
    capturing = True
    monkeypatch.setattr(fx, "_capturing", lambda: capturing)

    class Forbidden(Event):
        def query(self):
            assert not capturing
            return super().query()

    old = Forbidden()
    old.done = True
    handle("eager", old).close()
    x = handle("captured")
    x.mark()
    assert x._last is None
    x.close()
    assert destroyed == []
    capturing = False
    handle("next", Event()).close()
    assert destroyed == ["eager", "captured"] and [h for _, h in fx._retired] == ["next"]


@pytest.mark.gpu
def test_captured_step(fxlib):
    """A FusedLoss step captured while an eager step's handle is dropped,
    replayed, and followed by eager steps whose handles are all destroyed."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    F = fxlib.FusedLoss()
    torch.manual_seed(0)

    def matrix(r, c):
        return fxlib.colmajor(r, c, torch.float32).copy_(torch.randn(c, r, device="cuda").t() * 0.5)

    X, W, Y = (matrix(200, 150) for _ in range(3))
    b = torch.randn(200, device="cuda") * 0.5
    params = [t.requires_grad_(True) for t in (X, W, b)]

    def step():
        for t in params:
            t.grad = None
        out = F.apply("sigmoid_sqloss", fxlib.FX_F32, X, W, Y, b)
        out.backward()
        return out

    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        for _ in range(3):
            L = step()
    torch.cuda.synchronize()
    ref = [L.detach().clone()] + [t.grad.clone() for t in params]
    for t in params:
        t.grad = None
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        L = step()  # the eager step's graph, and its handle with it, go here
        gc.collect()
    for _ in range(3):
        graph.replay()
    torch.cuda.synchronize()
    assert all(torch.equal(a, r) for a, r in zip([L.detach()] + [t.grad for t in params], ref))
    del L, graph
    for _ in range(40):
        L = step()
    torch.cuda.synchronize()
    assert all(torch.equal(a, r) for a, r in zip([L.detach()] + [t.grad for t in params], ref))
    del L
    gc.collect()
    x = fxlib.Expr("add2", fxlib.FX_F32)
    x.mark()
    torch.cuda.synchronize()
    x.close()
    assert fxlib._retired == []
