"""A handle that its owner drops while its launches run is destroyed only
after they have finished (fx_expr_destroy itself waits for nothing)."""
import pytest

import paper_2604_22242_gb300 as fx


class Event:
    def __init__(self):
        self.done = False
        self.waits = 0

    def query(self):
        return self.done

    def synchronize(self):
        self.waits += 1
        self.done = True


@pytest.fixture
def destroyed(monkeypatch):
    out = []
    monkeypatch.setattr(fx, "_retired", [])
    monkeypatch.setattr(fx, "fx_expr_destroy", out.append)
    return out


def handle(name, event=None):
    x = fx.Expr.__new__(fx.Expr)
    x.h, x._last = name, event
    return x


def test_idle_handle_is_destroyed_at_once(destroyed):
    handle("a").close()
    assert destroyed == ["a"]


def test_busy_handle_waits_for_its_event(destroyed):
    e = Event()
    x = handle("a", e)
    x.close()
    x.close()
    assert destroyed == []
    e.done = True
    handle("b", Event()).close()
    assert destroyed == ["a"]


def test_held_handles_are_bounded(destroyed):
    events = [Event() for _ in range(fx._RETIRED_MAX + 3)]
    for k, e in enumerate(events):
        handle(k + 1, e).close()
    assert destroyed == [1, 2, 3] and [e.waits for e in events[:4]] == [1, 1, 1, 0]
