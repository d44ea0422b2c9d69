"""Handles dropped while others are being retired: by a finalizer that runs in
the middle of it, and by another thread while one waits for the GPU."""
import threading

from test_retire import Event, destroyed, handle  # noqa: F401  (destroyed is the fixture)

import paper_2604_22242_gb300 as fx


class Hook(Event):
    """An event whose query or wait runs something, as a garbage collection
    or another thread would."""

    def __init__(self, on_query=None, on_wait=None):
        super().__init__()
        self.on_query, self.on_wait = on_query, on_wait

    def query(self):
        if self.on_query:
            f, self.on_query = self.on_query, None
            f()
        return self.done

    def synchronize(self):
        if self.on_wait:
            self.on_wait()
        super().synchronize()


def run_bounded(f):
    t = threading.Thread(target=f, daemon=True)
    t.start()
    t.join(20)
    assert not t.is_alive(), "hung"


def test_finalizer_inside_retire(destroyed):
    inner, outer = Event(), Hook()
    outer.on_query = handle("inner", inner).close
    run_bounded(handle("outer", outer).close)
    inner.done = outer.done = True
    done = Event()
    done.done = True
    run_bounded(handle("last", done).close)
    run_bounded(handle("after", done).close)
    assert sorted(destroyed) == ["after", "inner", "last", "outer"] and fx._retired == []


def test_other_threads_do_not_wait_for_the_gpu(destroyed):
    def other():
        handle("other", Event()).close()

    first = Hook(on_wait=lambda: run_bounded(other))
    events = [first] + [Event() for _ in range(fx._RETIRED_MAX)]
    for k, e in enumerate(events):
        run_bounded(handle(k + 1, e).close)
    # the other thread's handle was added meanwhile, and room made for it too
    assert destroyed == [1, 2] and [e.waits for e in events[:3]] == [1, 1, 0]
    assert "other" in [h for _, h in fx._retired] and len(fx._retired) == fx._RETIRED_MAX


def test_every_handle_is_destroyed_once_under_threads(destroyed):
    events = []

    def work(base):
        for k in range(200):
            e = Event()
            events.append(e)
            handle(base + k, e).close()
            if k % 3 == 0:
                for x in events:
                    x.done = True

    ts = [threading.Thread(target=work, args=(1000 * i + 1,)) for i in range(4)]
    for t in ts:
        t.start()
    for t in ts:
        t.join(60)
        assert not t.is_alive()
    for e in events:
        e.done = True
    last = Event()
    last.done = True
    handle("end", last).close()
    handle("end2", last).close()
    assert len(destroyed) == len(set(destroyed)) == 802 and fx._retired == []
