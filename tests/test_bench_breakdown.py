"""bench.stepwise_breakdown on fakes of the pool and of CUDA events, no GPU: a
report waits for its restore alone, so every event that a time is taken between
has been waited for by itself."""
import sys
import types

import pytest

import bench


class _Event:
    def __init__(self, enable_timing=False):
        self.recorded = self.done = False

    def record(self, stream):
        self.recorded = True

    def synchronize(self):
        assert self.recorded
        self.done = True

    def elapsed_time(self, other):
        if not (self.done and other.done):
            raise RuntimeError("device not ready")
        return 1.0


def test_breakdown_waits_for_its_events(monkeypatch):
    class Event(_Event):
        made = []

        def __init__(self, enable_timing=False):
            super().__init__()
            Event.made.append(self)

        def synchronize(self):        # an event's end is that of all recorded before it
            for e in Event.made[: Event.made.index(self) + 1]:
                e.done = e.recorded

    calls = []
    cuda = types.SimpleNamespace(Event=Event, current_stream=lambda: "stream")
    monkeypatch.setitem(sys.modules, "torch", types.SimpleNamespace(cuda=cuda))
    pool = types.SimpleNamespace(**{n: (lambda *a, n=n: calls.append(n))
                                    for n in ("ingest", "scan", "restore", "advance", "close_slice", "report")})
    got = bench.stepwise_breakdown(pool, ["batch", "batch"], types.SimpleNamespace(k=3), 3)
    assert got == pytest.approx({"ingest": 1.0, "scan": 1.0, "restore": 1.0, "refresh": 1.0, "fused_close": 1.0})
    assert calls.count("report") == 6
