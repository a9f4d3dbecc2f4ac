"""The autotuner's choice between forms that are nearly as fast, with a clock that drifts (no GPU: fake events)."""
import types

from paper_2509_06433_gb300 import autotune


def test_forms_timed_in_turn_are_compared_fairly(monkeypatch):
    now, speed = [0.0], [1.0]

    class Event:
        def __init__(self, enable_timing):
            self.at = None

        def record(self, stream):
            self.at = now[0]

        def elapsed_time(self, other):
            return other.at - self.at

    monkeypatch.setattr(autotune.torch, "cuda", types.SimpleNamespace(Event=Event, synchronize=lambda: None))

    def form(ms):
        def run():
            now[0] += ms * speed[0]
            speed[0] *= 1.01  # every launch makes the next one 1% slower
        return run

    two, one = form(1.03), form(1.00)
    assert autotune._time(two, 7, None) < autotune._time(one, 7, None)  # one after the other: the first one wins
    slow, fast = autotune._time_in_turn([two, one], 7, None)
    assert fast < slow
