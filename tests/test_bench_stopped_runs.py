"""The benchmark times only attempts that ran.  A relaxation that has stopped
returns from further attempts at once, so a block of timed attempts in which a
run stops is dropped and the run starts again from its initial state; a run
that stops within its first block is an error (no GPU: the device's part is
played by counters)."""
import types

import numpy as np
import pytest

import bench


class _Relax:
    """Runs `life` attempts of 2 ms after set_x; those after that return in
    0.05 ms."""

    def __init__(self, life):
        self.life, self.ran, self.starts, self.clock = life, 0, 0, 0.0

    def set_B0(self, B0):
        pass

    def set_x(self, x):
        self.ran, self.starts = 0, self.starts + 1

    def attempts(self, n):
        for _ in range(n):
            live = self.ran < self.life
            self.ran += live
            self.clock += 2.0 if live else 0.05

    def profile_attempt(self):
        live = self.ran < self.life
        self.attempts(1)
        return [0.25 if live else 0.01] * 7

    def stats(self):
        return {"accepted": self.ran, "rejected": 0}


def _time(monkeypatch, life, min_s, steps=5):
    r = _Relax(life)

    class Event:
        def __init__(self, enable_timing):
            pass

        def record(self):
            self.t = r.clock

        def elapsed_time(self, other):
            return other.t - self.t

    tensor = types.SimpleNamespace(cuda=lambda: None)
    torch = types.SimpleNamespace(
        from_numpy=lambda a: tensor,
        cuda=types.SimpleNamespace(Event=Event, synchronize=lambda: None))
    monkeypatch.setattr(bench, "new_relaxation", lambda *a: r)
    w = types.SimpleNamespace(x0=None, B0=None)
    flush = types.SimpleNamespace(zero_=lambda: None)
    out = bench.time_mode(None, torch, w, "fp64", "nnn", steps, 3, flush, min_s)
    return r, out[1], out[2]


@pytest.mark.parametrize("life", [13, 14, 18, 23, 1000])
def test_every_timed_attempt_ran(monkeypatch, life):
    r, whole, split = _time(monkeypatch, life, min_s=0.1)
    assert len(whole) % 5 == 0 and np.allclose(whole, 2.0) and whole.sum() >= 100.0
    assert split.shape == (5, 7) and np.all(split == 0.25)
    assert r.starts == 1 if life == 1000 else r.starts > 1


def test_a_run_that_stops_at_once_is_an_error(monkeypatch):
    with pytest.raises(RuntimeError):
        _time(monkeypatch, 7, min_s=0.1)
