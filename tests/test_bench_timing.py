"""bench.time_steps on the CPU, with the CUDA clock replaced: every operator's first calls (kernel
loading, host schedules) stay outside its timed steps, and bench.py times nothing but through it."""
import inspect
import re

import torch

import bench


def test_first_calls_are_not_timed(monkeypatch):
    now = [0.0]

    class Event:
        def __init__(self, enable_timing):
            assert enable_timing

        def record(self):
            self.t = now[0]

        def elapsed_time(self, other):
            return other.t - self.t

    monkeypatch.setattr(torch.cuda, "Event", Event)
    monkeypatch.setattr(torch.cuda, "synchronize", lambda: None)
    calls = []

    def step(i):
        now[0] += 100.0 if not calls else 1.0  # the first call is slow
        calls.append(i)

    assert bench.time_steps(20, step, 3, 1, torch.device("cpu")) == 1.0
    assert calls == [0, 1, 2, *range(20)]


def test_every_timing_but_the_warmed_ones_warms_up():
    src = inspect.getsource(bench.run_cuda)
    assert "elapsed_time(e1)" not in src  # (no other clock around steps)
    cold = re.findall(r"timed\((?:[^()]|\([^()]*\))*warmup=0\)", src)
    # the headline (warmed up before its graphs), the per-kernel pass after it, and the end-to-end and
    # copy loops (run twice before)
    assert len(cold) == 4, cold
    assert "def timed(n, fn, warmup=3)" in src
