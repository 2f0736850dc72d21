"""The bench's extrapolation of the CPU oracle from a sample, on a clock that the test drives: start-up costs of the first
call (thread pools, page faults) and single slow calls are not charged to every shell."""
import numpy as np
import pytest

import bench
import workloads
from oracle import decomposition, sigw as osigw, synth


class Clock:
    def __init__(self):
        self.t = 0.0

    def perf_counter(self):
        return self.t


@pytest.fixture
def clock(monkeypatch):
    c = Clock()
    dec = type("D", (), {"edges": None, "sigma": {"s": np.zeros(50)}, "phi": {"s": np.zeros((50, 1))}})

    def synthesis(*a):
        c.t += 2.0
        return None, 0

    monkeypatch.setattr(bench, "time", c)
    monkeypatch.setattr(decomposition, "build", lambda: dec)
    monkeypatch.setattr(synth, "phi_tilde", synthesis)
    return c


@pytest.mark.parametrize("extra", [[9.0], [9.0, 0.0, 3.0], [0.0, 4.0], []])
def test_start_up_and_slow_calls_are_left_out(clock, monkeypatch, extra):
    costs = iter(extra)

    def fields(Phi, L, edges, sigma, phi, n_c):
        clock.t += 0.5 + 1.5 * len(sigma) + next(costs, 0.0)

    monkeypatch.setattr(osigw, "envelope_fields", fields)
    spec = workloads.workload("usr256")
    for _ in range(2):
        r = bench.oracle_sample(spec, 2)
        assert r["seconds_per_spectrum"] == pytest.approx(2.0 + 128 * 2 * (0.5 + 50 * 1.5))
        costs = iter([])


def test_no_difference_is_charged_once(clock, monkeypatch):
    def fields(Phi, L, edges, sigma, phi, n_c):
        clock.t += 3.0

    monkeypatch.setattr(osigw, "envelope_fields", fields)
    r = bench.oracle_sample(workloads.workload("usr256"), 1)
    assert r["seconds_per_spectrum"] == pytest.approx(2.0 + 128 * 2 * 50 * 1.5)
