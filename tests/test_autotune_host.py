"""The batch autotuner's choice, without a GPU: runs longer than two probes are judged by their
second stretch, shorter ones by the probe itself."""
import types

import pytest

from paper_2002_11710_gb300 import api, gen


@pytest.fixture
def clock(monkeypatch):
    """solve_batch advances a clock by a start and a rate per candidate's block size (ms)."""
    now = [0.0]
    cost = {512: (1.0, 0.030), 256: (4.0, 0.020)}

    class Event:
        def __init__(self, enable_timing=False):
            self.t = None

        def record(self):
            self.t = now[0]

        def synchronize(self):
            pass

        def elapsed_time(self, other):
            return other.t - self.t

    def solve_batch(bp, params, out=None):
        start, rate = cost[params.block_threads]
        now[0] += start + rate * params.iterations

    monkeypatch.setattr(api.torch.cuda, "Event", Event)
    monkeypatch.setattr(api, "solve_batch", solve_batch)
    return types.SimpleNamespace(alloc_output=lambda: None)


@pytest.mark.parametrize("iterations,best", [(150, 512), (200, 512), (400, 512), (2000, 256)])
def test_choice_follows_the_length_of_the_run(clock, iterations, best):
    choice, times = api.autotune_batch(clock, api.make_params(5, iterations, gen.PENALTY, 1000),
                                       candidates=((512, False, 1), (256, False, 1)))
    assert choice == (best, False, 1)
    if iterations == 2000:
        assert times == {(512, False, 1): pytest.approx(6.0), (256, False, 1): pytest.approx(4.0)}
