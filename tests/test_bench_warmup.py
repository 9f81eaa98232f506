"""bench.py runs exactly the warm-up steps that its line states (CPU, a stand-in solver)."""
import pytest

import bench


class Solver:
    def __init__(self, steps_of):
        self.steps_of, self.calls = steps_of, []

    def launch_steps(self, n):
        return self.steps_of(n)

    def step(self, n):
        self.calls.append(n)


@pytest.mark.parametrize("warmup", [3, 4, 5, 20])
@pytest.mark.parametrize("spl", [1, 2, 4])
def test_warm_up_takes_its_steps_and_no_more(warmup, spl):
    s = Solver(lambda n: min(n, spl))
    assert bench.warm_up(s, warmup) == spl
    assert sum(s.calls) == warmup
    assert set(s.calls[1:]) <= {spl}  # a remainder first, then calls like the timed ones
