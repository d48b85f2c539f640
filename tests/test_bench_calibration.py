"""The bench's calibration of the pipeline's compute phase against models of a call's time: rounds
that add to it, and rounds that misses hide until they take longer than those."""
import os
import sys

import pytest

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench  # noqa: E402


class Call:
    """time_ms(rounds) of a call with misses of `io` ms and rounds of `cost` ms, +-2% by turns."""

    def __init__(self, io, cost, hidden):
        self.io, self.cost, self.hidden, self.longest, self.calls = io, cost, hidden, 0.0, 0

    def __call__(self, rounds):
        self.calls += 1
        t = max(self.io, self.cost * rounds) if self.hidden else self.io + self.cost * rounds
        t *= 1.02 if self.calls % 2 else 0.98
        self.longest = max(self.longest, t)
        return t


@pytest.mark.parametrize("hidden", [False, True])
@pytest.mark.parametrize("io", [0.02, 0.3, 5.0, 100.0])
@pytest.mark.parametrize("cost", [1e-6, 1e-5, 1e-3])
def test_cost_of_a_round(io, cost, hidden):
    call = Call(io, cost, hidden)
    got = bench.compute_round_ms(call)
    # the noise of two calls over a doubling, from cost * n >= 2 io on: at most
    # 0.02 * (1.5 + 2.5) cost * n
    assert got == pytest.approx(cost, rel=0.09)
    # none is longer than the last doubling (or the smallest one, of 4,000 rounds)
    assert call.longest <= 1.05 * max(12 * io + 1.0, io + 4000 * cost)


def test_gives_up_on_rounds_that_take_no_time():
    with pytest.raises(RuntimeError):
        bench.compute_round_ms(lambda rounds: 1.0)
