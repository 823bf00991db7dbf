"""The autotuner does not leave a simulation slower than untuned (host logic,
fake simulation and events of test_tune.py): the automatic launch shape is a
candidate, every form of the step can be reached, and what a shape's first run
does once (capturing its graph) is not timed."""

import pytest

from paper_1501_03857_gb300 import tune
from test_tune import FakeClock, FakeSim, clear_cache  # noqa: F401


def test_keeps_the_automatic_choice_where_it_is_fastest():
    cost = {c: 4.9e-3 for c in tune.SIM_CANDIDATES}
    cost[(0, 0)] = 4.25e-3
    sim = FakeSim(cost, Lx=100, Ly=100)
    assert tune.tune_simulation(sim)[:2] == (0, 0) and sim.shape == (0, 0)


def test_reaches_every_form():
    """64 marches, 128 is the 24-row tiles, 256 the 16-, 14- and 12-row tiles
    (for more than 4, 3 to 4, and up to 2 rows)."""
    tiles = {s for bx, s in tune.SIM_CANDIDATES if bx == 256}
    assert {64, 128, 256} <= {bx for bx, _ in tune.SIM_CANDIDATES}
    assert tiles & {1, 2} and tiles & {3, 4} and any(s == 0 or s > 4 for s in tiles)


class CapturingSim(FakeSim):
    """A run of 32 steps or more costs `capture` once per shape."""

    def __init__(self, cost, capture, **kw):
        super().__init__(cost, **kw)
        self.capture, self.captured = capture, set()

    def step(self, n):
        super().step(n)
        if n >= 32 and self.shape not in self.captured:
            self.captured.add(self.shape)
            FakeClock.now += self.capture[self.shape]


@pytest.mark.parametrize("steps", [None, 64])
def test_capture_is_not_timed(steps):
    cost = {(0, 0): 0.010, (64, 0): 0.012}
    sim = CapturingSim(cost, {(0, 0): 5.0, (64, 0): 0.1}, Lx=90)
    kw = {} if steps is None else {"steps": steps}
    bx, seg, ms = tune.tune_simulation(sim, candidates=list(cost), **kw)
    assert (bx, seg) == (0, 0) and ms == pytest.approx(0.010)
    assert (0, 0) in sim.captured  # what was timed is what long runs replay
