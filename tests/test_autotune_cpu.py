"""What the tuner times, keeps and leaves alone, on a stand-in for a lattice."""
import pytest

from paper_1505_02037_gb300 import autotune


class Stand:
    """Form i takes `ms[i]` a step; counts the steps it was made to take."""

    def __init__(self, ms, shift=False, streaming=1, shape=(64, 64, 64)):
        self.vset, self.storage, self.streaming, self.shape = 3, 0, streaming, shape
        self.cells = shape[0] * shape[1] * shape[2]
        self.deriv_mode = 0
        self.variants = list(ms)
        self.ms = list(ms.values())
        self.variant = 0
        self.steps = 0
        self.has_shift = shift

    def set_variant(self, v):
        self.variant = v

    def step_timed(self, n=1):
        self.steps += n
        return 0.0, n * self.ms[self.variant]


@pytest.fixture(autouse=True)
def fresh(monkeypatch):
    monkeypatch.setattr(autotune, "_cache", {})


def test_fastest_form_is_kept_and_found_again():
    a = Stand({"x": 3.0, "y": 1.0, "z": 2.0})
    assert set(autotune.tune(a)) == {"x", "y", "z"} and a.variant == 1
    b = Stand({"x": 3.0, "y": 1.0, "z": 2.0})
    assert autotune.tune(b) == {} and b.variant == 1 and b.steps == 0


def test_shifted_lattice_is_left_alone():
    # every form runs the same kernel: whichever is "fastest" is noise
    a = Stand({"x": 1.0, "y": 0.99}, shift=True)
    assert autotune.tune(a) == {} and a.variant == 0 and a.steps == 0
    b = Stand({"x": 1.0, "y": 2.0})
    assert autotune.tune(b) and b.variant == 0


@pytest.mark.parametrize("shape,streaming,tried", [
    ((20, 20, 20), 1, True), ((16384, 1, 1), 1, True), ((16385, 1, 1), 1, False),
    ((64, 64, 64), 1, False), ((20, 20, 20), 2, False)])
def test_lane_forms_are_tried_where_they_can_win(shape, streaming, tried):
    a = Stand({"P1-reread": 2.0, "lanes16": 3.0, "lanes8": 1.0}, streaming=streaming, shape=shape)
    times = autotune.tune(a)
    assert ("lanes16" in times) == tried and ("lanes8" in times) == tried
    assert a.variant == (2 if tried else 0)
