"""The autotuner against leaving the rasterizer alone (no GPU): its present setting,
by default the library's automatic choice, competes with the candidates, and a
choice timed on another build or device is not applied."""
import types

import pytest

from paper_2505_13215_gb300 import abi, autotune


class FakeR:
    W, H, V = [64], [48], 1
    capacity = 1000

    def __init__(self):
        self.options = abi.options()

    def autotune_capacity(self, G):
        return 777

    def set_options(self, ppl_fwd=None, ppl_bwd=None, **kw):
        self.options.pixels_per_lane_fwd, self.options.pixels_per_lane_bwd = ppl_fwd, ppl_bwd

    def setting(self):
        return self.options.pixels_per_lane_fwd, self.options.pixels_per_lane_bwd


G = types.SimpleNamespace(n3=10, n4=5, dtype="float32")


@pytest.fixture
def cache(monkeypatch, tmp_path):
    monkeypatch.setattr(autotune, "CACHE", str(tmp_path / "autotune.json"))


def timer(monkeypatch, ms):
    monkeypatch.setattr(autotune, "_time_steps", lambda R, G, target, reps: ms.get(R.setting(), 5.0))


@pytest.mark.parametrize("present", [(0, 0), (2, 2), (0, 8)])
def test_present_setting_competes(monkeypatch, cache, present):
    timer(monkeypatch, {present: 1.0, (2, 4): 2.0})
    R = FakeR()
    R.set_options(*present)
    r = autotune.tune(R, G, target=None, reps=1)
    assert (r["ppl_fwd"], r["ppl_bwd"]) == present == R.setting() and r["ms"] == 1.0
    # and is applied again from the cache
    R = FakeR()
    assert autotune.tune(R, G, target=None)["cached"] and R.setting() == present


def test_a_faster_candidate_still_wins(monkeypatch, cache):
    timer(monkeypatch, {(0, 0): 2.0, (2, 4): 1.0})
    R = FakeR()
    autotune.tune(R, G, target=None, reps=1)
    assert R.setting() == (2, 4)


def test_given_candidates_are_the_only_ones(monkeypatch, cache):
    timer(monkeypatch, {(0, 0): 1.0})
    R = FakeR()
    autotune.tune(R, G, target=None, reps=1, candidates=((8, 8), (4, 4)))
    assert R.setting() == (8, 8)


def test_choices_of_another_build_are_not_applied(monkeypatch, cache):
    timer(monkeypatch, {(4, 4): 1.0})
    assert not autotune.tune(FakeR(), G, target=None, reps=1)["cached"]
    assert autotune.tune(FakeR(), G, target=None, reps=1)["cached"]
    monkeypatch.setattr(autotune, "_build_key", lambda: "another")
    assert not autotune.tune(FakeR(), G, target=None, reps=1)["cached"]
