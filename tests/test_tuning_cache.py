"""The tuner's cache (host logic, fake solver and batch): a choice saved for other kernels or out of the present
range is not applied."""
import json

import pytest

from paper_2601_04400_gb300 import tuning
from paper_2601_04400_gb300 import workloads as W


class _Solver:
    _spec = dict(nx=128, ny=64, mu=1e-3, nu=0.0)
    has_ib = True
    variant = None

    def set_tuning(self, v):
        self.variant = v

    def tuning(self):
        return 0, 5


class _Batch:
    set = None

    def __init__(self, most=4):
        self.most = most

    def tuning(self):
        return self.most, self.most, 0, 3

    def set_tuning(self, bps, sched):
        self.set = (bps, sched)

    def set_states(self, states):
        pass


@pytest.fixture
def cache(tmp_path, monkeypatch):
    f = tmp_path / "tuning.json"
    monkeypatch.setattr(tuning, "_CACHE", str(f))
    return lambda d: f.write_text(json.dumps(d))


PROBS = [W.riemann2d(40, ny=30), W.shock_cylinder(nx=64, ny=48)]


def test_choices_of_other_kernels_are_not_applied(cache, monkeypatch):
    s = _Solver()
    # a key as it was when variants named tile shapes, without the kernels' sources
    cache({"128x64|visc=1|av=0|ib=1": {"variant": 2}})
    assert tuning.apply_cached(s) is None and s.variant is None
    cache({tuning._key(s): {"variant": 1}})
    assert tuning.apply_cached(s) == 1 and s.variant == 1
    batch_key = tuning.batch_key(PROBS)
    cache({batch_key: {"choice": [2, 1]}, tuning._key(s): {"variant": 1}})
    assert tuning.autotune_batch(_Batch(), PROBS, []) == {}
    monkeypatch.setattr(tuning, "_sources", lambda: "other")
    assert tuning.cached_variant(s) is None
    assert tuning.batch_key(PROBS) != batch_key


@pytest.mark.parametrize("saved", [-1, 3, 4, "1", None])
def test_variants_out_of_range_are_not_applied(cache, saved):
    s = _Solver()
    cache({tuning._key(s): {"variant": saved}})
    assert tuning.cached_variant(s) is None


@pytest.mark.parametrize("saved,most,want", [([2, 1], 4, (2, 1)), ([0, 2], 4, (0, 2)), ([4, 0], 4, (4, 0)),
                                             ([5, 0], 4, None), ([3, 0], 2, None), ([1, 3], 4, None), ([-1, 0], 4, None),
                                             ([1], 4, None), (None, 4, None)])
def test_batch_choices_out_of_range_are_not_applied(cache, saved, most, want):
    b = _Batch(most)
    cache({tuning.batch_key(PROBS): {"choice": saved}})
    assert tuning.cached_batch_choice(b, PROBS) == want
    if want is not None:
        assert tuning.autotune_batch(b, PROBS, []) == {}
        assert b.set == want
