"""What the autotuner's cache is keyed by (``autotune.py``, CPU, stand-in plans and
clock of ``test_autotune_cpu``): the columns and working grid a cell and cutoff
give, and the library's kernels; a cached tiling a plan does not have is dropped."""

import json

from paper_1305_7313_gb300 import autotune
from tests.test_autotune_cpu import FakePlan, FakePsi, FakeTiledPlan, clock  # noqa: F401


class FakeCellPlan(FakePlan):
    """A plan on 72^3 whose working grid holds ``kept`` of ``total`` columns."""

    def __init__(self, kept, total):
        super().__init__(72)
        self.kept, self.total = kept, total

    def columns(self):
        return self.kept, self.total


def tune(clock, plan, nb=64):  # noqa: F811
    clock["cost"] = lambda s: 1.0
    clock["probe"] = lambda: None
    return autotune.tune_apply(plan, FakePsi(nb), None)


def test_the_cell_and_the_cutoff_are_part_of_the_key(clock, monkeypatch):  # noqa: F811
    on64, on72 = (2500, 64 * 66), (3200, 72 * 74)
    assert not tune(clock, FakeCellPlan(*on64)).get("cached")
    assert tune(clock, FakeCellPlan(*on64)).get("cached")
    assert not tune(clock, FakeCellPlan(*on72)).get("cached")  # another cell: other work on the same grid
    monkeypatch.setattr(autotune, "FockBatch", None)
    keys = []
    monkeypatch.setattr(autotune, "_load_cache", lambda: type("D", (), {"get": lambda self, k: keys.append(k) or
                                                                       {"band_block": 16}})())
    for columns in (on64, on72):
        autotune.tune_batch([FakeCellPlan(*columns)], [FakePsi(8)], None)
    assert keys[0] != keys[1]


def test_other_kernels_are_timed_anew(clock, monkeypatch):  # noqa: F811
    assert len(autotune._kernels()) == 12
    assert not tune(clock, FakePlan()).get("cached")
    assert tune(clock, FakePlan()).get("cached")
    monkeypatch.setattr(autotune, "_kernels", lambda: "another")
    assert not tune(clock, FakePlan()).get("cached")


def test_a_cached_tiling_the_plan_does_not_have_is_not_set(clock, tmp_path):  # noqa: F811
    # the column pass of the stand-in has one tiling
    assert not tune(clock, FakeTiledPlan()).get("cached")
    path = tmp_path / "tune.json"
    data = json.loads(path.read_text())
    for hit in data.values():
        hit["tiles"] = [1, 1, 0]
    path.write_text(json.dumps(data))
    plan = FakeTiledPlan()
    assert tune(clock, plan).get("cached") and plan.tiles == [1, 0, 0]
