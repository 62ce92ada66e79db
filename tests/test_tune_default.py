"""Host logic of the autotuner beside the library's own height rule (no GPU):
the rule (height 0) is timed in turn with the fastest fixed height and kept
where it is no slower, for a grid and for a patch level, and a choice is read
back only for the library it was timed on."""
import json

import pytest

from paper_1605_05320_gb300 import tune


class FakeObject:
    """A patch set of one level, or a grid."""
    patches = [(1, 0.0, 0.0, 40, 40, 1.0, 1.0)]
    levels = [1]
    h = object()

    class desc:
        nx, ny = 64, 64

    def step(self, *a):
        pass


def setup(monkeypatch, path, times, lib="a"):
    """times: us per step by height.  Returns the heights applied, in order."""
    monkeypatch.setenv("SWA_TUNE_CACHE", str(path))
    monkeypatch.setattr(tune, "_cache", {})
    monkeypatch.setattr(tune, "_loaded_from", None)
    monkeypatch.setattr(tune, "_device", lambda: "GPU-under-test")
    monkeypatch.setattr(tune, "_library", lambda: lib, raising=False)
    applied = []
    monkeypatch.setattr(tune.S, "swa_patches_set_tile_rows", lambda h, lv, r: applied.append(r))
    monkeypatch.setattr(tune.S, "swa_grid_set_strip_rows", lambda h, r: applied.append(r))
    monkeypatch.setattr(tune, "_time", lambda fn, steps: times[applied[-1]])

    def in_turn(apply, rows, run, steps):
        out = []
        for r in rows:
            apply(r)
            out.append(times[r])
        return out

    monkeypatch.setattr(tune, "_time_in_turn", in_turn, raising=False)
    return applied


def tune_level():
    return tune.tune_patches(FakeObject())[1]


def tune_grid():
    return tune.tune_grid(FakeObject())


@pytest.mark.parametrize("run", [tune_level, tune_grid])
@pytest.mark.parametrize("rule,expect", [(5.0, 0), (7.0, 0), (7.5, 16)])
def test_rule_is_kept_where_it_is_no_slower(monkeypatch, tmp_path, run, rule, expect):
    applied = setup(monkeypatch, tmp_path / "t.json", {0: rule, 16: 7.0, 32: 9.0, 64: 8.0})
    assert run() == expect
    assert applied[-1] == expect           # and applied to the object


def test_choice_of_another_library_is_timed_again(monkeypatch, tmp_path):
    path = tmp_path / "t.json"
    # a choice made before the rule was a candidate: the key named no library
    path.write_text(json.dumps({tune._key(["GPU-under-test"] + tune._level_signature(
        FakeObject(), 1)): 32}))
    setup(monkeypatch, path, {0: 1.0, 16: 7.0, 32: 9.0}, lib="a")
    assert tune_level() == 0
    setup(monkeypatch, path, {0: 9.0, 16: 7.0, 32: 8.0}, lib="b")
    assert tune_level() == 16
    applied = setup(monkeypatch, path, {}, lib="a")   # read back: nothing is timed
    assert tune_level() == 0 and applied == [0]
