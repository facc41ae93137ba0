"""Host logic of the autotuner, with the timed launches replaced by a table.

Left alone, the library cuts a join's work items by its size (item_grain 0)
and merges lists by what they can be searched with (merge_min = merge_ratio =
0).  A tuned configuration must never lose to passing nothing, so that
configuration is among those timed.
"""
import json

import pytest

import paper_2502_06715_gb300 as hc
from paper_2502_06715_gb300 import autotune


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2502_06715_gb300 import build

    build.build_library()


def _tune(monkeypatch, q, ms, mode="count", path=None):
    """The tuner's choice when a configuration takes ms(cfg, materializing)."""
    seen = []

    def fake(query, indexes, cfg, reps, stream, **extra):
        seen.append((cfg.key(), extra.get("mode", "count")))
        return ms(cfg, extra.get("mode") == "materialize")

    monkeypatch.setattr(autotune, "_time", fake)
    idx = [hc.Index.from_stats(100_000, 20_000, 0, 50_000, 50_000) for _ in q.atoms]
    cfg = autotune.Tuner(path=path, reps=1).tune(q, idx, P_list=(4, 16), stream=object(), mode=mode)
    return cfg, seen


def _is_default(cfg):
    return (cfg.item_grain, cfg.merge_min, cfg.merge_ratio) == (0, 0, 0)


@pytest.mark.parametrize("q", [hc.TRIANGLE, hc.FOUR_CYCLE], ids=["triangle", "4-cycle"])
@pytest.mark.parametrize("mode", ["count", "materialize"])
def test_library_defaults_are_tried_and_kept_when_fastest(monkeypatch, q, mode):
    cfg, _ = _tune(monkeypatch, q, lambda c, mat: 1.0 if _is_default(c) else 2.0, mode)
    assert _is_default(cfg) and cfg.ms == 1.0


def test_automatic_merge_is_rechosen_for_materializing(monkeypatch):
    """Counting favours an explicit merge, writing the automatic rule."""
    def ms(c, mat):
        auto = (c.merge_min, c.merge_ratio) == (0, 0)
        return 1.0 if auto == mat else 2.0

    cfg, seen = _tune(monkeypatch, hc.TRIANGLE, ms, "materialize")
    assert (cfg.merge_min, cfg.merge_ratio) == (0, 0)
    assert any(mode == "materialize" and key[2:4] == (0, 0) for key, mode in seen)


def test_explicit_values_still_win_when_faster(monkeypatch):
    cfg, _ = _tune(monkeypatch, hc.TRIANGLE,
                   lambda c, mat: 1.0 + (c.item_grain != 16) + (c.merge_min != autotune.MERGE_OFF))
    assert cfg.item_grain == 16 and cfg.merge_min == autotune.MERGE_OFF


def test_choices_cached_before_the_defaults_were_tried_are_not_used(monkeypatch, tmp_path):
    """A cache file written by a tuner that never timed the defaults keeps its
    old key; the new tuner times again and adds its own."""
    path = str(tmp_path / "tune.json")
    q = hc.TRIANGLE
    idx = [hc.Index.from_stats(100_000, 20_000, 0, 50_000, 50_000) for _ in q.atoms]
    old = {autotune.shape_key(q, idx) + "|P(4, 16)|min1":
           {"shares": [4, 1, 1], "item_grain": 64, "merge_min": 32, "merge_ratio": 4, "slice_grain": 256, "ms": 0.5}}
    with open(path, "w") as f:
        json.dump(old, f)
    cfg, seen = _tune(monkeypatch, q, lambda c, mat: 1.0 if _is_default(c) else 2.0, path=path)
    assert seen and _is_default(cfg)
    with open(path) as f:
        assert len(json.load(f)) == 2
