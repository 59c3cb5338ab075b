"""The autotuner times steps alone (a restored state is brought into the form of the step, and
graphs are captured, beforehand), and leaves cache entries from before the link segments."""
import json

import pytest

from paper_1807_01148_gb300 import scenarios as S

pytestmark = pytest.mark.gpu


def _sim():
    from paper_1807_01148_gb300 import gbtraffic as G
    g = G.Sim(S.small_grid(n=6, n_trips=216, steps=600, window_steps=300))
    g.route()
    g.step(250)
    return g


def test_short_trials_pick_the_faster_form(tmp_path):
    # 240 lanes: a step takes 21 us in graphs (sorted form), 14 us in the persistent launch
    # (segments); laying the segments out takes some 60 us once
    picks = [_sim().autotune(4, str(tmp_path / f"t{k}.jsonl"))["mode"] for k in range(5)]
    assert sum(picks) >= 3, picks


def test_entry_from_before_the_segments(tmp_path):
    first, cache = tmp_path / "first.jsonl", tmp_path / "tune.jsonl"
    _sim().autotune(10, str(first))
    line = json.loads(first.read_text())
    line["key"] = line["key"].removesuffix("|seg")
    line.update(mode=0, threads=256, blocks_per_sm=0, grid_per_sm=3)   # 3 is no candidate
    cache.write_text(json.dumps(line) + "\n")
    assert _sim().autotune(10, str(cache))["grid_per_sm"] != 3
    assert len(cache.read_text().splitlines()) == 2
    assert _sim().autotune(10, str(cache)) is not None
    assert len(cache.read_text().splitlines()) == 2   # a hit
