"""Cached tunings from before the level-by-level search, whose knobs would turn it off."""
from __future__ import annotations

import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("labels,levels", [(4, True), (70, False)])
def test_a_setting_tuned_without_the_level_search_is_not_taken_over(labels, levels, tmp_path):
    import paper_2507_04130_gb300 as hm

    G = hm.Graph.from_synth(synth.er_graph(2000, 20000, labels, 1, seed=1))
    P = [hm.Pattern.from_synth(p) for p in synth.config4_patterns(count=4)]
    cache = tmp_path / "tune.txt"
    try:
        hm.autotune(G, P, hm.MONO, budget_ms=200, cache=str(cache))
        line = cache.read_text().split(" ", 1)
        # the same key without what it says about the search, and a knob that only the depth-first search reads
        cache.write_text(line[0][line[0].index("g"):] + " " + line[1].replace("split_min=", "split_min=1024 was=", 1))
        hm.set_tuning()
        again = hm.autotune(G, P, hm.MONO, budget_ms=200, cache=str(cache))
        assert again["from_cache"] == (not levels)
        assert hm.autotune(G, P, hm.MONO, budget_ms=200, cache=str(cache))["from_cache"]
    finally:
        hm.set_tuning()
