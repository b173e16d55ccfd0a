"""A server's memory budget: rows may fill all that queries leave of it."""
from __future__ import annotations

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

BATCH_FIXED = 12 << 20


def test_rows_that_fill_the_budget_are_kept():
    """Ordered pairs of a hub's 7,400 neighbours (657 MB of rows) under a budget of 1 MB more than they need."""
    import paper_2507_04130_gb300 as hm

    d = 7400
    z = np.zeros(d, np.int32)
    G = hm.Graph(d + 1, z, np.arange(1, d + 1, dtype=np.int32), np.zeros(d + 1, np.int32), z)
    fan = synth.Pattern(3, z[:2], np.array([1, 2], np.int32), z[:3], z[:2])
    budget = 12 * d * (d - 1) + BATCH_FIXED + 24 * d + (1 << 20)
    srv = hm.Server(G, slots=1, max_batch=4, mem_budget=budget)
    try:
        r = srv.result(srv.submit(fan, hm.MONO))
        assert r["count"] == d * (d - 1) and not r["rows_dropped"]
        rows = r["rows"]
        assert np.array_equal(rows[:, 1], np.repeat(np.arange(1, d + 1, dtype=np.int32), d - 1))
        assert not rows[:, 0].any() and (rows[:, 1] != rows[:, 2]).all()
        assert (np.diff(rows[:, 2].reshape(d, d - 1), axis=1) > 0).all()
    finally:
        srv.close()


@pytest.mark.parametrize("slots,budget", [(1, 13 << 20), (2, 64 << 20), (4, 1 << 30), (4, 0)])
def test_bursts_of_deep_patterns_under_any_budget(slots, budget):
    import paper_2507_04130_gb300 as hm

    G = hm.Graph.from_synth(synth.er_graph(600, 3600, 1, 1, seed=4))
    pats = [synth.Pattern(k, np.arange(k - 1, dtype=np.int32), np.arange(1, k, dtype=np.int32),
                          np.zeros(k, np.int32), np.zeros(k - 1, np.int32)) for k in (3, 5, 7)]
    want = [hm.count_matches(G, hm.Pattern.from_synth(p), hm.INDUCED) for p in pats]
    srv = hm.Server(G, slots=slots, max_batch=2, mem_budget=budget)
    try:
        ids = [srv.submit(pats[i % 3], hm.INDUCED, want_rows=i % 3 == 0) for i in range(18)]
        assert [srv.result(q)["count"] for q in ids] == want * 6
    finally:
        srv.close()
