"""Two-vertex patterns: scanned where every one of many arcs carries the labels, level by level elsewhere; the same answers."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nv,ne,n", [(1, 1, 200), (1, 1, 900), (2, 1, 900), (1, 3, 900)])
@pytest.mark.parametrize("arcs", [[(0, 1)], [(0, 1), (1, 0)]])
def test_pairs(nv, ne, n, arcs):
    import paper_2507_04130_gb300 as hm

    g = synth.small_random_graph(n, 0.08, nv, ne, seed=7, recip=0.5, hub=True)
    scanned = nv * ne == 1 and g.m >= 1 << 16
    assert scanned == (nv * ne == 1 and n == 900)
    G, og = hm.Graph.from_synth(g), oracle.OracleGraph.from_synth(g)
    a = np.array(arcs, np.int32)
    p = synth.Pattern(2, a[:, 0].copy(), a[:, 1].copy(), np.zeros(2, np.int32), np.zeros(len(arcs), np.int32))
    P = hm.Pattern.from_synth(p)
    mask = (np.arange(g.n) % 3 == 0).astype(np.uint8)
    for mode in (hm.MONO, hm.INDUCED):
        want, rows = og.match(p, mode)
        rows = rows.reshape(-1, 2)
        assert hm.count_matches(G, P, mode) == want
        by_length = len(arcs) == 1 and mode == hm.MONO
        assert (hm.last_stats()["extend_grid"] == 0) == (scanned and not by_length)
        assert np.array_equal(hm.enumerate_matches(G, P, mode).cpu().numpy(), rows)
        assert (hm.last_stats()["extend_grid"] == 0) == scanned
        for root in (0, 1):
            assert hm.count_matches_rooted(G, P, mode, root, mask) == int(mask[rows[:, root]].sum())
        assert hm.count_batch(G, [P, P], mode) == [want, want]
        assert all(np.array_equal(r.cpu().numpy(), rows) for r in hm.enumerate_batch(G, [P, P], mode))
