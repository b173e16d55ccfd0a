"""Row order at the sizes where the small sort can go wrong: list lengths around
a warp's, a tile's and the path's limits, keys that leave room for the row
number in 128 bits, that just fit, and that do not fit.

The target is N disjoint directed paths of k vertices with shuffled ids, so a
k-vertex path pattern has exactly N matches (the paths) and the expected rows
are the paths sorted lexicographically, from numpy alone.
"""
from __future__ import annotations

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def _paths(k, count, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    rows = rng.permutation(k * count).astype(np.int32).reshape(count, k)
    src, dst = rows[:, :-1].reshape(-1), rows[:, 1:].reshape(-1)
    n = k * count
    g = synth.Graph(n, src, dst, np.zeros(n, np.int32), np.zeros(src.shape[0], np.int32))
    return g, rows[np.lexsort(rows.T[::-1])]


def _path_pattern(k, vlab=0):
    a = np.arange(k, dtype=np.int32)
    return synth.Pattern(k, a[:-1], a[1:], np.full(k, vlab, np.int32), np.zeros(k - 1, np.int32))


@pytest.mark.parametrize("k,count", [
    (2, 1), (2, 2), (2, 15), (2, 16), (2, 17), (2, 63), (2, 64), (2, 65), (2, 127), (2, 128), (2, 129),
    (2, 12287), (2, 12288), (2, 12289),          # the last counted and the first radix-sorted size
    (3, 1000), (4, 4099), (5, 700),
    (6, 10923), (7, 2341), (8, 1000), (8, 4097),  # 6 x 17 + 14, 7 x 15 + 12, 8 x 13 + 10 bits; 8 x 16 + 13: too long
    (9, 1500), (10, 2000), (20, 300),             # keys of more than 128 bits
])
def test_rows_of_disjoint_paths(k, count):
    import paper_2507_04130_gb300 as hm

    g, want = _paths(k, count, seed=1000 * k + count)
    G = hm.Graph.from_synth(g)
    got = hm.enumerate_matches(G, hm.Pattern.from_synth(_path_pattern(k)), hm.MONO).cpu().numpy()
    assert np.array_equal(got, want)


@pytest.mark.parametrize("counts", [(1, 0, 64, 65), (300, 2, 1, 129), (3000, 5, 700, 4096), (24000, 100, 3, 1)])
def test_rows_of_a_batch(counts):
    """Paths of 2, 3, 7 and 10 vertices, each length with its own vertex label, as one batch."""
    import paper_2507_04130_gb300 as hm

    ks, n, src, dst, vlab, wants = (2, 3, 7, 10), 0, [], [], [], []
    for lab, (k, c) in enumerate(zip(ks, counts)):
        g, want = _paths(k, c, seed=17 * k + c)
        src.append(g.src + n)
        dst.append(g.dst + n)
        vlab.append(np.full(g.n, lab, np.int32))
        wants.append(want + n)
        n += g.n
    src, dst = np.concatenate(src).astype(np.int32), np.concatenate(dst).astype(np.int32)
    G = hm.Graph(n, src, dst, np.concatenate(vlab), np.zeros(src.shape[0], np.int32))
    pats = [hm.Pattern.from_synth(_path_pattern(k, lab)) for lab, k in enumerate(ks)]
    for got, want in zip(hm.enumerate_batch(G, pats, hm.INDUCED), wants):
        assert np.array_equal(got.cpu().numpy(), want)
