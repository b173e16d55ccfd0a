"""A batch's row lists at the line between sorting by counting and the radix sort.

The target is disjoint directed paths with shuffled ids (lists as long as there are paths), so the
expected rows come from numpy alone.
"""
from __future__ import annotations

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("long,short,by_counting", [
    (16384, 0, True), (16385, 0, False), (20000, 700, False), (16384, 16384, True), (16384, 700, True), (2, 16385, False)])
def test_long_lists_are_radix_sorted(long, short, by_counting):
    """Three-vertex paths of label 0 and two-vertex paths of label 1."""
    import paper_2507_04130_gb300 as hm

    rng = np.random.Generator(np.random.PCG64(long + short))
    ids = rng.permutation(3 * long + 2 * short).astype(np.int32)
    a, b = ids[:3 * long].reshape(long, 3), ids[3 * long:].reshape(short, 2)
    vlab = np.zeros(ids.size, np.int32)
    vlab[b.reshape(-1)] = 1
    src, dst = np.concatenate([a[:, 0], a[:, 1], b[:, 0]]), np.concatenate([a[:, 1], a[:, 2], b[:, 1]])
    G = hm.Graph(ids.size, src, dst, vlab, np.zeros(src.size, np.int32))
    z = np.zeros(2, np.int32)
    pats = [synth.Pattern(3, np.array([0, 1], np.int32), np.array([1, 2], np.int32), np.zeros(3, np.int32), z),
            synth.Pattern(2, z[:1], z[:1] + 1, np.ones(2, np.int32), z[:1])]
    got = hm.enumerate_batch(G, [hm.Pattern.from_synth(p) for p in pats], hm.MONO, counts=[long, short])
    # counting: the search and two launches
    assert (hm.last_stats()["kernel_launches"] == 3) == by_counting
    for rows, want in zip(got, (a, b)):
        assert np.array_equal(rows.cpu().numpy(), want[np.lexsort(want.T[::-1])])
