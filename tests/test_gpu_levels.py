"""The level-by-level extension at its edges: lists around a chunk's 32 candidates
and a group's 32 states, label sets with and without dense group offsets,
levels that do not fit their buffers, every depth, and agreement with the
depth-first search (chosen by any non-default knob)."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


def _pattern(k, arcs, vlab=None, elab=None):
    a = np.array(arcs, dtype=np.int32).reshape(-1, 2)
    return synth.Pattern(k, a[:, 0].copy(), a[:, 1].copy(),
                         np.zeros(k, np.int32) if vlab is None else np.array(vlab, np.int32),
                         np.zeros(len(a), np.int32) if elab is None else np.array(elab, np.int32))


@pytest.mark.parametrize("d", [1, 2, 31, 32, 33, 63, 64, 65, 1000])
def test_fans_of_every_size(d):
    """A hub with d out-neighbours and three more with d, 1 and 0: ordered pairs, and pairs with a common end."""
    import paper_2507_04130_gb300 as hm

    n = d + 4
    hubs = [(0, d), (1, d), (2, 1), (3, 0)]
    src = np.concatenate([np.full(c, h) for h, c in hubs]).astype(np.int32)
    dst = np.concatenate([np.arange(4, 4 + c) for _, c in hubs]).astype(np.int32)
    G = hm.Graph(n, src, dst, np.zeros(n, np.int32), np.zeros(len(src), np.int32))
    fan = hm.Pattern.from_synth(_pattern(3, [(0, 1), (0, 2)]))
    rows = hm.enumerate_matches(G, fan, hm.MONO, capacity=2 * d * d + 8).cpu().numpy()
    want = np.array([(h, a, b) for h, c in hubs for a in range(4, 4 + c) for b in range(4, 4 + c) if a != b],
                    dtype=np.int32).reshape(-1, 3)
    assert np.array_equal(rows, want)
    # 0 -> 1 <- 2 -> 3: the two full hubs (both ways, distinct ends), and the small one with each of them
    zigzag = hm.Pattern.from_synth(_pattern(4, [(0, 1), (2, 1), (2, 3)]))
    outs = {h: set(range(4, 4 + c)) for h, c in hubs}
    count = sum(len(outs[b] - {x}) for a in outs for b in outs if a != b for x in outs[a] & outs[b])
    assert hm.count_matches(G, zigzag, hm.MONO) == count


@pytest.mark.parametrize("nv,ne,shift", [(1, 1, 0), (8, 8, 0), (13, 5, 0), (4, 3, -7), (3, 2, 1 << 20)])
def test_label_sets(nv, ne, shift):
    """64 classes have dense group offsets, 65 do not; labels may be any int32."""
    import paper_2507_04130_gb300 as hm

    g0 = synth.er_graph(120, 2600, nv, ne, seed=nv * 10 + ne)
    g = synth.Graph(g0.n, g0.src, g0.dst, g0.vlab + np.int32(shift), g0.elab - np.int32(shift))
    G, og = hm.Graph.from_synth(g), oracle.OracleGraph.from_synth(g)
    rng = np.random.default_rng(5)
    for k in (3, 4, 5):
        for _ in range(3):
            # an induced piece of the graph, so that there are matches; and a label the graph does not have
            p = synth.random_pattern(rng, k, 0.45, n_vlab=nv, n_elab=ne)
            p = synth.Pattern(k, p.src, p.dst, p.vlab + np.int32(shift), p.elab - np.int32(shift))
            q = synth.Pattern(k, p.src, p.dst, p.vlab, np.where(np.arange(p.mp) == p.mp - 1, p.elab + 999, p.elab)
                              .astype(np.int32))
            for mode in (hm.MONO, hm.INDUCED):
                want, rows = og.match(p, mode)
                got = hm.enumerate_matches(G, hm.Pattern.from_synth(p), mode)
                assert np.array_equal(got.cpu().numpy(), rows.reshape(-1, k))
                assert hm.count_matches(G, hm.Pattern.from_synth(p), mode) == want
                assert hm.count_matches(G, hm.Pattern.from_synth(q), mode) == 0


def test_every_depth_agrees_with_the_depth_first_search():
    import paper_2507_04130_gb300 as hm

    g = synth.er_graph(1500, 6000, 2, 1, seed=31)
    G = hm.Graph.from_synth(g)
    rng = np.random.default_rng(8)
    pats = []
    for k in list(range(3, 13)) + [16, 20]:
        p = synth.random_pattern(rng, k, min(1.0, (k + 2) / (k * (k - 1))), n_vlab=2, n_elab=1)
        pats.append(hm.Pattern.from_synth(p))
    level = [[hm.count_matches(G, p, mode) for mode in (hm.MONO, hm.INDUCED)] for p in pats]
    batch = [hm.count_batch(G, pats, mode) for mode in (hm.MONO, hm.INDUCED)]
    hm.set_tuning(seeds_per_fetch=2)
    try:
        deep = [[hm.count_matches(G, p, mode) for mode in (hm.MONO, hm.INDUCED)] for p in pats]
    finally:
        hm.set_tuning()
    assert level == deep and [list(c) for c in zip(*batch)] == deep
    assert sum(c for c, _ in deep) > 0


def test_levels_that_do_not_fit_are_worked_off_in_parts():
    """A server under a small budget gives the extension 8 MiB: the inner levels here need many times that."""
    import paper_2507_04130_gb300 as hm

    g = synth.config2_graph(scale=11)
    g = synth.Graph(g.n, g.src, g.dst, np.zeros(g.n, np.int32), np.zeros(g.m, np.int32))
    G = hm.Graph.from_synth(g)
    pats = [_pattern(4, [(0, 1), (1, 2), (2, 3), (3, 0)]), _pattern(5, [(0, 1), (1, 2), (2, 0), (2, 3), (3, 0), (4, 0), (4, 3)]),
            _pattern(3, [(0, 1), (1, 2), (0, 2)])]
    want = [hm.count_matches(G, hm.Pattern.from_synth(p), hm.INDUCED) for p in pats]
    srv = hm.Server(G, slots=1, max_batch=8, mem_budget=(12 << 20) + 72 * g.m + (1 << 20))
    try:
        ids = [srv.submit(p, hm.INDUCED, want_rows=False) for p in pats]
        assert [srv.result(q)["count"] for q in ids] == want
    finally:
        srv.close()
    assert min(want) > 0


def test_filter_by_endpoint_agrees_with_the_depth_first_search():
    """From 2^23 arcs on the level search probes words of the fixed vertex's own: hubs, arcs
    at both ends of the id range, long runs of isolated vertices between, two arc labels."""
    import paper_2507_04130_gb300 as hm

    rng = np.random.default_rng(12)
    n, core, m = 400_000, 70_000, (1 << 23) + 999
    u = rng.integers(0, core, m + 400_000)
    v = rng.integers(0, core, m + 400_000)
    u[:20_000], v[:20_000] = 5, np.arange(100, 20_100)
    u[20_000:40_000], v[20_000:40_000] = np.arange(100, 20_100), 5
    key = np.unique(np.where(u < core // 2, u, n - core + u) * n + np.where(v < core // 2, v, n - core + v))
    key = key[key // n != key % n]
    key = np.sort(rng.permutation(key)[:m])
    assert key.size == m
    G = hm.Graph(n, (key // n).astype(np.int32), (key % n).astype(np.int32), rng.integers(0, 2, n).astype(np.int32),
                 rng.integers(3, 5, m).astype(np.int32))
    pats = [hm.Pattern.from_synth(p) for p in (
        _pattern(3, [(0, 1), (1, 2), (2, 0)], [0, 1, 0], [3, 4, 3]),
        _pattern(3, [(0, 1), (1, 2), (0, 2)], [1, 1, 0], [4, 4, 3]),
        _pattern(4, [(0, 1), (1, 2), (2, 3), (3, 0), (0, 2)], [0, 1, 1, 0], [3, 3, 4, 4, 3]))]
    level = [[hm.count_matches(G, p, mode) for mode in (hm.MONO, hm.INDUCED)] for p in pats]
    batch = [hm.count_batch(G, pats, mode) for mode in (hm.MONO, hm.INDUCED)]
    hm.set_tuning(seeds_per_fetch=2)
    try:
        deep = [[hm.count_matches(G, p, mode) for mode in (hm.MONO, hm.INDUCED)] for p in pats]
    finally:
        hm.set_tuning()
    assert level == deep and [list(c) for c in zip(*batch)] == deep
    assert min(c for c, _ in deep) > 0
