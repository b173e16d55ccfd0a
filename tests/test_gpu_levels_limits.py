"""The level-by-level search at its limits: sums of list lengths that pass 32 bits, the time
limit when phases are short, levels that pause with rows waiting."""
from __future__ import annotations

import time

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def _pattern(k, arcs, vlab=None, elab=None):
    a = np.array(arcs, dtype=np.int32).reshape(-1, 2)
    return synth.Pattern(k, a[:, 0].copy(), a[:, 1].copy(),
                         np.zeros(k, np.int32) if vlab is None else np.array(vlab, np.int32),
                         np.zeros(len(a), np.int32) if elab is None else np.array(elab, np.int32))


def test_a_group_of_states_with_more_than_32_bits_of_candidates():
    """33 vertices -> hub -> 2^27 + 5 vertices: the 32 states of a full group have 2^32 + 160 candidates."""
    import torch

    import paper_2507_04130_gb300 as hm

    a, d = 33, (1 << 27) + 5
    n = 1 + a + d
    dev = {"dtype": torch.int32, "device": "cuda"}
    src = torch.cat([torch.arange(1, 1 + a, **dev), torch.zeros(d, **dev)])
    dst = torch.cat([torch.zeros(a, **dev), torch.arange(1 + a, n, **dev)])
    G = hm.Graph(n, src, dst, torch.zeros(n, **dev), torch.zeros(a + d, **dev))
    del src, dst
    # the hub, then its in-neighbours, then its out-neighbours one by one (a root mask keeps the
    # last position from being counted by the length of its list)
    path = hm.Pattern.from_synth(_pattern(3, [(0, 1), (1, 2)]), order=[1, 0, 2])
    mask = torch.ones(n, dtype=torch.uint8, device="cuda")
    hm.set_tuning(share_seeds=-1)
    try:
        assert hm.count_matches_rooted(G, path, hm.MONO, 2, mask) == a * d
        mask[1 + a::2] = 0
        assert hm.count_matches_rooted(G, path, hm.MONO, 2, mask) == a * (d // 2)
    finally:
        hm.set_tuning()


def _expect_timeout(hm, call, limit_ms):
    """The call must end with HM_ERR_BUDGET, and within a second or two of its limit."""
    hm.set_budget(limit_ms, 0)
    try:
        t0 = time.perf_counter()
        with pytest.raises(hm.HMError) as ei:
            call()
        took = time.perf_counter() - t0
    finally:
        hm.set_budget(60_000, 0)
    assert ei.value.status == hm.binding.HM_ERR_BUDGET
    assert limit_ms / 1e3 <= took < limit_ms / 1e3 + 2


@pytest.mark.parametrize("k,n,m", [(20, 1500, 6000), (12, 3000, 20000), (20, 100, 300)])
def test_time_limit_of_searches_with_short_phases(k, n, m):
    """Paths in sparse random graphs: far more than the limit allows, in phases of a few chunks per warp."""
    import paper_2507_04130_gb300 as hm

    G = hm.Graph.from_synth(synth.er_graph(n, m, 1, 1, seed=k + n))
    P = hm.Pattern.from_synth(_pattern(k, [(i, i + 1) for i in range(k - 1)]))
    triangle = hm.Pattern.from_synth(_pattern(3, [(0, 1), (1, 2), (2, 0)]))
    want = hm.count_matches(G, triangle, hm.INDUCED)
    _expect_timeout(hm, lambda: hm.count_matches(G, P, hm.MONO), 300)
    _expect_timeout(hm, lambda: hm.count_batch(G, [triangle, P], hm.MONO), 300)
    _expect_timeout(hm, lambda: hm.enumerate_matches(G, P, hm.MONO, capacity=1000), 300)
    assert hm.count_matches(G, triangle, hm.INDUCED) == want
    assert hm.count_batch(G, [triangle], hm.INDUCED) == [want]


def test_time_limit_of_a_server_with_little_memory():
    """A slot whose levels hold 8 MiB works a deep pattern off in many small parts."""
    import paper_2507_04130_gb300 as hm

    G = hm.Graph.from_synth(synth.er_graph(1500, 6000, 1, 1, seed=9))
    P = _pattern(20, [(i, i + 1) for i in range(19)])
    srv = hm.Server(G, slots=1, max_batch=2, mem_budget=(13 << 20))
    try:
        _expect_timeout(hm, lambda: srv.result(srv.submit(P, hm.MONO, want_rows=False)), 300)
        assert srv.result(srv.submit(_pattern(2, [(0, 1)]), hm.MONO, want_rows=False))["count"] == 6000
    finally:
        srv.close()


@pytest.mark.parametrize("k,arcs,n,m", [
    (5, [(0, 1), (1, 2), (2, 3), (3, 4), (4, 0), (4, 1)], 64, 1300),  # no symmetry; 500,000 states of four positions
    (5, [(0, 1), (0, 2), (0, 3), (4, 1), (4, 2), (4, 3)], 80, 2320),  # every match has six images; 290,000 such states
])
def test_levels_that_pause_keep_their_rows(k, arcs, n, m):
    """Inner levels over what a graph of this size gives them, with rows: one call, and as a batch."""
    import torch

    import paper_2507_04130_gb300 as hm

    G = hm.Graph.from_synth(synth.er_graph(n, m, 1, 1, seed=n))
    P = hm.Pattern.from_synth(_pattern(k, arcs), order=list(range(k)))
    got = hm.enumerate_matches(G, P, hm.MONO)
    both = hm.enumerate_batch(G, [P, P], hm.MONO)
    hm.set_tuning(seeds_per_fetch=2)
    try:
        want = hm.enumerate_matches(G, P, hm.MONO, capacity=len(got) + 1)
    finally:
        hm.set_tuning()
    assert len(want) > 100_000
    assert torch.equal(got, want) and torch.equal(both[0], want) and torch.equal(both[1], want)


@pytest.mark.parametrize("k,arcs,mode,n,m", [
    (7, [(0, j) for j in range(1, 7)], 1, 9542, 100_000),      # 107 of 220 ms at 166,000 arcs; 934 in parts of 8 MiB
    (6, [(j, j + 1) for j in range(5)] + [(5, 0)], 0, 2000, 60_000),
])
def test_levels_hold_enough_states_to_match_the_depth_first_search(k, arcs, mode, n, m):
    """Searches of many states on graphs of few arcs: about half the depth-first search's time, and several
    times it where the levels hold too few states."""
    import paper_2507_04130_gb300 as hm

    G = hm.Graph.from_synth(synth.er_graph(n, m, 1, 1, seed=k))
    P = hm.Pattern.from_synth(_pattern(k, arcs))

    def best():
        took = []
        for _ in range(4):
            t0 = time.perf_counter()
            count = hm.count_matches(G, P, mode)
            took.append(time.perf_counter() - t0)
        return count, min(took)

    level = best()
    hm.set_tuning(poll_every=64)  # as fast as the default, and chooses the depth-first search
    try:
        deep = best()
    finally:
        hm.set_tuning()
    assert level[0] == deep[0] and level[1] < 1.3 * deep[1], (level, deep)


@pytest.mark.parametrize("k,n,m,at_least,at_most", [
    (5, 60, 1800, 64, 1 << 20),   # few arcs, much work: more blocks than one per 256 arcs
    (3, 1000, 5000, 1, 64),       # a short call: a small grid, whose barriers cost less
    (2, 1000, 5000, 1, 64),
])
def test_blocks_follow_the_work_not_only_the_arcs(k, n, m, at_least, at_most):
    import oracle
    import paper_2507_04130_gb300 as hm

    g = synth.er_graph(n, m, 1, 1, seed=k)
    G, p = hm.Graph.from_synth(g), _pattern(k, [(i, j) for i in range(k) for j in range(i + 1, k)])
    assert hm.count_matches(G, hm.Pattern.from_synth(p), hm.MONO) == oracle.OracleGraph.from_synth(g).match(p, hm.MONO)[0]
    assert at_least <= hm.last_stats()["extend_grid"] <= at_most
    hm.count_batch(G, [hm.Pattern.from_synth(p)] * 2, hm.MONO)
    assert at_least <= hm.last_stats()["extend_grid"] <= at_most


@pytest.mark.parametrize("arcs", [
    [(0, 1), (0, 2)], [(1, 0), (2, 0), (3, 0)], [(0, 1), (0, 2), (0, 3), (0, 4)],         # ordered leaves
    [(0, 1), (0, 2), (3, 0), (4, 0)], [(0, 1), (1, 0), (0, 2), (0, 3)],                  # two kinds of leaves
    [(0, 1), (1, 2), (3, 1), (1, 4)], [(0, 2), (1, 2), (2, 3)], [(0, 1), (2, 1), (2, 3), (4, 3)],  # leaves that earlier images may be
])
def test_ordered_last_positions_are_counted_by_length(arcs):
    import oracle
    import paper_2507_04130_gb300 as hm

    k = max(max(a) for a in arcs) + 1
    pats = [_pattern(k, arcs), _pattern(k, arcs, elab=[1] * len(arcs))]
    for g in (synth.small_random_graph(40, 0.15, 1, 2, seed=k, recip=0.4, hub=True), synth.er_graph(25, 300, 1, 2, seed=k)):
        G, og = hm.Graph.from_synth(g), oracle.OracleGraph.from_synth(g)
        P = [hm.Pattern.from_synth(p) for p in pats]
        want = [og.match(p, hm.MONO)[0] for p in pats]
        assert [hm.count_matches(G, p, hm.MONO) for p in P] == want
        assert hm.count_batch(G, P, hm.MONO) == want
        hm.set_tuning(share_seeds=-1)
        try:
            assert [hm.count_matches(G, p, hm.MONO) for p in P] == want
        finally:
            hm.set_tuning()
        assert min(want) > 0


def test_ordered_leaves_of_a_hub_are_not_read_one_by_one():
    import paper_2507_04130_gb300 as hm

    d = 3000
    z = np.zeros(d, np.int32)
    G = hm.Graph(d + 1, z, np.arange(1, d + 1, dtype=np.int32), np.zeros(d + 1, np.int32), z)
    fan = hm.Pattern.from_synth(_pattern(3, [(0, 1), (0, 2)]))
    assert fan.automorphisms() == 2
    assert hm.count_matches(G, fan, hm.MONO) == d * (d - 1)
    assert hm.last_stats()["chunks"] < d  # d * d / 32 one by one


def test_a_threads_end_does_not_wait_for_other_streams():
    """A thread that made one call ends while another stream's kernel is still running."""
    import threading

    import torch

    import paper_2507_04130_gb300 as hm

    G = hm.Graph.from_synth(synth.er_graph(1000, 5000, 1, 1, seed=2))
    P = hm.Pattern.from_synth(_pattern(3, [(0, 1), (1, 2), (2, 0)]))
    want, got = hm.count_matches(G, P, hm.MONO), []
    side, own = torch.cuda.Stream(), torch.cuda.Stream()
    done = torch.cuda.Event()

    def once():
        got.append(hm.count_matches(G, P, hm.MONO, stream=own))

    with torch.cuda.stream(side):
        torch.cuda._sleep(2_000_000_000)  # about a second on one SM
        done.record()
    for _ in range(20):
        t = threading.Thread(target=once)
        t.start()
        t.join()
    assert not done.query()
    torch.cuda.synchronize()
    assert got == [want] * 20


def test_more_calls_at_once_than_page_locked_blocks():
    import threading

    import torch

    import paper_2507_04130_gb300 as hm

    G = hm.Graph.from_synth(synth.er_graph(1000, 5000, 1, 1, seed=2))
    pats = [hm.Pattern.from_synth(_pattern(k, [(i, (i + 1) % k) for i in range(k)])) for k in (3, 4, 5)]
    want = [hm.count_matches(G, p, hm.MONO) for p in pats]
    many = [hm.Pattern.from_synth(_pattern(3, [(0, 1), (1, 2)]))] * 4097  # more counts than a block holds
    lots, got = hm.count_batch(G, many[:1], hm.MONO)[0], []

    def work(i):
        s = torch.cuda.Stream()
        for _ in range(20):
            got.append((i % 3, hm.count_matches(G, pats[i % 3], hm.MONO, stream=s)))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(40)]
    for t in threads:
        t.start()
    assert hm.count_batch(G, many, hm.MONO) == [lots] * 4097
    for t in threads:
        t.join()
    assert len(got) == 800 and all(c == want[i] for i, c in got)


def test_a_batch_on_few_arcs_matches_the_depth_first_search():
    """64 six-vertex paths on 916 arcs: states by the million of every pattern, whose levels must not be sized by the arcs."""
    import paper_2507_04130_gb300 as hm

    G = hm.Graph.from_synth(synth.er_graph(70, 916, 1, 1, seed=92))
    P = [hm.Pattern.from_synth(_pattern(6, [(i, i + 1) for i in range(5)]))] * 64

    def best():
        took = []
        for _ in range(5):
            t0 = time.perf_counter()
            counts = hm.count_batch(G, P, hm.MONO)
            took.append(time.perf_counter() - t0)
        return counts, min(took)

    level = best()
    hm.set_tuning(poll_every=64)
    try:
        deep = best()
    finally:
        hm.set_tuning()
    assert level[0] == deep[0] and level[1] < deep[1], (level[1], deep[1])
