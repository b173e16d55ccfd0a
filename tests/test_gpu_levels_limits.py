"""The level-by-level search at its limits: sums of list lengths that pass 32 bits."""
from __future__ import annotations

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
