"""What the framework's speed is measured on: labelled subgraph matching through its Python front end.

A case is a target graph (drawn on the GPU from a seed), one or more patterns (fixed by the case, so that graphs of
another seed cost the same) and a call:

  count         count_matches, one call per pattern
  rows          enumerate_matches of one pattern into the caller's buffer of `capacity` rows
  batch_count   count_batch of many patterns
  batch_rows    the C ABI's hm_enumerate_batch of many patterns into one buffer with a region of `capacity` rows for each
  load          Graph(...) from arrays on the device, then one enumerate_matches: a graph that is asked one question
  serve         a burst of queries to a running Server, every one of them waited for

Buffers are filled with -1 before the first pass, so that what a pass returns is the whole buffer: its rows, sorted, then
what was there before.

The graphs are Erdos-Renyi, R-MAT (a power law with hubs) and connectome-shaped (dense power law, cell-type labels).
"""
import ctypes
import math
import random

import numpy as np
import torch

import paper_2507_04130_gb300 as hm
from paper_2507_04130_gb300 import binding

RMAT_ABC = (0.57, 0.19, 0.19)
CELL_TYPES = (0.40, 0.25, 0.15, 0.10, 0.06, 0.04)
ZIPF8 = tuple(w / sum(i ** -1.2 for i in range(1, 9)) for w in (i ** -1.2 for i in range(1, 9)))

# the motifs: arcs (all with label 0) and vertex labels
MOTIFS = {
    "triangle": ([(0, 1), (1, 2), (2, 0)], [0, 0, 0]),
    "cycle3": ([(0, 1), (1, 2), (2, 0)], [0, 1, 2]),
    "ffl_out": ([(0, 1), (1, 2), (0, 2), (2, 3)], [0, 1, 0, 1]),
    "bifan": ([(0, 2), (0, 3), (1, 2), (1, 3)], [0, 1, 0, 1]),
    "cycle4": ([(0, 1), (1, 2), (2, 3), (3, 0)], [0, 1, 0, 1]),
}


def listed():
    return [
        # the smallest call: a graph of 5,000 arcs without labels, about a hundred rows; what launches and waiting cost
        {"name": "er1k_triangle_rows", "graph": "er", "n": 1000, "m": 5000, "vlabs": 1, "elabs": 1, "op": "rows",
         "pattern": "triangle", "mode": "mono", "capacity": 1 << 10, "rows": 125},
        # a larger pattern (the evaluated range is 3 to 20 vertices): a deep search on an ordinary random graph
        {"name": "er20k_k8_count", "graph": "er", "n": 20000, "m": 400000, "vlabs": 4, "elabs": 2, "op": "count",
         "pattern": "random", "k": 8, "density": 0.15, "patterns": 1, "pattern_seed": 5, "mode": "mono", "rows": 0},
        # an ordinary count on a power-law graph of a million arcs
        {"name": "rmat16_ffl_count", "graph": "rmat", "scale": 16, "samples": 1 << 20, "op": "count",
         "pattern": "ffl_out", "mode": "mono", "rows": 0},
        # an ordinary listing of triangles (rows of three vertices), odd number of samples
        {"name": "rmat17_cycle3_rows", "graph": "rmat", "scale": 17, "samples": 2000003, "op": "rows",
         "pattern": "cycle3", "mode": "mono", "capacity": 1 << 16, "rows": 6000},
        # the benchmark's three induced motifs on R-MAT scale 20, with rows
        {"name": "rmat20_ffl_rows", "graph": "rmat", "scale": 20, "samples": 16 << 20, "op": "rows",
         "pattern": "ffl_out", "mode": "induced", "capacity": 1 << 24, "rows": 7000000},
        {"name": "rmat20_bifan_rows", "graph": "rmat", "scale": 20, "samples": 16 << 20, "op": "rows",
         "pattern": "bifan", "mode": "induced", "capacity": 1 << 21, "rows": 920000},
        {"name": "rmat20_cycle4_rows", "graph": "rmat", "scale": 20, "samples": 16 << 20, "op": "rows",
         "pattern": "cycle4", "mode": "induced", "capacity": 1 << 21, "rows": 920000},
        # the largest: five 5-vertex motifs counted in a connectome of 150 million arcs
        {"name": "conn150m_5x_count", "graph": "conn", "n": 300000, "m": 142500000, "recip": 7500000, "op": "count",
         "pattern": "random", "k": 5, "density": 0.5, "patterns": 5, "pattern_seed": 3, "mode": "mono", "rows": 0},
        # many motifs at once: a census of 256 random patterns, counts only
        {"name": "rmat20_batch256_count", "graph": "rmat", "scale": 20, "samples": 16 << 20, "op": "batch_count",
         "pattern": "random", "k": 0, "density": 0.0, "patterns": 256, "pattern_seed": 2, "mode": "mono", "rows": 0},
        # the same with rows, induced, on a smaller graph
        {"name": "rmat18_batch64_rows", "graph": "rmat", "scale": 18, "samples": 4 << 20, "op": "batch_rows",
         "pattern": "random", "k": 0, "density": 0.0, "patterns": 64, "pattern_seed": 7, "mode": "induced",
         "capacity": 1 << 16, "rows": 33000},
        # a new graph of four million arcs, loaded and asked one question
        {"name": "rmat18_load_cycle3", "graph": "rmat", "scale": 18, "samples": 4 << 20, "op": "load",
         "pattern": "cycle3", "mode": "mono", "capacity": 1 << 17, "rows": 19000},
        # a burst of 48 queries to a server with a resident graph
        {"name": "rmat18_serve48", "graph": "rmat", "scale": 18, "samples": 4 << 20, "op": "serve",
         "pattern": "random", "k": 0, "density": 0.0, "patterns": 48, "pattern_seed": 11, "mode": "mono",
         "capacity": 1 << 15, "rows": 11000},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["er", "er", "rmat", "rmat", "rmat", "conn", "batch", "load", "serve"])
    mode = rng.choice(["mono", "induced"])
    if kind == "er":
        # label groups of about one to eight neighbours, which bounds the search of larger patterns
        n, vlabs, elabs = _log(rng, 1000, 60000), rng.randint(2, 6), rng.randint(1, 3)
        m = int(n * min(40.0, vlabs * elabs * rng.uniform(1.5, 8))) | 1
        c = {"graph": "er", "n": n, "m": m, "vlabs": vlabs, "elabs": elabs, "mode": mode, "rows": 0}
        if rng.random() < 0.5:
            return dict(c, op="rows", capacity=1 << 22, pattern=rng.choice(["ffl_out", "bifan", "cycle4"]))
        return dict(c, op="count", pattern="random", k=rng.randint(3, 7), density=round(rng.uniform(0.25, 0.4), 3),
                    patterns=1, pattern_seed=rng.randint(0, 10 ** 6))
    if kind == "conn":
        n = _log(rng, 20000, 300000)
        m = int(n * rng.uniform(100, 450)) | 1
        return {"graph": "conn", "n": n, "m": m, "recip": m // 20, "op": "count", "pattern": "random", "k": 5,
                "density": round(rng.uniform(0.5, 0.7), 3), "patterns": rng.randint(1, 3),
                "pattern_seed": rng.randint(0, 10 ** 6), "mode": mode, "rows": 0}
    scale = rng.randint(11, {"rmat": 19, "batch": 18, "load": 18, "serve": 17}[kind])
    c = {"graph": "rmat", "scale": scale, "samples": int((1 << scale) * rng.uniform(6, 16)) | 1, "mode": mode, "rows": 0}
    if kind == "batch":
        return dict(c, op=rng.choice(["batch_count", "batch_rows"]), pattern="random", k=0, density=0.0, capacity=1 << 17,
                    patterns=_log(rng, 4, 64), pattern_seed=rng.randint(0, 10 ** 6))
    if kind == "serve":
        return dict(c, op="serve", pattern="random", k=0, density=0.0, patterns=rng.randint(4, 48), capacity=1 << 17,
                    pattern_seed=rng.randint(0, 10 ** 6))
    if kind == "load":
        return dict(c, op="load", pattern="cycle3", capacity=1 << 17)
    return dict(c, op=rng.choice(["count", "rows"]), pattern=rng.choice(["cycle3", "ffl_out", "bifan", "cycle4"]),
                capacity=1 << 24)


# ---- graphs ------------------------------------------------------------------

def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _labels(gen, count, weights):
    cum = torch.cumsum(torch.tensor(weights, dtype=torch.float64, device="cuda"), 0)
    r = torch.rand(count, generator=gen, device="cuda", dtype=torch.float64) * cum[-1]
    return torch.searchsorted(cum, r, right=True).clamp_(max=len(weights) - 1).to(torch.int32)


def _er_keys(gen, n, m):
    keys = torch.empty(0, dtype=torch.int64, device="cuda")
    while keys.numel() < m:
        b = 2 * (m - keys.numel()) + 1024
        u = torch.randint(0, n, (b,), generator=gen, device="cuda")
        v = torch.randint(0, n - 1, (b,), generator=gen, device="cuda")
        keys = torch.unique(torch.cat([keys, u * n + v + (v >= u)]))
    return keys[torch.randperm(keys.numel(), generator=gen, device="cuda")[:m]]


def _rmat_keys(gen, scale, samples):
    n = 1 << scale
    a, ab, abc = RMAT_ABC[0], sum(RMAT_ABC[:2]), sum(RMAT_ABC)
    src = torch.zeros(samples, dtype=torch.int64, device="cuda")
    dst = torch.zeros_like(src)
    for _ in range(scale):
        r = torch.rand(samples, generator=gen, device="cuda")
        src.mul_(2).add_(r >= ab)
        dst.mul_(2).add_(((r >= a) & (r < ab)) | (r >= abc))
    keys = torch.unique((src * n + dst)[src != dst])
    perm = torch.randperm(n, generator=gen, device="cuda")
    return perm[keys // n] * n + perm[keys % n]


def _conn_keys(gen, n, m, recip):
    """Chung-Lu: weights from a power law d^-2.1, m distinct arcs, `recip` of them also reversed."""
    dmax = min(50000, max(n // 6, 200))
    dmin = min(98, max(dmax // 20, 2))
    support = torch.arange(dmin, dmax + 1, dtype=torch.float64, device="cuda")
    cum = torch.cumsum(support ** -2.1, 0)

    def weights():
        r = torch.rand(n, generator=gen, device="cuda", dtype=torch.float64) * cum[-1]
        return torch.cumsum(support[torch.searchsorted(cum, r).clamp_(max=support.numel() - 1)], 0)

    w_out, w_in = weights(), weights()

    def ends(w, b):
        r = torch.rand(b, generator=gen, device="cuda", dtype=torch.float64) * w[-1]
        return torch.searchsorted(w, r).clamp_(max=n - 1)

    keys = torch.empty(0, dtype=torch.int64, device="cuda")
    while keys.numel() < m:
        b = int(1.15 * (m - keys.numel())) + 1024
        u, v = ends(w_out, b), ends(w_in, b)
        keys = torch.unique(torch.cat([keys, (u * n + v)[u != v]]))
    if keys.numel() > m:  # evenly spread ones are left out
        drop = torch.linspace(0, keys.numel() - 1, keys.numel() - m, device="cuda", dtype=torch.float64).long()
        keep = torch.ones(keys.numel(), dtype=torch.bool, device="cuda")
        keep[drop] = False
        keys = keys[keep]
    back = keys[torch.randint(0, keys.numel(), (recip,), generator=gen, device="cuda")]
    return torch.unique(torch.cat([keys, (back % n) * n + back // n]))


def _label_weights(case):
    if case["graph"] == "er":
        return (1.0,) * case["vlabs"], case["elabs"]
    return (ZIPF8, 4) if case["graph"] == "rmat" else (CELL_TYPES, 3)


def _arrays(case, seed):
    """n, src, dst, vertex labels, arc labels (int32, on the GPU)."""
    gen = _generator(seed)
    if case["graph"] == "er":
        n, keys = case["n"], _er_keys(gen, case["n"], case["m"])
    elif case["graph"] == "rmat":
        n, keys = 1 << case["scale"], _rmat_keys(gen, case["scale"], case["samples"])
    else:
        n, keys = case["n"], _conn_keys(gen, case["n"], case["m"], case["recip"])
    src, dst = (keys // n).to(torch.int32), (keys % n).to(torch.int32)
    vw, ne = _label_weights(case)
    vlab = _labels(gen, n, vw)
    elab = torch.randint(0, ne, (keys.numel(),), generator=gen, device="cuda", dtype=torch.int32)
    return n, src, dst, vlab, elab


# ---- patterns ----------------------------------------------------------------

class _P:
    """A pattern as plain host arrays."""

    def __init__(self, k, arcs, vlab, elab):
        self.k = k
        self.src = np.array([a for a, _ in arcs], dtype=np.int32)
        self.dst = np.array([b for _, b in arcs], dtype=np.int32)
        self.vlab = np.array(vlab, dtype=np.int32)
        self.elab = np.array(elab, dtype=np.int32)


def _connected(k, arcs):
    seen, todo = {0}, [0]
    while todo:
        x = todo.pop()
        for a, b in arcs:
            for y in ([b] if a == x else []) + ([a] if b == x else []):
                if y not in seen:
                    seen.add(y)
                    todo.append(y)
    return len(seen) == k


def _patterns(case):
    if case["pattern"] in MOTIFS:
        arcs, vlab = MOTIFS[case["pattern"]]
        return [_P(len(vlab), arcs, vlab, [0] * len(arcs))]
    vw, ne = _label_weights(case)
    rng = random.Random(case["pattern_seed"])
    out = []
    for _ in range(case["patterns"]):
        # many patterns at once: sizes and densities of a census
        k = case["k"] or rng.randint(3, 6)
        density = case["density"] or rng.uniform(0.4, 1.0)
        pairs = [(i, j) for i in range(k) for j in range(k) if i != j]
        count = min(max(round(density * len(pairs)), k if case["k"] == 0 else k - 1), len(pairs))
        while True:
            arcs = sorted(rng.sample(pairs, count))
            if _connected(k, arcs):
                break
        # batches and bursts ask for every label alike, single queries for labels as frequent as the graph's
        vlab = rng.choices(range(len(vw)), weights=vw if case["k"] else None, k=k)
        out.append(_P(k, arcs, vlab, [rng.randrange(ne) for _ in arcs]))
    return out


# ---- a pass ------------------------------------------------------------------

def prepare(case, seed):
    mode = hm.MONO if case["mode"] == "mono" else hm.INDUCED
    arrays = _arrays(case, seed)
    plain = _patterns(case)
    st = {"op": case["op"], "mode": mode, "plain": plain}
    if case["op"] == "load":
        st["arrays"] = arrays
    else:
        st["graph"] = hm.Graph(*arrays)
    if case["op"] == "serve":
        st["server"] = hm.Server(st["graph"])
        st["out"] = np.full((len(plain), case["capacity"], max(p.k for p in plain)), -1, np.int32)
    else:
        st["patterns"] = [hm.Pattern.from_synth(p) for p in plain]
    if case["op"] in ("rows", "load"):
        st["out"] = torch.full((case["capacity"] * plain[0].k,), -1, dtype=torch.int32, device="cuda")
    if case["op"] == "batch_rows":
        ends = np.cumsum([0] + [case["capacity"] * p.k for p in plain])
        st["out"] = torch.full((int(ends[-1]),), -1, dtype=torch.int32, device="cuda")
        st["ends"] = ends.astype(np.uint64)
        st["handles"] = (ctypes.c_void_p * len(plain))(*[p.handle.value for p in st["patterns"]])
        st["modes"] = np.full(len(plain), mode, np.int32)
    return st


def _batch_rows(st):
    counts = np.zeros(len(st["plain"]), np.uint64)

    def at(a):
        return ctypes.c_void_p(a.ctypes.data)

    binding.check(binding.lib.hm_enumerate_batch(
        st["graph"].handle, ctypes.cast(st["handles"], ctypes.c_void_p), at(st["modes"]), len(counts),
        ctypes.c_void_p(st["out"].data_ptr()), at(st["ends"]), at(counts),
        ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)), "hm_enumerate_batch")
    return counts.astype(np.int64)


def run(st):
    op, mode = st["op"], st["mode"]
    if op == "count":
        return [hm.count_matches(st["graph"], p, mode) for p in st["patterns"]]
    if op == "rows":
        return len(hm.enumerate_matches(st["graph"], st["patterns"][0], mode, out=st["out"])), st["out"]
    if op == "batch_count":
        return np.array(hm.count_batch(st["graph"], st["patterns"], mode), dtype=np.int64)
    if op == "batch_rows":
        return _batch_rows(st), st["out"]
    if op == "load":
        graph = hm.Graph(*st["arrays"])
        count = len(hm.enumerate_matches(graph, st["patterns"][0], mode, out=st["out"]))
        graph.close()
        return count, st["out"]
    counts = []
    for i, q in enumerate([st["server"].submit(p, mode) for p in st["plain"]]):
        got = st["server"].result(q)
        counts.append(got["count"])
        if got["rows"] is not None:
            st["out"][i, :got["count"], :st["plain"][i].k] = got["rows"]
    return np.array(counts, dtype=np.int64), st["out"]


def _classes(case):
    """The distinct (arc label, source label, target label) of all pattern arcs of a case."""
    return {(int(l), int(p.vlab[a]), int(p.vlab[b]))
            for p in _patterns(case) for a, b, l in zip(p.src, p.dst, p.elab)}


def work(case):
    """The arcs that carry the labels of some pattern arc, read once (two int32 each), and the rows; `load` reads all arrays."""
    m = case["samples"] if case["graph"] == "rmat" else case["m"] + case.get("recip", 0)
    vw, ne = _label_weights(case)
    total = sum(vw)
    arcs = sum(m * vw[a] * vw[b] / (total * total * ne) for _, a, b in _classes(case))
    k = max(p.k for p in _patterns(case))
    out = 4 * k * case["rows"]
    if case["op"] == "load":
        n = 1 << case["scale"]
        return {"bytes": 12 * m + 4 * n + out, "flops": 0}
    return {"bytes": 8 * arcs + out + 64, "flops": 0}


# ---- plain answers -----------------------------------------------------------

class _TooLong(Exception):
    pass


class _Plain:
    """Matching by joins of label classes of arcs, in plain torch (int64)."""

    CHUNK, MOST = 1 << 24, 1 << 31

    def __init__(self, n, src, dst, vlab, elab):
        key, order = torch.sort(src.long() * n + dst.long())
        self.n, self.key, self.vlab = n, key, vlab
        self.elab = elab[order]
        self.src, self.dst = key // n, key % n
        self.joined = 0

    def _list(self, lab, ls, ld, by_dst):
        """Offsets by one end and the other ends, of the arcs with these labels."""
        keep = (self.elab == lab) & (self.vlab[self.src] == ls) & (self.vlab[self.dst] == ld)
        here, there = (self.dst[keep], self.src[keep]) if by_dst else (self.src[keep], self.dst[keep])
        here, order = torch.sort(here, stable=True)
        return torch.searchsorted(here, torch.arange(self.n + 1, device=here.device)), there[order]

    def _label(self, u, v):
        """The label of the arc u -> v, -1 where there is none."""
        if not self.key.numel():
            return torch.full_like(u, -1)
        at = torch.searchsorted(self.key, u * self.n + v).clamp_(max=self.key.numel() - 1)
        return torch.where(self.key[at] == u * self.n + v, self.elab[at].long(), -1)

    def match(self, p, induced):
        arcs = {(int(a), int(b)): int(l) for a, b, l in zip(p.src, p.dst, p.elab)}
        degree = [sum(v in e for e in arcs) for v in range(p.k)]
        order = [max(range(p.k), key=lambda v: degree[v])]
        while len(order) < p.k:
            order.append(max((v for v in range(p.k) if v not in order),
                             key=lambda v: (sum((v, q) in arcs or (q, v) in arcs for q in order), degree[v])))
        rows = torch.nonzero(self.vlab == int(p.vlab[order[0]]))
        for d in range(1, p.k):
            v, done = order[d], order[:d]
            q = min(i for i in range(d) if (done[i], v) in arcs or (v, done[i]) in arcs)
            back = (done[q], v) not in arcs  # the arc to join along runs from v to done[q]
            a, b = (v, done[q]) if back else (done[q], v)
            off, other = self._list(arcs[a, b], int(p.vlab[a]), int(p.vlab[b]), by_dst=back)
            count = (off[1:] - off[:-1])[rows[:, q]]
            ends = torch.cumsum(count, 0)
            total = int(ends[-1]) if len(rows) else 0
            self.joined += total
            if self.joined > self.MOST:
                raise _TooLong
            kept = [rows.new_zeros((0, d + 1))]
            for lo in range(0, total, self.CHUNK):
                j = torch.arange(lo, min(total, lo + self.CHUNK), device=rows.device)
                r = torch.searchsorted(ends, j, right=True)
                c = other[off[rows[r, q]] + j - (ends[r] - count[r])]
                ok = torch.ones_like(c, dtype=torch.bool)
                for i, u in enumerate(done):
                    x = rows[r, i]
                    ok &= x != c
                    for f, s, t in ((arcs.get((u, v)), x, c), (arcs.get((v, u)), c, x)):
                        if f is not None:
                            ok &= self._label(s, t) == f
                        elif induced:
                            ok &= self._label(s, t) < 0
                kept.append(torch.cat([rows[r[ok]], c[ok, None]], 1))
            rows = torch.cat(kept)
        rows = rows[:, torch.tensor([order.index(v) for v in range(p.k)], device=rows.device)]
        for col in range(p.k - 1, -1, -1):
            rows = rows[torch.sort(rows[:, col], stable=True)[1]]
        return rows


def exact(case, seed):
    if case["graph"] == "conn":
        return None
    plain = _Plain(*_arrays(case, seed))
    try:
        rows = [plain.match(p, case["mode"] == "induced") for p in _patterns(case)]
    except _TooLong:
        return None
    counts = [len(r) for r in rows]
    if case["op"] == "count":
        return counts
    if case["op"] == "batch_count":
        return np.array(counts, dtype=np.int64)
    k = max(r.shape[1] for r in rows)
    if case["op"] in ("rows", "load"):
        out = torch.full((case["capacity"], k), -1, dtype=torch.int32, device="cuda")
        out[:counts[0]] = rows[0]
        return counts[0], out.view(-1)
    if case["op"] == "batch_rows":
        out = [torch.full((case["capacity"], r.shape[1]), -1, dtype=torch.int32, device="cuda") for r in rows]
        for o, r in zip(out, rows):
            o[:len(r)] = r
        return np.array(counts, dtype=np.int64), torch.cat([o.view(-1) for o in out])
    out = np.full((len(rows), case["capacity"], k), -1, np.int32)
    for o, r in zip(out, rows):
        o[:len(r), :r.shape[1]] = r.cpu().numpy()
    return np.array(counts, dtype=np.int64), out
