// hm_levels.cu -- state extension, level by level, in one persistent launch.
//
// The states of a level (p mapped positions each) are extended together: every
// candidate of every state is one lane's work, so the lanes are full and all
// warps finish at the same time, whatever the distribution of the degrees.
// (The depth-first search with one warp per state, k_extend, kept 2 to 30 % of
// the warps busy wherever a few hubs own the work: a connectome query of 121 M
// leaf candidates took 17.4 ms, of which 90 % was waiting for the last warps.)
//
// A level has two phases, each ended by a grid barrier:
//   ranges   one thread per state: the anchors' label groups (dense group
//            offsets: one lookup of two neighbouring words each), the shortest
//            of which holds the candidates; a state whose anchor has an empty
//            group dies here.  States are taken in groups of up to 32, and a
//            prefix sum over the groups' chunks of 32 candidates numbers all
//            chunks of the level.
//   expand   each warp takes runs of consecutive chunks, finds the group a
//            run starts in, and reads 32 candidates at a time: the filter
//            probes of the other positive conditions reject most; survivors
//            wait in the warp's buffer until 128 are there, then
//            the exact checks run on full warps and the survivors of those
//            become states of the next level, or matches.
// Memory is bounded: an expansion takes no more chunks than the next level's
// buffer can hold survivors of, then the deeper levels are worked off before
// the rest (depth first over slices of levels).
//
// Bound by the latency of its lookups in L2 and HBM (list entry, then filter
// word, per candidate), which many independent warps hide.
#include <algorithm>
#include <atomic>
#include <cstring>
#include <vector>

#include "hm_levels.cuh"

namespace hm {
namespace {

constexpr int kLvThreads = 512;
constexpr int kLvWarps = kLvThreads / 32;
constexpr int kLvMinBlocks = 2;
constexpr uint32_t kFull = 0xffffffffu;
constexpr int kLvBuf = 160;       // survivors of a warp waiting for the exact checks
constexpr int kLvDrain = 128;     // checked when this many wait (a chunk adds at most 32)
constexpr int kLvMaxGrid = 1024;
constexpr int kLvMaxGroups = 1024;  // groups of one block in the ranges phase
constexpr int64_t kLvSeedSlice = 1 << 21;  // depth-2 states taken at a time
constexpr uint64_t kLvBarrierNs = 10ull * 1000 * 1000 * 1000;

struct LvArgs {
  DevGraph G;
  LvCtl *ctl;
  const int32_t *base[kMaxK + 2];  // states of each level; stride[p] words each
  int4 *rng[kMaxK + 2];            // {first candidate, number, driving condition, pattern}
  unsigned long long *upre[kMaxK + 2];  // chunks of the earlier groups of the same block
  unsigned long long *bsum[kMaxK + 2];  // chunks of each block's groups
  int32_t stride[kMaxK + 2];
  int64_t fcap;                    // states a level's buffer holds
  int64_t slice;                   // depth-2 states of a slice
  const unsigned long long *nseeds;
  const int4 *groups;
  const int2 *sorted_seeds;
  const uint8_t *root_mask;
  unsigned long long budget_ns;
  int32_t *rows;
  unsigned long long cap;
  const int32_t *seed_pid;
  const LevelPlan *levels;         // batch: [pattern][kmax]
  const EmitPlan *emit;
  const int8_t *aut;
  unsigned long long *counts;
  const unsigned long long *row_off, *row_cap;
  unsigned long long *row_cursor;
  int32_t kmax;                    // levels 2 .. kmax - 1 (kmax: the deferred position 1)
  int32_t ndefer;
  Cons defer[kMaxCons];
  EmitPlan emit1;
  LevelPlan level1[kMaxK];
};

struct LvShared {
  unsigned long long sum[kLvMaxGroups];      // ranges: chunks of this block's groups
  unsigned long long first[kLvMaxGrid];      // expand: first chunk of each block's groups
  unsigned long long wsum[kLvWarps];
  int4 rec[kLvWarps][32];                    // the group's states with candidates, in order
  int2 buf[kLvWarps][kLvBuf];                // {state, candidate}
  // values all warps share, and each warp's matches, kept out of the registers of the expansion
  unsigned long long made, deadline, begin, take;
  unsigned long long count[kLvWarps];
  uint32_t run_len, nrun;
  unsigned int *claim;
  int ok;
};

__device__ __forceinline__ bool lv_barrier(const LvArgs &A, LvShared &sm, unsigned int target) {
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(&A.ctl->bar, 1u);
    int ok = 1;
    for (;;) {
      if (*(volatile unsigned int *)&A.ctl->bar >= target) break;
      if (*(volatile int32_t *)&A.ctl->status != 0) break;
      if (globaltimer_ns() > sm.deadline + kLvBarrierNs) {
        atomicCAS(&A.ctl->status, 0, kStatQueue);
        break;
      }
      __nanosleep(32);
    }
    __threadfence();
    if (*(volatile int32_t *)&A.ctl->status != 0) ok = 0;
    sm.ok = ok;
  }
  __syncthreads();
  return sm.ok != 0;
}

// Exclusive prefix sum over the block of one value per thread; *total is the sum.
__device__ __forceinline__ unsigned long long lv_block_scan(unsigned long long v, LvShared &sm,
                                                            unsigned long long *total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned long long x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long y = __shfl_up_sync(kFull, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) sm.wsum[warp] = x;
  __syncthreads();
  unsigned long long before = 0, all = 0;
#pragma unroll
  for (int w = 0; w < kLvWarps; ++w) {
    const unsigned long long s = sm.wsum[w];
    if (w < warp) before += s;
    all += s;
  }
  __syncthreads();
  *total = all;
  return before + x - v;
}

// States per group: all 32 lanes' worth when there are enough states for every
// warp, else fewer, so that a small level still spreads over the warps.
// Positions inside a group are 32-bit: g lists of at most maxdeg entries.
__device__ __forceinline__ int lv_group_size(unsigned long long cnt, unsigned long long warps, int32_t maxdeg) {
  int g = 32;
  while (g > 1 && (unsigned long long)maxdeg * g > 0xffffffffull) g >>= 1;
  while (g > 1 && cnt < (unsigned long long)g * warps) g >>= 1;
  return g;
}

__device__ __forceinline__ const int32_t *lv_state(const LvArgs &A, int p, int64_t s) {
  return A.base[p] + s * A.stride[p];
}

// A state's first four images, in registers: most patterns' checks read no
// more of it.  What is not a vertex (unmapped positions, the group in the
// place of a deferred position 1, a pattern number) is -1.
template <bool kShared>
__device__ __forceinline__ int4 lv_images(const int32_t *mp, int p) {
  int4 m;
  if (p == 2) {
    const int2 v = *reinterpret_cast<const int2 *>(mp);
    m = make_int4(v.x, v.y, -1, -1);
  } else {
    m = *reinterpret_cast<const int4 *>(mp);
    if (p == 3) m.w = -1;
  }
  if (kShared) m.y = -1;
  return m;
}

__device__ __forceinline__ int32_t lv_image(const int4 &m, const int32_t *mp, int q) {
  if (q >= 4) return mp[q];
  const int32_t a = q & 1 ? m.y : m.x, b = q & 1 ? m.w : m.z;
  return q & 2 ? b : a;
}

// The candidates of state `s` of level p: {first, number, driving condition | list << 8, pattern}.
// list: 0 out-groups, 1 in-groups, 2 the seeds of a shared group.
template <bool kBatch, bool kShared, bool kSym>
__device__ __forceinline__ int4 lv_range(const LvArgs &A, int p, int64_t s, int32_t pid) {
  const int32_t *mp = lv_state(A, p, s);
  if (kShared && p == A.kmax) {
    const int4 gr = __ldg(A.groups + mp[1]);
    return make_int4(gr.y, gr.z - gr.y, 2 << 8, 0);
  }
  const LevelPlan &L = kBatch ? A.levels[(int64_t)pid * A.kmax + p] : A.level1[p];
  if (kSym && p == 2) {
    // the order constraint between positions 0 and 1 (the injected states stay the validators' output)
    const LevelPlan &L1 = kBatch ? A.levels[(int64_t)pid * A.kmax + 1] : A.level1[1];
    if ((L1.sym_gt && mp[1] <= mp[0]) || (L1.sym_lt && mp[1] >= mp[0])) return make_int4(0, 0, 0, pid);
  }
  int32_t best = INT32_MAX, lo = 0, what = 0;
  for (int j = 0; j < L.npos; ++j) {
    const LvCons cs = L.cons[j];
    if (cs.cls < 0) return make_int4(0, 0, 0, pid);
    const int32_t *ofs = cs.kind == kOut ? A.G.gofs_out : A.G.gofs_in;
    const int64_t at = (int64_t)mp[cs.q] * A.G.ncls + cs.cls;
    const int32_t a = __ldg(ofs + HM_AT(A.G, at, (int64_t)A.G.n * A.G.ncls, kChkGroup));
    const int32_t b = __ldg(ofs + at + 1);
    if (b - a < best) {
      best = b - a;
      lo = a;
      what = j | (cs.kind == kOut ? 0 : 1 << 8);
    }
  }
  return make_int4(lo, best, what, pid);
}

template <bool kBatch, bool kShared, bool kRows, bool kSym>
__device__ __forceinline__ void lv_ranges(const LvArgs &A, LvShared &sm, int p, unsigned long long first,
                                          unsigned long long cnt, int g) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t chunks = (int64_t)((cnt + 31) >> 5), per = (chunks + gridDim.x - 1) / gridDim.x;
  const int64_t c0 = min(chunks, (int64_t)blockIdx.x * per), c1 = min(chunks, c0 + per);
  const int gpc = 32 / g, ngl = (int)(c1 - c0) * gpc;
  for (int64_t c = c0 + warp; c < c1; c += kLvWarps) {
    const unsigned long long i = (unsigned long long)c * 32 + lane;
    int4 r = make_int4(0, 0, 0, 0);
    bool matched = false;
    if (i < cnt) {
      const int64_t s = (int64_t)(first + i);
      int32_t pid = 0;
      if (kBatch) pid = p == 2 ? __ldg(A.seed_pid + s) : lv_state(A, p, s)[p];
      matched = kBatch && A.levels[(int64_t)pid * A.kmax + p].done;
      if (!matched) r = lv_range<kBatch, kShared, kSym>(A, p, s, pid);
      else r.w = pid;
      A.rng[p][i] = r;
    }
    if (kBatch && __any_sync(kFull, matched)) {
      // two-vertex patterns: the validated seed is the match
      const uint32_t peers = __match_any_sync(kFull, matched ? r.w : -1 - lane);
      const int leader = __ffs(peers) - 1;
      unsigned long long at = 0;
      if (matched && lane == leader) {
        atomicAdd(A.counts + r.w, (unsigned long long)__popc(peers));
        if (kRows) at = atomicAdd(A.row_cursor + r.w, (unsigned long long)__popc(peers));
      }
      if (kRows) {
        at = __shfl_sync(kFull, at, leader) + __popc(peers & lanemask_lt());
        if (matched && at < A.row_cap[r.w]) {
          const int32_t *mp = lv_state(A, p, (int64_t)(first + i));
          int32_t *row = A.rows + A.row_off[r.w] + at * 2;
          const EmitPlan &E = A.emit[r.w];
          row[E.orig[0]] = mp[0];
          row[E.orig[1]] = mp[1];
        }
      }
    }
    unsigned long long t = (unsigned long long)(uint32_t)r.y;
    for (int o = 1; o < g; o <<= 1) t += __shfl_xor_sync(kFull, t, o);
    if ((lane & (g - 1)) == 0) sm.sum[(c - c0) * gpc + lane / g] = (t + 31) >> 5;
  }
  __syncthreads();
  // prefix sum over the block's groups
  constexpr int kPer = kLvMaxGroups / kLvThreads;
  unsigned long long v[kPer], sum = 0, all;
#pragma unroll
  for (int t = 0; t < kPer; ++t) {
    const int i = threadIdx.x * kPer + t;
    v[t] = i < ngl ? sm.sum[i] : 0;
    sum += v[t];
  }
  unsigned long long run = lv_block_scan(sum, sm, &all);
#pragma unroll
  for (int t = 0; t < kPer; ++t) {
    const int i = threadIdx.x * kPer + t;
    if (i < ngl) A.upre[p][c0 * gpc + i] = run;
    run += v[t];
  }
  if (threadIdx.x == 0) A.bsum[p][blockIdx.x] = all;
}

// Is x among the group's images sorted_seeds[lo, hi).y (ascending)?
__device__ __forceinline__ bool lv_group_has(const int2 *__restrict__ sv, int32_t lo, int32_t hi, int32_t x) {
  while (lo < hi) {
    const int32_t mid = lo + ((hi - lo) >> 1);
    const int32_t y = __ldg(&sv[mid].y);
    if (y < x) lo = mid + 1;
    else if (y > x) hi = mid;
    else return true;
  }
  return false;
}

// The cheap checks: candidate c of the state at mp for position p.
template <bool kShared, bool kSym>
__device__ __forceinline__ bool lv_first_checks(const LvArgs &A, const LevelPlan &L, const int32_t *mp, int p,
                                                int drive, int32_t c, Bytes &none) {
  const int4 m = lv_images<kShared>(mp, p);
  if (m.x == c || m.y == c || m.z == c || m.w == c) return false;  // injective
  for (int i = 4; i < p; ++i)
    if (mp[i] == c) return false;
  if (L.root && !A.root_mask[c]) return false;
  if (kSym) {
    uint32_t g = L.sym_gt, l = L.sym_lt;
    while (g) {
      const int q = __ffs(g) - 1;
      g &= g - 1;
      if (c <= mp[q]) return false;
    }
    while (l) {
      const int q = __ffs(l) - 1;
      l &= l - 1;
      if (c >= mp[q]) return false;
    }
  }
  for (int j = 0; j < L.npos; ++j) {
    if (j == drive) continue;
    const LvCons cs = L.cons[j];
    const int32_t f = lv_image(m, mp, cs.q);
    ArcKey k = pair_key(cs.kind == kOut ? f : c, cs.kind == kOut ? c : f);
    k.a += cs.la;
    k.b += cs.lb;
    if (!filter_has<false>(A.G, k, none)) return false;
  }
  return true;
}

// The exact checks of a candidate that passed the cheap ones.
template <bool kShared>
__device__ __forceinline__ bool lv_exact_checks(const LvArgs &A, const LevelPlan &L, const int32_t *mp, int p, int drive,
                                                int32_t c, Bytes &none) {
  const int4 m = lv_images<kShared>(mp, p);
  if (L.need_deg) {
    const int4 vi = __ldg(&A.G.vi[HM_AT(A.G, c, A.G.n, kChkVertex)]);
    if (vi.y < L.dout || vi.z < L.din) return false;
  }
  for (int j = 0; j < L.ncons; ++j) {
    if (j == drive) continue;
    const LvCons cs = L.cons[j];
    const int32_t f = lv_image(m, mp, cs.q);
    const bool fwd = cs.kind == kOut || cs.kind == kNotOut;
    const int32_t x = fwd ? f : c, y = fwd ? c : f;
    int32_t lab;
    if (cs.kind <= kIn) {
      if (!arc_find<false>(A.G, x, y, &lab, none) || lab != cs.lab) return false;
    } else if (arc_maybe<false>(A.G, x, y, none) && arc_find<false>(A.G, x, y, &lab, none)) {
      return false;
    }
  }
  return true;
}

// Position 1 chosen from a shared group: v must differ from the match's other
// images and keep the induced non-arcs.
__device__ __forceinline__ bool lv_defer_checks(const LvArgs &A, const int32_t *mp, int k, int32_t v, Bytes &none) {
  for (int i = 0; i < k; ++i)
    if (i != 1 && mp[i] == v) return false;
  for (int j = 0; j < A.ndefer; ++j) {
    const Cons cs = A.defer[j];
    const int32_t f = mp[cs.q];
    const bool fwd = cs.kind == kNotOut;  // the forbidden arc is f(q) -> v
    int32_t lab;
    if (arc_maybe<false>(A.G, fwd ? f : v, fwd ? v : f, none) && arc_find<false>(A.G, fwd ? f : v, fwd ? v : f, &lab, none))
      return false;
  }
  return true;
}

__device__ __forceinline__ void lv_write_row(const EmitPlan &E, int32_t *row, const int32_t *mp, int p, int32_t c,
                                             bool deferred) {
  if (deferred) {
    for (int i = 0; i < E.k; ++i) row[E.orig[i]] = i == 1 ? c : mp[i];
    return;
  }
  for (int i = 0; i < p; ++i) row[E.orig[i]] = mp[i];
  row[E.orig[p]] = c;
}

// The rows of a match and of its automorphic images, from row r on.
__device__ __forceinline__ void lv_write_images(const EmitPlan &E, const int8_t *aut, int32_t *rows,
                                                unsigned long long r, unsigned long long cap, const int32_t *mp,
                                                int p, int32_t c) {
  for (int s = 0; s < E.naut && r + s < cap; ++s)
    for (int v = 0; v < E.k; ++v) {
      const int i = aut[s * kMaxK + v];
      rows[(r + s) * E.k + v] = i < p ? mp[i] : c;
    }
}

// Exact checks on the nbuf waiting survivors; those that pass become states of
// the next level (whose counter stood at sm.made when its buffer was empty) or
// matches.
template <bool kRows, bool kBatch, bool kShared, bool kSym>
__device__ __forceinline__ void lv_drain(const LvArgs &A, LvShared &sm, int p, unsigned long long slice_first,
                                         int2 *buf, int nbuf, int lane) {
  Bytes none;
  const uint32_t lt = lanemask_lt();
  const bool deferred = kShared && p == A.kmax;
  int nok = 0;
  for (int b = 0; b < nbuf; b += 32) {
    const int e = b + lane;
    bool ok = false;
    int2 sc = make_int2(0, 0);
    if (e < nbuf) {
      sc = buf[e];
      const int32_t *mp = lv_state(A, p, (int64_t)(slice_first + (uint32_t)sc.x));
      if (deferred) {
        ok = lv_defer_checks(A, mp, p, sc.y, none);
      } else {
        const int4 r = A.rng[p][(uint32_t)sc.x];
        const LevelPlan &L = kBatch ? A.levels[(int64_t)r.w * A.kmax + p] : A.level1[p];
        ok = lv_exact_checks<kShared>(A, L, mp, p, r.z & 0xff, sc.y, none);
      }
    }
    const uint32_t bal = __ballot_sync(kFull, ok);
    if (ok) buf[nok + __popc(bal & lt)] = sc;  // at or before the entry just read
    nok += __popc(bal);
    __syncwarp();
  }
  if (!nok) return;
  if (kBatch) {
    for (int b = 0; b < nok; b += 32) {
      const int e = b + lane;
      const bool valid = e < nok;
      const int2 sc = valid ? buf[e] : make_int2(0, 0);
      const int64_t s = (int64_t)(slice_first + (uint32_t)sc.x);
      const int32_t *mp = lv_state(A, p, s);
      const int32_t pid = valid ? A.rng[p][(uint32_t)sc.x].w : -1;
      const bool last = valid && A.levels[(int64_t)pid * A.kmax + p].last;
      const uint32_t peers = __match_any_sync(kFull, last ? pid : -1 - lane);
      const int leader = __ffs(peers) - 1;
      if (last) {
        const int naut = kSym ? A.emit[pid].naut : 1;
        unsigned long long at = 0;
        if (lane == leader) {
          atomicAdd(A.counts + pid, (unsigned long long)__popc(peers) * naut);
          if (kRows) at = atomicAdd(A.row_cursor + pid, (unsigned long long)__popc(peers) * naut);
        }
        if (kRows) {
          at = __shfl_sync(peers, at, leader) + (unsigned long long)__popc(peers & lt) * naut;
          const EmitPlan &E = A.emit[pid];
          int32_t *rows = A.rows + A.row_off[pid];
          if (naut > 1) lv_write_images(E, A.aut + E.aut, rows, at, A.row_cap[pid], mp, p, sc.y);
          else if (at < A.row_cap[pid]) lv_write_row(E, rows + at * E.k, mp, p, sc.y, false);
        }
      }
      const bool inner = valid && !last;
      const uint32_t bal = __ballot_sync(kFull, inner);
      if (bal) {
        unsigned long long at = 0;
        if (lane == 0) at = atomicAdd(&A.ctl->next_n[p + 1], (unsigned long long)__popc(bal));
        at = __shfl_sync(kFull, at, 0) - sm.made + __popc(bal & lt);
        if (inner) {
          int32_t *dst = const_cast<int32_t *>(lv_state(A, p + 1, (int64_t)at));
          for (int i = 0; i < p; ++i) dst[i] = mp[i];
          dst[p] = sc.y;
          dst[p + 1] = pid;
        }
      }
    }
    __syncwarp();
    return;
  }
  const bool last = deferred || A.level1[p].last;
  if (kShared && !deferred && last && !kRows && A.ndefer == 0) {
    // a count without induced non-arcs: every image of the group that the match does not use
    unsigned long long add = 0;
    for (int e = lane; e < nok; e += 32) {
      const int2 sc = buf[e];
      const int32_t *mp = lv_state(A, p, (int64_t)(slice_first + (uint32_t)sc.x));
      const int4 gr = __ldg(A.groups + (p == 2 ? (int64_t)(slice_first + (uint32_t)sc.x) : (int64_t)mp[1]));
      int used = lv_group_has(A.sorted_seeds, gr.y, gr.z, sc.y) ? 1 : 0;
      for (int i = 0; i < p; ++i)
        if (i != 1 && lv_group_has(A.sorted_seeds, gr.y, gr.z, mp[i])) ++used;
      add += (unsigned long long)(gr.z - gr.y - used);
    }
    for (int o = 16; o; o >>= 1) add += __shfl_xor_sync(kFull, add, o);
    if (lane == 0) sm.count[threadIdx.x >> 5] += add;
  } else if (last && (!kShared || deferred)) {
    const int naut = kSym ? A.emit1.naut : 1;
    if (lane == 0) sm.count[threadIdx.x >> 5] += (unsigned long long)nok * naut;
    if (kRows) {
      unsigned long long at = 0;
      if (lane == 0) at = atomicAdd(&A.ctl->rows, (unsigned long long)nok * naut);
      at = __shfl_sync(kFull, at, 0);
      for (int e = lane; e < nok; e += 32) {
        const int2 sc = buf[e];
        const int32_t *mp = lv_state(A, p, (int64_t)(slice_first + (uint32_t)sc.x));
        const unsigned long long r = at + (unsigned long long)e * naut;
        if (kSym && naut > 1) lv_write_images(A.emit1, A.aut, A.rows, r, A.cap, mp, p, sc.y);
        else if (r < A.cap) lv_write_row(A.emit1, A.rows + r * A.emit1.k, mp, p, sc.y, deferred);
      }
    }
  } else {
    unsigned long long at = 0;
    if (lane == 0) at = atomicAdd(&A.ctl->next_n[p + 1], (unsigned long long)nok);
    at = __shfl_sync(kFull, at, 0) - sm.made;
    for (int e = lane; e < nok; e += 32) {
      const int2 sc = buf[e];
      const int64_t s = (int64_t)(slice_first + (uint32_t)sc.x);
      const int32_t *mp = lv_state(A, p, s);
      int32_t *dst = const_cast<int32_t *>(lv_state(A, p + 1, (int64_t)(at + e)));
      if (p <= 3) {
        int4 v = make_int4(mp[0], mp[1], 0, 0);
        if (kShared && p == 2) v.y = (int32_t)s;  // the group, in the place of position 1's image
        if (p == 3) v.z = mp[2];
        if (p == 2) v.z = sc.y; else v.w = sc.y;
        *reinterpret_cast<int4 *>(dst) = v;
      } else {
        for (int i = 0; i < p; ++i) dst[i] = mp[i];
        dst[p] = sc.y;
      }
    }
  }
  __syncwarp();
}

// The group that chunk x of the level lies in: the last one whose first chunk
// is at or before x.  Returns its number in the slice; *start is that first
// chunk.  `gi` is the group of the chunk before x, in the block's groups that
// begin at chunk `b0` and end at group `b1` (b1 = 0: none): mostly x lies
// in one of the 32 groups after it, which takes one load; otherwise the block
// is searched for in shared memory and the group in two loads.
__device__ __forceinline__ uint32_t lv_locate(const LvArgs &A, const LvShared &sm, int p, unsigned long long x,
                                              uint32_t ngroups, uint32_t per_groups, int lane, uint32_t gi,
                                              unsigned long long &b0, uint32_t &b1, unsigned long long *start) {
  const unsigned long long *up = A.upre[p];
  if (b1) {
    const uint32_t i = gi + 1 + lane;
    const unsigned long long u = i < b1 ? up[i] : ~0ull;
    const uint32_t le = __ballot_sync(kFull, u <= x - b0);
    // the last of them starts at or before x: it is the group unless all 32 do or the block ends there
    if (le && le != kFull && gi + 1 + __popc(le) < b1) {
      const int at = 31 - __clz(le);
      *start = b0 + __shfl_sync(kFull, u, at);
      return gi + 1 + at;
    }
  }
  int lo = 0, hi = (int)gridDim.x - 1;  // the last block whose first chunk is <= x
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (sm.first[mid] <= x) lo = mid; else hi = mid - 1;
  }
  b0 = sm.first[lo];
  uint32_t a = (uint32_t)lo * per_groups, n = min(per_groups, ngroups - a);  // groups [a, a + n)
  b1 = a + n;
  while (n > 1) {
    const uint32_t step = (n + 31) >> 5;
    const uint32_t i = (uint32_t)lane * step;
    const bool le = i < n && up[a + i] <= x - b0;
    const uint32_t at = (31 - __clz(__ballot_sync(kFull, le))) * step;  // lane 0 always holds
    a += at;
    n = min(step, n - at);
  }
  *start = b0 + up[a];
  return a;
}

// The expansion of the level's chunks [sm.begin, sm.begin + sm.take) by this
// warp: run `run` of sm.nrun, then runs claimed from the level's counter.
// Returns the number of chunks it took.
template <bool kRows, bool kBatch, bool kShared, bool kSym>
__device__ __forceinline__ uint32_t lv_expand(const LvArgs &A, LvShared &sm, int p, unsigned long long first,
                                              unsigned long long cnt, int g, uint32_t run) {
  Bytes none;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t lt = lanemask_lt();
  int4 *rec = sm.rec[warp];
  int2 *buf = sm.buf[warp];
  const int64_t chunks = (int64_t)((cnt + 31) >> 5), per = (chunks + gridDim.x - 1) / gridDim.x;
  const uint32_t per_groups = (uint32_t)(per * (32 / g)), ngroups = (uint32_t)(chunks * (32 / g));
  uint32_t gi = 0, b1 = 0;
  unsigned long long b0 = 0;
  const bool deferred = kShared && p == A.kmax;
  const int32_t *states = A.base[p] + first * A.stride[p];
  int nbuf = 0;
  uint32_t look = 0;
  while (run < sm.nrun) {
    unsigned long long x = sm.begin + (unsigned long long)run * sm.run_len;
    uint32_t left = (uint32_t)min((unsigned long long)sm.run_len, sm.take - (unsigned long long)run * sm.run_len);
    // the next run, claimed early so that its number is there when this one is done
    if (lane == 0) run = atomicAdd(sm.claim, 1u);
    b1 = 0;
    while (left) {
      unsigned long long start;
      gi = lv_locate(A, sm, p, x, ngroups, per_groups, lane, gi, b0, b1, &start);
      // the group's states that have candidates, in order, to shared memory
      const unsigned long long i = (unsigned long long)gi * g + lane;
      int4 r = make_int4(0, 0, 0, 0);
      if (lane < g && i < cnt) r = A.rng[p][i];
      const uint32_t have = __ballot_sync(kFull, r.y > 0);
      uint32_t incl = (uint32_t)r.y;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += y;
      }
      const uint32_t total = __shfl_sync(kFull, incl, 31);
      const uint32_t excl = r.y > 0 ? incl - (uint32_t)r.y : 0xffffffffu;
      if (r.y > 0) rec[__popc(have & lt)] = make_int4((int32_t)((uint32_t)r.x - excl), r.z, (int32_t)i, r.w);
      __syncwarp();
      uint32_t pos0 = (uint32_t)(x - start) << 5;
      if (x - start >= ((unsigned long long)total + 31) >> 5) {
        // cannot happen (the ranges phase counted the same chunks); never spin
        if (lane == 0) atomicCAS(&A.ctl->status, 0, kStatQueue);
        return look;
      }
      const uint32_t n = min(left, ((total - 1) >> 5) + 1 - (pos0 >> 5));  // chunks of this group
      left -= n;
      x += n;
      for (uint32_t c0 = 0; c0 < n; ++c0, pos0 += 32) {
        if ((++look & 31u) == 0) {
          int stop = 0;
          if (lane == 0) {
            if (*(volatile int32_t *)&A.ctl->status != 0) stop = 1;
            else if (globaltimer_ns() > sm.deadline) {
              atomicCAS(&A.ctl->status, 0, kStatBudget);
              stop = 1;
            }
          }
          if (__shfl_sync(kFull, stop, 0)) return look;
        }
        // the owner of position pos0 + lane: states that start at or before pos0, then the starts inside the chunk
        const uint32_t rel = excl - pos0;
        const uint32_t starts = __reduce_or_sync(kFull, r.y > 0 && excl > pos0 && rel < 32 ? 1u << rel : 0u);
        const int before = __popc(__ballot_sync(kFull, excl <= pos0 && r.y > 0)) - 1;
        const int ow = before + __popc(starts & (lt | (1u << lane)));
        bool ok = false;
        int32_t c = 0, s = 0;
        if (total - pos0 > (uint32_t)lane) {
          const int4 o = rec[ow];
          s = o.z;
          const uint32_t at = (uint32_t)o.x + pos0 + lane;
          const int list = o.y >> 8;
          if (kShared && list == 2)
            c = __ldg(&A.sorted_seeds[at].y);
          else
            c = __ldg((list ? A.G.gin_adj : A.G.gout_adj) + HM_AT(A.G, at, A.G.m, kChkList));
          if (deferred) {
            ok = true;
          } else {
            const LevelPlan &L = kBatch ? A.levels[(int64_t)o.w * A.kmax + p] : A.level1[p];
            ok = lv_first_checks<kShared, kSym>(A, L, states + (uint64_t)(uint32_t)s * (uint32_t)A.stride[p], p,
                                                o.y & 0xff, c, none);
          }
        }
        const uint32_t bal = __ballot_sync(kFull, ok);
        if (ok) buf[nbuf + __popc(bal & lt)] = make_int2(s, c);
        nbuf += __popc(bal);
        __syncwarp();
        if (nbuf >= kLvDrain) {
          lv_drain<kRows, kBatch, kShared, kSym>(A, sm, p, first, buf, nbuf, lane);
          nbuf = 0;
        }
      }
      __syncwarp();  // every lane is done with rec
    }
    run = gridDim.x * kLvWarps + __shfl_sync(kFull, run, 0);
  }
  if (nbuf) lv_drain<kRows, kBatch, kShared, kSym>(A, sm, p, first, buf, nbuf, lane);
  return look;
}

template <bool kRows, bool kBatch, bool kShared, bool kSym>
__global__ void __launch_bounds__(kLvThreads, kLvMinBlocks) k_levels(const __grid_constant__ LvArgs A) {
  extern __shared__ __align__(16) unsigned char s_raw[];
  LvShared &sm = *reinterpret_cast<LvShared *>(s_raw);
  const unsigned long long warps = (unsigned long long)gridDim.x * kLvWarps;
  const uint32_t me = blockIdx.x * kLvWarps + (threadIdx.x >> 5);
  const int last = kShared && (kRows || A.ndefer) ? A.kmax : A.kmax - 1;  // the deepest level
  const unsigned long long nseeds = *A.nseeds;
  if ((threadIdx.x & 31) == 0) sm.count[threadIdx.x >> 5] = 0;
  if (threadIdx.x == 0) sm.deadline = globaltimer_ns() + A.budget_ns;
  __syncthreads();
  unsigned long long my_chunks = 0, cursor = 0;
  unsigned int target = 0, turn = 0;
  // the levels being worked on: states [first, first + n) and chunks [done, total)
  unsigned long long first = 0;
  unsigned long long n[kMaxK + 2], done[kMaxK + 2], total[kMaxK + 2];
  unsigned long long made[kMaxK + 2];  // states each level's counter had counted when last read
  for (int i = 0; i < kMaxK + 2; ++i) made[i] = 0;
  int p = 1;
  bool ok = true;
  while (ok) {
    if (p == 1) {  // the next slice of depth-2 states
      if (cursor >= nseeds) break;
      p = 2;
      first = cursor;
      n[2] = min((unsigned long long)A.slice, nseeds - cursor);
      cursor += n[2];
    } else if (done[p] < total[p]) {
      // expand as many chunks as the next level can hold survivors of
      const unsigned long long left = total[p] - done[p];
      const unsigned long long take = p < last ? min(left, (unsigned long long)(A.fcap >> 5)) : left;
      // runs of chunks: the first is the warp's own, the rest are claimed, so that
      // warps with cheap chunks (lists in cache) take more of them
      if (threadIdx.x == 0) {
        const unsigned long long run = max(take / (warps * 8), 1ull);
        sm.begin = done[p];
        sm.take = take;
        sm.run_len = (uint32_t)min(run, 1ull << 31);
        sm.nrun = (uint32_t)((take + sm.run_len - 1) / sm.run_len);
        sm.made = made[p + 1];
        sm.claim = &A.ctl->claim[turn % 3];
        if (blockIdx.x == 0) A.ctl->claim[(turn + 1) % 3] = 0;  // read two expansions ago
      }
      ++turn;
      __syncthreads();
      my_chunks += lv_expand<kRows, kBatch, kShared, kSym>(A, sm, p, p == 2 ? first : 0, n[p],
                                                           lv_group_size(n[p], warps, A.G.maxdeg), me);
      done[p] += take;
      if (p == last && done[p] == total[p]) {  // nothing below: up again, past levels that are done too
        while (p > 1 && done[p] == total[p]) --p;
        if (p == 1 && cursor >= nseeds) break;
        // the next step overwrites buffers that other warps may still read
        target += gridDim.x;
        ok = lv_barrier(A, sm, target);
        if (p > 1) goto reload;
        continue;
      }
      target += gridDim.x;
      if (!(ok = lv_barrier(A, sm, target))) break;
      if (p == last) continue;
      const unsigned long long now = *(volatile unsigned long long *)&A.ctl->next_n[p + 1];
      const unsigned long long fresh = now - made[p + 1];
      made[p + 1] = now;
      if (fresh == 0) {
        // another block may not have read the counter yet that the next expansion adds to
        target += gridDim.x;
        if (!(ok = lv_barrier(A, sm, target))) break;
        if (done[p] < total[p]) continue;
        while (p > 1 && done[p] == total[p]) --p;
        if (p > 1) goto reload;
        continue;
      }
      ++p;
      n[p] = fresh;
    } else {
      while (p > 1 && done[p] == total[p]) --p;
      if (p > 1) goto reload;
      continue;
    }
    // the ranges of the new states
    lv_ranges<kBatch, kShared, kRows, kSym>(A, sm, p, p == 2 ? first : 0, n[p], lv_group_size(n[p], warps, A.G.maxdeg));
    target += gridDim.x;
    if (!(ok = lv_barrier(A, sm, target))) break;
    done[p] = 0;
  reload: {
      // the first chunk of each block's groups at this level
      unsigned long long all = 0, run = 0;
      for (int b = 0; b < (int)gridDim.x; b += kLvThreads) {
        const int i = b + threadIdx.x;
        const unsigned long long v = i < (int)gridDim.x ? __ldcg(A.bsum[p] + i) : 0;
        const unsigned long long at = lv_block_scan(v, sm, &all);
        if (i < (int)gridDim.x) sm.first[i] = run + at;
        run += all;
      }
      total[p] = run;
      __syncthreads();
    }
  }
  if ((threadIdx.x & 31) == 0) {
    const unsigned long long count = sm.count[threadIdx.x >> 5];
    if (count) atomicAdd(&A.ctl->count, count);
    if (my_chunks) atomicAdd(&A.ctl->chunks, my_chunks);
  }
}

using LvKernel = void (*)(LvArgs);

LvKernel lv_kernel(bool rows, bool batch, bool shared, bool sym) {
  if (batch) {
    if (sym) return rows ? k_levels<true, true, false, true> : k_levels<false, true, false, true>;
    return rows ? k_levels<true, true, false, false> : k_levels<false, true, false, false>;
  }
  if (shared) return rows ? k_levels<true, false, true, false> : k_levels<false, false, true, false>;
  if (sym) return rows ? k_levels<true, false, false, true> : k_levels<false, false, false, true>;
  return rows ? k_levels<true, false, false, false> : k_levels<false, false, false, false>;
}

// Resident blocks of a variant (0: the device cannot run it).
int lv_grid(LvKernel f, int slot) {
  static std::atomic<int> cache[16];
  int v = cache[slot].load(std::memory_order_relaxed);
  if (!v) {
    int per_sm = 0, coop = 0, dev = 0;
    cudaGetDevice(&dev);
    if (cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess || !coop ||
        cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(LvShared)) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, f, kLvThreads, sizeof(LvShared)) != cudaSuccess)
      per_sm = 0;
    (void)cudaGetLastError();
    v = per_sm > 0 ? std::min(per_sm * num_sms(), kLvMaxGrid) : -1;
    cache[slot].store(v, std::memory_order_relaxed);
  }
  return std::max(v, 0);
}

int16_t lv_class(const hm_graph *g, int32_t alab, int32_t vlab) {
  const int64_t a = (int64_t)alab - g->al0, v = (int64_t)vlab - g->vl0;
  if (a < 0 || a >= g->nal || v < 0 || v >= g->nvl) return -1;
  return (int16_t)(a * g->nvl + v);
}

void lv_level(const hm_graph *g, const Plan &P, int p, LevelPlan &L) {
  std::memset(&L, 0, sizeof(L));
  if (p >= P.k) return;
  L.npos = (int16_t)P.npos[p];
  L.ncons = (int16_t)P.ncons[p];
  L.last = p == P.k - 1;
  L.root = P.root_pos == p;
  L.dout = P.dout[p];
  L.din = P.din[p];
  L.sym_gt = P.sym_gt[p];
  L.sym_lt = P.sym_lt[p];
  for (int j = 0; j < P.ncons[p]; ++j) {
    const Cons cs = P.cons[p][j];
    const ArcKey l = j < P.npos[p] ? labelled_key(ArcKey{0, 0}, cs.lab) : ArcKey{0, 0};
    L.cons[j] = LvCons{cs.q, cs.kind, j < P.npos[p] ? lv_class(g, cs.lab, P.vlab[p]) : (int16_t)0, cs.lab, l.a, l.b};
  }
  // arcs to later positions: one or two are found missing by the next ranges phase anyway
  L.need_deg = !L.last && P.dout[p] + P.din[p] - P.npos[p] >= 2;
}

void lv_emit(const Plan &P, EmitPlan &E, std::vector<int8_t> &aut) {
  std::memset(&E, 0, sizeof(E));
  E.k = P.k;
  E.naut = std::max(P.naut, 1);
  for (int i = 0; i < P.k; ++i) E.orig[i] = P.orig[i];
  E.aut = (int32_t)aut.size();
  if (P.naut > 1)
    for (int s = 0; s < P.naut; ++s) aut.insert(aut.end(), P.aut[s], P.aut[s] + kMaxK);
}

}  // namespace

hm_status levels_run(const LvLaunch &L, cudaStream_t s, bool *ran, int *grid_out, int *threads_out) {
  *ran = false;
  const hm_graph *g = L.g;
  if (!g->ncls || filter_min() != 1) return HM_OK;
  const bool batch = L.npat > 0, shared = L.groups != nullptr;
  bool sym = false;
  int kmax = 0;
  if (batch) {
    for (int32_t i = 0; i < L.npat; ++i) {
      sym |= L.plans[i].naut > 1;
      kmax = std::max({kmax, (int)L.plans[i].k, 3});
    }
  } else {
    sym = L.plan->naut > 1;
    kmax = L.plan->k;
  }
  const LvKernel f = lv_kernel(L.want_rows, batch, shared, sym);
  int grid = lv_grid(f, (L.want_rows ? 8 : 0) + (batch ? 4 : 0) + (shared ? 2 : 0) + (sym ? 1 : 0));
  if (grid <= 0) return HM_OK;
  // a small graph's levels do not need every block, and barriers cost less with fewer
  grid = (int)std::max<int64_t>(1, std::min<int64_t>(grid, (g->m + 255) / 256));

  const int64_t warps = (int64_t)grid * kLvWarps;
  const int top = shared ? kmax : kmax - 1;  // deepest level with states
  LvArgs A{};
  // a quarter of the workspace for the depth-2 states' ranges, the rest for the deeper levels
  A.slice = std::max<int64_t>(1, std::min<int64_t>({L.max_seeds, kLvSeedSlice, (int64_t)kLvMaxGroups * 32 * grid,
                                                    (int64_t)(L.workspace / 4 / 32)}));
  // bytes per state of all levels; the buffers are sized by the workspace and the graph
  int64_t per_state = 0;
  for (int p = 3; p <= top; ++p) per_state += 16 + 4 * ((p + (batch ? 1 : 0) + 3) / 4 * 4) + 1;
  int64_t fcap = per_state ? (int64_t)(L.workspace / 4 * 3 / (uint64_t)per_state) : 0;
  fcap = std::min<int64_t>({fcap, std::max<int64_t>(8 * g->m, 1 << 16), (int64_t)kLvMaxGroups * 32 * grid,
                            (int64_t)1 << 24});
  fcap = std::max<int64_t>(fcap & ~int64_t(31), 4096);
  A.fcap = fcap;
  auto round = [](size_t b) { return (b + 255) / 256 * 256; };
  auto groups_of = [&](int64_t states) { return (size_t)(states / 32 + 2 * warps + 64); };
  size_t bytes = 0, at_rng[kMaxK + 2] = {}, at_up[kMaxK + 2] = {}, at_bs[kMaxK + 2] = {}, at_st[kMaxK + 2] = {};
  for (int p = 2; p <= top; ++p) {
    const int64_t states = p == 2 ? A.slice : fcap;
    A.stride[p] = p == 2 ? (shared ? 4 : 2) : (p + (batch ? 1 : 0) + 3) / 4 * 4;
    at_rng[p] = bytes;
    bytes += round(sizeof(int4) * (size_t)states);
    at_up[p] = bytes;
    bytes += round(8 * groups_of(states));
    at_bs[p] = bytes;
    bytes += round(8 * (size_t)grid);
    at_st[p] = bytes;
    if (p > 2) bytes += round(4 * (size_t)A.stride[p] * (size_t)states);
  }
  // batch: level and emission plans; symmetric patterns: automorphisms
  std::vector<int8_t> aut;
  std::vector<LevelPlan> levels;
  std::vector<EmitPlan> emit;
  if (batch) {
    levels.resize((size_t)L.npat * kmax);
    emit.resize(L.npat);
    for (int32_t i = 0; i < L.npat; ++i) {
      for (int p = 1; p < kmax; ++p) lv_level(g, L.plans[i], p, levels[(size_t)i * kmax + p]);
      levels[(size_t)i * kmax + 2].done = L.plans[i].k == 2;
      lv_emit(L.plans[i], emit[i], aut);
    }
  } else {
    for (int p = 1; p < kmax; ++p) lv_level(g, *L.plan, p, A.level1[p]);
    lv_emit(*L.plan, A.emit1, aut);
    A.ndefer = shared ? L.plan->ndefer : 0;
    for (int j = 0; j < A.ndefer; ++j) A.defer[j] = L.plan->defer[j];
  }
  const size_t at_tab = bytes;
  const size_t tab_levels = round(sizeof(LevelPlan) * levels.size()), tab_emit = round(sizeof(EmitPlan) * emit.size());
  bytes += tab_levels + tab_emit + round(aut.size());

  unsigned char *ws = nullptr;
  HM_CUDA_TRY(cudaMallocAsync((void **)&ws, std::max<size_t>(bytes, 256), s));
  for (int p = 2; p <= top; ++p) {
    A.rng[p] = reinterpret_cast<int4 *>(ws + at_rng[p]);
    A.upre[p] = reinterpret_cast<unsigned long long *>(ws + at_up[p]);
    A.bsum[p] = reinterpret_cast<unsigned long long *>(ws + at_bs[p]);
    A.base[p] = reinterpret_cast<const int32_t *>(ws + at_st[p]);
  }
  A.base[2] = shared ? reinterpret_cast<const int32_t *>(L.groups) : reinterpret_cast<const int32_t *>(L.seeds);
  cudaError_t e = cudaSuccess;
  auto up = [&](size_t at, const void *src, size_t n) {
    if (n && e == cudaSuccess) e = cudaMemcpyAsync(ws + at, src, n, cudaMemcpyHostToDevice, s);
  };
  up(at_tab, levels.data(), sizeof(LevelPlan) * levels.size());
  up(at_tab + tab_levels, emit.data(), sizeof(EmitPlan) * emit.size());
  up(at_tab + tab_levels + tab_emit, aut.data(), aut.size());
  A.levels = reinterpret_cast<const LevelPlan *>(ws + at_tab);
  A.emit = reinterpret_cast<const EmitPlan *>(ws + at_tab + tab_levels);
  A.aut = reinterpret_cast<const int8_t *>(ws + at_tab + tab_levels + tab_emit);
  A.G = g->dev();
  A.ctl = L.ctl;
  A.nseeds = L.nseeds;
  A.groups = L.groups;
  A.sorted_seeds = L.sorted_seeds;
  A.root_mask = L.root_mask;
  A.budget_ns = budget_ms() * 1000000ull;
  A.rows = L.rows;
  A.cap = L.cap;
  A.seed_pid = L.seed_pid;
  A.counts = L.counts;
  A.row_off = L.row_off;
  A.row_cap = L.row_cap;
  A.row_cursor = L.row_cursor;
  A.kmax = kmax;
  if (e == cudaSuccess) {
    void *args[] = {&A};
    const cudaError_t le = cudaLaunchCooperativeKernel((const void *)f, dim3(grid), dim3(kLvThreads), args,
                                                       sizeof(LvShared), s);
    if (le == cudaSuccess) *ran = true;
    else (void)cudaGetLastError();  // not launched: the caller searches depth first
  }
  cudaFreeAsync(ws, s);
  if (e != cudaSuccess) {
    (void)cudaGetLastError();
    return HM_ERR_CUDA;
  }
  if (grid_out) *grid_out = grid;
  if (threads_out) *threads_out = kLvThreads;
  return HM_OK;
}

}  // namespace hm
