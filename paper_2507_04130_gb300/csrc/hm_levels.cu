// hm_levels.cu -- a whole match, level by level, in one persistent launch.
//
// The states of a level (p mapped positions each) are extended together: every
// candidate of every state is one lane's work, so the lanes are full and all
// warps finish at the same time, whatever the distribution of the degrees.
// (The depth-first search with one warp per state, k_extend, kept 2 to 30 % of
// the warps busy wherever a few hubs own the work: a connectome query of 121 M
// leaf candidates took 17.4 ms, of which 90 % was waiting for the last warps.)
//
// The first level is the vertices with position 0's label and a neighbour that
// position 1 could take (listed per class when the graph is loaded); position 1
// is extended like every other, along the seeding arc's label group.  That takes
// the place of the scan over all arcs (the loop over E2 of the HiPerMotif
// algorithm): only arcs with the seeding arc's three labels are read, 4 bytes
// each and in source order, instead of 12 bytes of every arc and two vertex
// records per candidate.
//
// Expanding a level: its states stand in groups of up to 32, and the groups'
// chunks of 32 candidates are numbered through.  Each warp takes runs of
// consecutive chunks, finds the group a run starts in, and reads 32 candidates
// at a time: the filter probes of the other positive conditions reject most;
// survivors wait in the warp's buffer until 64 are there, then the exact checks
// run on full warps.  What passes becomes a match, or a state of the next
// level: its anchors' label groups (dense group offsets: one lookup of two
// neighbouring words each), the shortest of which holds its candidates.  A
// state whose anchor has an empty group is dropped, and so is one whose last
// position has no other condition, if only its number is asked for: it is the
// group's length (where symmetry is broken, that of the part between two
// images).  Up to 64 states go to the next level with one addition, which
// reserves their groups and numbers their chunks.  A grid barrier ends the
// expansion.
// Memory is bounded: when the states of some warp do not fit the next level any
// more, all remember where they stand; the deeper levels are worked off, and
// then they go on (depth first over parts of levels).
//
// A pendant position 1 (Plan::defer1: no later position has an arc to it) is
// matched last, so the search over the others is shared by all its images.
//
// Bound by the latency of its lookups in L2 and HBM (list entry, then filter
// word, per candidate), which many independent warps hide.
#include <algorithm>
#include <cstring>
#include <mutex>
#include <vector>

#include "hm_levels.cuh"

namespace hm {
namespace {

constexpr int kLvThreads = 512;
constexpr int kLvWarps = kLvThreads / 32;
constexpr int kLvMinBlocks = 2;
constexpr uint32_t kFull = 0xffffffffu;
constexpr int kLvBuf = 96;        // survivors of a warp waiting for the exact checks
constexpr int kLvDrain = 64;      // checked when this many wait (a chunk adds at most 32)
constexpr int kLvChunkBits = 40;  // of a level's counter; the groups are above
constexpr unsigned long long kLvChunkMask = (1ull << kLvChunkBits) - 1;
constexpr int64_t kLvMaxGroups = 1 << 20;  // of a level (2^24 would fit the counter)
// A group's candidates are numbered in 32 bits while it is expanded, and 32 states
// on a hub of 2^27 arcs have 2^32: where the sum reaches this, every state
// becomes a group of its own (a list has less than 2^31 entries).
constexpr unsigned long long kLvGroupCands = 1ull << 31;

// A condition of a level: Cons with the class (arc label, vertex label) whose
// group of f(q) holds the candidates, -1 if the graph has no such label.
struct LvCons {
  int8_t q, kind;
  int16_t cls;
  int32_t lab;
  uint64_t la;  // the label's part of the arc filter's hash
};

// What a candidate for one position must satisfy.
struct LevelPlan {
  int16_t npos, ncons;    // positive conditions first
  int8_t last;            // the position completes a match
  int8_t need_deg;        // test the degrees: at least two pattern arcs lead to positions after the next
  int8_t root;            // the root mask applies to this position
  int8_t closed;          // the last position has one condition (order constraints apart), and only the number of its images is wanted
  int8_t final;           // level 1 of a plan with a deferred position 1: the level that matches it, else 0
  int32_t dout, din;
  uint32_t sym_gt, sym_lt;
  int32_t cons;           // its first condition in the table
};

// How a pattern's matches are written.
struct EmitPlan {
  int32_t k, naut;
  int32_t aut;            // first byte of its automorphisms in the table, kMaxK each
  int32_t orig[kMaxK];
};

// A group of states: its first chunk and its number of states (up to 32, with
// fewer than kLvGroupCands candidates in all).  Its states are those numbered
// from 32 times the group's number on.
struct LvGroup {
  unsigned long long start;
  uint32_t n, pad;
};

// Where a warp goes on whose states did not fit the next level.
struct LvPause {
  unsigned long long x;     // next chunk
  uint32_t left, run;       // chunks left of the run; the claimed run after it
  int32_t on, nwait, nbuf, pad;  // paused at all; states waiting for room, survivors waiting for their checks
  int2 buf[kLvBuf];         // both, {parent, candidate}
};

struct LvArgs {
  DevGraph G;
  LvCtl *ctl;
  // each level: states (their images, stride[p] words each), their candidates {first, number,
  // driving condition | list << 6 | pattern << 7, 0}, groups
  int32_t *base[kMaxK + 1];
  int4 *rng[kMaxK + 1];
  LvGroup *grp[kMaxK + 1];
  LvPause *pause[kMaxK + 1];
  int32_t stride[kMaxK + 1];
  uint32_t gcap[kMaxK + 1];        // groups each level holds
  uint32_t fill_warps;             // warps that fill the first level
  unsigned long long slice;        // vertices of a slice of the first level
  unsigned long long nvert;        // vertices the first level starts from
  const int32_t *vert;
  // batch: vertices are numbered pattern after pattern (vert_n), vertex s of pattern pid is vert_at[pid][s]
  const unsigned long long *vert_n;
  const int32_t *const *vert_at;
  int32_t npat;
  int32_t dout0, din0, root0;      // position 0 of a single pattern: degrees, root mask
  const int2 *deg0;                // batch: {out, in}
  const uint8_t *root_mask;
  unsigned long long budget_ns;
  int32_t *rows;
  unsigned long long cap;
  const LevelPlan *levels;         // batch: [pattern][kmax]
  const LvCons *cons;              // batch: the levels' conditions
  const EmitPlan *emit;
  const int8_t *aut;
  unsigned long long *counts;
  const unsigned long long *row_off, *row_cap;
  unsigned long long *row_cursor;
  int32_t kmax;                    // levels 1 .. kmax - 1
  EmitPlan emit1;
  LevelPlan level1[kMaxK];
  LvCons cons1[kMaxK * (kMaxK - 1)];  // two for every pair of positions at most
};

// Condition j of the level whose plan is L.
template <bool kBatch>
__device__ __forceinline__ const LvCons &lv_cons(const LvArgs &A, const LevelPlan &L, int j) {
  return kBatch ? A.cons[L.cons + j] : A.cons1[L.cons + j];
}

struct LvShared {
  // the group's states: {first candidate - first position, flags, partial hash of the first probe},
  // the first four images, the region of that probe, and in a batch the pattern
  int4 rec[kLvWarps][32];
  Region reg[kLvWarps][32];
  int4 img[kLvWarps][32];
  int32_t pid[kLvWarps][32];
  int2 buf[kLvWarps][kLvBuf];      // {state, candidate}
  int4 fresh[kLvWarps][kLvDrain];  // states of the next level: {first candidate, number, what, parent}
  // values all warps share, and each warp's matches, kept out of the registers of the expansion
  unsigned long long deadline, total;
  unsigned long long count[kLvWarps];
  uint32_t injected[kLvWarps];
  unsigned long long *made;        // the next level's counter
  uint32_t run_len, nrun, ngroup;
  unsigned int *claim, *paused;
  int ok;
};

// The time limit is looked at here too, so at least once per phase: a phase may
// give each warp fewer chunks than lv_expand takes between two looks, and a search
// have any number of such phases.  It also bounds the wait.
__device__ __forceinline__ bool lv_barrier(const LvArgs &A, LvShared &sm, unsigned int target) {
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(&A.ctl->bar, 1u);
    int ok = 1;
    for (;;) {
      if (globaltimer_ns() > sm.deadline) {
        atomicCAS(&A.ctl->status, 0, kStatBudget);
        break;
      }
      if (*(volatile unsigned int *)&A.ctl->bar >= target) break;
      if (*(volatile int32_t *)&A.ctl->status != 0) break;
      __nanosleep(32);
    }
    __threadfence();
    if (*(volatile int32_t *)&A.ctl->status != 0) ok = 0;
    sm.ok = ok;
  }
  __syncthreads();
  return sm.ok != 0;
}

// A state's first four images, in registers: most patterns' checks read no
// more of it.  Unmapped positions are -1.
__device__ __forceinline__ int4 lv_images(const int32_t *mp, int p) {
  if (p == 1) return make_int4(mp[0], -1, -1, -1);
  if (p == 2) {
    const int2 v = *reinterpret_cast<const int2 *>(mp);
    return make_int4(v.x, v.y, -1, -1);
  }
  int4 m = *reinterpret_cast<const int4 *>(mp);
  if (p == 3) m.w = -1;
  return m;
}

__device__ __forceinline__ int32_t lv_image(const int4 &m, const int32_t *mp, int q) {
  if (q >= 4) return mp[q];
  const int32_t a = q & 1 ? m.y : m.x, b = q & 1 ? m.w : m.z;
  return q & 2 ? b : a;
}

// What is packed into a range's third word.
__device__ __forceinline__ int lv_drive(int32_t what) { return what & 63; }
__device__ __forceinline__ int lv_list(int32_t what) { return what >> 6 & 1; }
__device__ __forceinline__ int32_t lv_pid(int32_t what) { return what >> 7; }

// The group of f(q) = v that condition cs names.
__device__ __forceinline__ int2 lv_group(const LvArgs &A, const LvCons &cs, int32_t v) {
  const int32_t *ofs = cs.kind == kOut ? A.G.gofs_out : A.G.gofs_in;
  const int64_t at = (int64_t)v * A.G.ncls + cs.cls;
  const int32_t a = __ldg(ofs + HM_AT(A.G, at, (int64_t)A.G.n * A.G.ncls, kChkGroup));
  return make_int2(a, __ldg(ofs + at + 1) - a);
}

// Has u a neighbour that the deferred position 1 (level plan Z) may take?  The
// search over the other positions would be for nothing.  With arcs in both
// directions, the filter is asked if the shorter list has at most 8 entries.
template <bool kBatch>
__device__ __forceinline__ bool lv_has_final(const LvArgs &A, const LevelPlan &Z, int32_t u) {
  const LvCons &c0 = lv_cons<kBatch>(A, Z, 0), &c1 = lv_cons<kBatch>(A, Z, 1);
  if (c0.cls < 0) return false;
  const int2 r = lv_group(A, c0, u);
  if (Z.npos < 2 || r.y == 0) return r.y > 0;
  if (c1.cls < 0) return false;
  const int2 r1 = lv_group(A, c1, u);
  const bool second = r1.y < r.y;
  const int2 w = second ? r1 : r;
  if (w.y > 8) return true;
  const LvCons &cs = second ? c1 : c0, &other = second ? c0 : c1;
  const int32_t *list = cs.kind == kOut ? A.G.gout_adj : A.G.gin_adj;
  Bytes none;
#pragma unroll 1
  for (int i = 0; i < w.y; ++i) {
    const int32_t c = __ldg(list + HM_AT(A.G, (int64_t)w.x + i, A.G.m, kChkList));
    if (arc_maybe_l<false>(A.G, other.kind == kOut ? u : c, other.kind == kOut ? c : u, other.lab, none)) return true;
  }
  return false;
}

// The first of the sorted entries [lo, lo + len) of a list that is at least x (lo + len: none).
__device__ __forceinline__ int32_t lv_lower(const DevGraph &G, const int32_t *list, int32_t lo, int32_t len, int32_t x) {
  while (len > 0) {
    const int32_t half = len >> 1;
    if (__ldg(list + HM_AT(G, (int64_t)lo + half, G.m, kChkList)) < x) {
      lo += half + 1;
      len -= half + 1;
    } else {
      len = half;
    }
  }
  return lo;
}

// The candidates of a state of level p: of the parent at mp (images m) with
// candidate c at position p - 1.  kClosed: this call only counts, and where the
// level is closed the matches are added to `found` instead.  The fourth word is
// not set.
template <bool kBatch, bool kClosed, bool kSym>
__device__ __forceinline__ int4 lv_range(const LvArgs &A, int p, const int4 &m, const int32_t *mp, int32_t c,
                                         int32_t pid, unsigned long long &found) {
  const LevelPlan &L = kBatch ? A.levels[(int64_t)pid * A.kmax + p] : A.level1[p];
  const int4 dead = make_int4(0, 0, 0, 0);
  if (p == 1) {
    // the vertex validator (Alg. 2; the label is the list's) and a root mask on position 0
    if (A.root0 && !A.root_mask[c]) return dead;
    const int2 need = kBatch ? A.deg0[pid] : make_int2(A.dout0, A.din0);
    const int4 vi = __ldg(&A.G.vi[HM_AT(A.G, c, A.G.n, kChkVertex)]);
    if (vi.y < need.x || vi.z < need.y) return dead;
    if (L.final && !lv_has_final<kBatch>(A, kBatch ? A.levels[(int64_t)pid * A.kmax + L.final] : A.level1[L.final],
                                         c))
      return dead;
  }
  int32_t best = INT32_MAX, lo = 0, what = 0;
  for (int j = 0; j < L.npos; ++j) {
    const LvCons cs = lv_cons<kBatch>(A, L, j);
    if (cs.cls < 0) return dead;
    const int2 r = lv_group(A, cs, cs.q == p - 1 ? c : lv_image(m, mp, cs.q));
    if (r.y < best) {
      best = r.y;
      lo = r.x;
      what = j | (cs.kind == kOut ? 0 : 1 << 6);
    }
  }
  if (kClosed && L.closed && best > 0) {
    // every entry of the group that the state does not use already
    const int32_t *list = lv_list(what) ? A.G.gin_adj : A.G.gout_adj;
    Bytes none;
    int used = 0;
    if (kSym && (L.sym_gt | L.sym_lt)) {
      // between the images that the order constraints name; groups are sorted.  (Read entry by
      // entry, six ordered leaves of a hub among 128 vertices took 15 ms in place of 42 depth first,
      // but ordered pairs on a million arcs 449 us in place of 403.)
      int32_t above = -1, below = INT32_MAX;
      for (int i = 0; i < p; ++i) {
        const int32_t x = i == p - 1 ? c : lv_image(m, mp, i);
        if (L.sym_gt >> i & 1u) above = max(above, x);
        if (L.sym_lt >> i & 1u) below = min(below, x);
      }
      const int32_t a = above < 0 ? lo : lv_lower(A.G, list, lo, best, above + 1);
      const int32_t z = below == INT32_MAX ? lo + best : lv_lower(A.G, list, a, lo + best - a, below);
      lo = a;
      best = max(z - a, 0);
    }
    for (int i = 0; i < p; ++i)
      if (search_g<false>(A.G, list, lo, best, i == p - 1 ? c : lv_image(m, mp, i), none) >= 0) ++used;
    found = (unsigned long long)(best - used);
    best = 0;
  }
  return make_int4(lo, best, what | pid << 7, 0);
}

// What the checks of a state's candidates have in common, in rec[].y: the list,
// whether there is a positive condition besides the driving one (its probe comes
// first), whether the candidate is the target of that arc, the driving
// condition, and the first condition after the probed one.
__device__ __forceinline__ int32_t lv_flags(int32_t list, bool probe, bool to, int32_t drive, int32_t next) {
  return list | (probe ? 2 : 0) | (to ? 4 : 0) | drive << 3 | next << 9;
}

// The cheap checks: candidate c of a state for position p.  o and m are the
// state's records, mp its images in memory (read beyond the fourth only).
template <bool kBatch, bool kSym>
__device__ __forceinline__ bool lv_first_checks(const LvArgs &A, const LevelPlan &L, const int4 &o, const int4 &m,
                                                const Region &g, const int32_t *mp, int p, int32_t c, Bytes &none) {
  if (m.x == c || m.y == c || m.z == c || m.w == c) return false;  // injective
  for (int i = 4; i < p; ++i)
    if (mp[i] == c) return false;
  if (L.root && !A.root_mask[c]) return false;
  if (kSym) {
    uint32_t g = L.sym_gt, l = L.sym_lt;
    while (g) {
      const int q = __ffs(g) - 1;
      g &= g - 1;
      if (c <= lv_image(m, mp, q)) return false;
    }
    while (l) {
      const int q = __ffs(l) - 1;
      l &= l - 1;
      if (c >= lv_image(m, mp, q)) return false;
    }
  }
  if (!(o.y & 2)) return true;
  const uint64_t part = (uint64_t)(uint32_t)o.w << 32 | (uint32_t)o.z;
  // the fixed endpoint's own words of the filter
  const ArcKey key{part + (o.y & 4 ? kHashV : kHashU) * (uint32_t)c};
  const uint2 w = __ldg((o.y & 4 ? A.G.rfilt_out : A.G.rfilt_in) +
                        HM_AT(A.G, (int64_t)g.base + filter_word(key, g.nword), A.G.rf_nword, kChkRegion));
  const uint2 b = filter_bits(key);
  if ((b.x & ~w.x) | (b.y & ~w.y)) return false;
  for (int j = o.y >> 9; j < L.npos; ++j) {
    if (j == (o.y >> 3 & 63)) continue;
    const LvCons cs = lv_cons<kBatch>(A, L, j);
    const int32_t f = lv_image(m, mp, cs.q);
    ArcKey k = pair_key(cs.kind == kOut ? f : c, cs.kind == kOut ? c : f);
    k.h += cs.la;
    if (!filter_has<false>(A.G, k, none)) return false;
  }
  return true;
}

// The exact checks of a candidate that passed the cheap ones.
template <bool kBatch>
__device__ __forceinline__ bool lv_exact_checks(const LvArgs &A, const LevelPlan &L, const int32_t *mp, int p, int drive,
                                                int32_t c, Bytes &none) {
  const int4 m = lv_images(mp, p);
  if (L.need_deg) {
    const int4 vi = __ldg(&A.G.vi[HM_AT(A.G, c, A.G.n, kChkVertex)]);
    if (vi.y < L.dout || vi.z < L.din) return false;
  }
  for (int j = 0; j < L.ncons; ++j) {
    if (j == drive) continue;
    const LvCons cs = lv_cons<kBatch>(A, L, j);
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

__device__ __forceinline__ void lv_write_row(const EmitPlan &E, int32_t *row, const int32_t *mp, int p, int32_t c) {
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

// Adds what a warp's lanes found in closed levels to the counts.
template <bool kBatch, bool kSym>
__device__ __forceinline__ void lv_add_found(const LvArgs &A, LvShared &sm, unsigned long long found, int32_t pid,
                                             int lane) {
  if (!__any_sync(kFull, found != 0)) return;
  if (kBatch) {
    if (kSym && found) found *= A.emit[pid].naut;
    // neighbouring states mostly belong to one pattern: one addition per warp then
    const int32_t p0 = __shfl_sync(kFull, pid, __ffs(__ballot_sync(kFull, found != 0)) - 1);
    const bool same = __all_sync(kFull, pid == p0 || !found);
    unsigned long long all = found;
    for (int o = 16; o; o >>= 1) all += __shfl_xor_sync(kFull, all, o);
    if (same ? lane == 0 : found != 0) atomicAdd(A.counts + (same ? p0 : pid), same ? all : found);
  } else {
    for (int o = 16; o; o >>= 1) found += __shfl_xor_sync(kFull, found, o);
    if (lane == 0) sm.count[threadIdx.x >> 5] += kSym ? found * A.emit1.naut : found;
  }
}

// The warp's n (at most 64) new states to level p: fresh[] holds their ranges and
// parents, buf[].y the candidates at position p - 1.  False: no room.
__device__ __noinline__ bool lv_append(const LvArgs &A, LvShared &sm, int p, const int4 *fresh, const int2 *buf,
                                          int n, int lane) {
  // chunks of the first and of the second group
  unsigned long long t0 = lane < n ? (uint32_t)fresh[lane].y : 0, t1 = lane + 32 < n ? (uint32_t)fresh[lane + 32].y : 0;
  for (int o = 16; o; o >>= 1) {
    t0 += __shfl_xor_sync(kFull, t0, o);
    t1 += __shfl_xor_sync(kFull, t1, o);
  }
  const bool apart = t0 >= kLvGroupCands || t1 >= kLvGroupCands;  // the same in every lane
  int ng = n > 32 ? 2 : 1;
  unsigned long long c0 = 0, c1 = 0;  // apart: chunks before this lane's states
  if (apart) {
    const unsigned long long own0 = lane < n ? ((uint32_t)fresh[lane].y + 31u) >> 5 : 0u;
    const unsigned long long own1 = lane + 32 < n ? ((uint32_t)fresh[lane + 32].y + 31u) >> 5 : 0u;
    c0 = own0;
    c1 = own1;
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long a = __shfl_up_sync(kFull, c0, o), b = __shfl_up_sync(kFull, c1, o);
      if (lane >= o) {
        c0 += a;
        c1 += b;
      }
    }
    t0 = __shfl_sync(kFull, c0, 31);
    t1 = __shfl_sync(kFull, c1, 31);
    c0 -= own0;
    c1 += t0 - own1;
    ng = n;
  } else {
    t0 = (t0 + 31) >> 5;
    t1 = (t1 + 31) >> 5;
  }
  const unsigned long long add = ((unsigned long long)ng << kLvChunkBits) + t0 + t1;
  unsigned long long at = 0;
  int fits = 0;
  if (lane == 0) {
    at = atomicAdd(sm.made, add);
    fits = (at >> kLvChunkBits) + ng <= A.gcap[p];
    // taken back, so the groups that were given stay without gaps: whoever adds
    // in between sees an even fuller level and takes back too
    if (!fits) atomicAdd(sm.made, 0ull - add);
  }
  if (!__shfl_sync(kFull, fits, 0)) return false;
  at = __shfl_sync(kFull, at, 0);
  const uint32_t g0 = (uint32_t)(at >> kLvChunkBits);
  const unsigned long long chunk = at & kLvChunkMask;
  if (apart) {
    if (lane < n) A.grp[p][g0 + lane] = LvGroup{chunk + c0, 1u, 0u};
    if (lane + 32 < n) A.grp[p][g0 + lane + 32] = LvGroup{chunk + c1, 1u, 0u};
  } else if (lane < ng) {
    LvGroup g;
    g.start = lane ? chunk + t0 : chunk;
    g.n = lane ? n - 32 : min(n, 32);
    g.pad = 0;
    A.grp[p][g0 + lane] = g;
  }
  for (int e = lane; e < n; e += 32) {
    const uint64_t slot = apart ? (uint64_t)(g0 + e) * 32 : (uint64_t)g0 * 32 + e;
    const int4 f = fresh[e];
    const int32_t c = buf[e].y;
    A.rng[p][slot] = make_int4(f.x, f.y, f.z, 0);
    int32_t *dst = A.base[p] + slot * (uint32_t)A.stride[p];
    if (p == 1) {
      dst[0] = c;
    } else {
      const int32_t *mp = A.base[p - 1] + (uint64_t)(uint32_t)f.w * (uint32_t)A.stride[p - 1];
      if (p == 2) {
        *reinterpret_cast<int2 *>(dst) = make_int2(mp[0], c);
      } else if (p <= 4) {
        int4 v = lv_images(mp, p - 1);
        if (p == 3) v.z = c; else v.w = c;
        *reinterpret_cast<int4 *>(dst) = v;
      } else {
        for (int i = 0; i < p - 1; ++i) dst[i] = mp[i];
        dst[p - 1] = c;
      }
    }
  }
  __syncwarp();
  return true;
}

// Exact checks on the nbuf waiting survivors of level p (verified: they passed
// them before); those that pass become matches, or states of the next level.
// Returns how many states wait in buf because the next level is full (0: none).
template <bool kRows, bool kBatch, bool kSym>
__device__ __forceinline__ int lv_drain(const LvArgs &A, LvShared &sm, int p, int2 *buf, int nbuf, bool verified,
                                        int lane) {
  Bytes none;
  const uint32_t lt = lanemask_lt();
  const int warp = threadIdx.x >> 5;
  int4 *fresh = sm.fresh[warp];
  int done = 0;  // entries [0, done) of buf: states of the next level, their ranges in fresh
  const bool all_last = !kBatch && A.level1[p].last;
  for (int b = 0; b < nbuf; b += 32) {
    const int e = b + lane;
    bool ok = false;
    int2 sc = make_int2(0, 0);
    int32_t pid = 0;
    const int32_t *mp = nullptr;
    if (e < nbuf) {
      sc = buf[e];
      const int4 r = A.rng[p][(uint32_t)sc.x];
      pid = lv_pid(r.z);
      mp = A.base[p] + (uint64_t)(uint32_t)sc.x * (uint32_t)A.stride[p];
      ok = verified ||
           lv_exact_checks<kBatch>(A, kBatch ? A.levels[(int64_t)pid * A.kmax + p] : A.level1[p], mp, p, lv_drive(r.z), sc.y,
                           none);
    }
    if (kBatch ? true : all_last) {
      const bool last = kBatch ? ok && A.levels[(int64_t)pid * A.kmax + p].last : ok;
      const uint32_t bal = __ballot_sync(kFull, last);
      if (bal) {
        if (kBatch) {
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
              else if (at < A.row_cap[pid]) lv_write_row(E, rows + at * E.k, mp, p, sc.y);
            }
          }
        } else {
          const int naut = kSym ? A.emit1.naut : 1;
          if (lane == 0) sm.count[warp] += (unsigned long long)__popc(bal) * naut;
          if (kRows) {
            unsigned long long at = 0;
            if (lane == 0) at = atomicAdd(&A.ctl->rows, (unsigned long long)__popc(bal) * naut);
            at = __shfl_sync(kFull, at, 0) + (unsigned long long)__popc(bal & lt) * naut;
            if (last) {
              if (kSym && naut > 1) lv_write_images(A.emit1, A.aut, A.rows, at, A.cap, mp, p, sc.y);
              else if (at < A.cap) lv_write_row(A.emit1, A.rows + at * A.emit1.k, mp, p, sc.y);
            }
          }
        }
      }
      ok = ok && !last;
    }
    if (all_last) continue;
    // the range of the new state
    int4 r = make_int4(0, 0, 0, 0);
    unsigned long long found = 0;
    if (ok) r = lv_range<kBatch, !kRows, kSym>(A, p + 1, lv_images(mp, p), mp, sc.y, pid, found);
    if (p == 1 && !verified) {
      const uint32_t made = __popc(__ballot_sync(kFull, ok));
      if (lane == 0) sm.injected[warp] += made;
    }
    if (!kRows) lv_add_found<kBatch, kSym>(A, sm, found, pid, lane);
    const uint32_t bal = __ballot_sync(kFull, r.y > 0);
    if (r.y > 0) {
      const int at = done + __popc(bal & lt);  // at or before the entry just read
      r.w = sc.x;
      buf[at] = sc;
      fresh[at] = r;
    }
    done += __popc(bal);
    __syncwarp();
  }
  if (!done) return 0;
  if (lv_append(A, sm, p + 1, fresh, buf, done, lane)) return 0;
  return done;
}

// The vertices [v0, v0 + cnt) of the first level's list, those with candidates, to level 1.
template <bool kRows, bool kBatch, bool kSym>
__device__ __forceinline__ void lv_fill(const LvArgs &A, LvShared &sm, unsigned long long v0, unsigned long long cnt,
                                        uint32_t me) {
  if (me >= A.fill_warps) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t lt = lanemask_lt();
  int4 *fresh = sm.fresh[warp];
  int2 *buf = sm.buf[warp];
  // each warp an equal piece of the list, so that its groups hold neighbours
  const unsigned long long chunks = (cnt + 31) >> 5;
  const unsigned long long a = chunks * me / A.fill_warps, b = chunks * (me + 1) / A.fill_warps;
  int n = 0;
  for (unsigned long long ch = a; ch < b; ++ch) {
    const unsigned long long i = ch * 32 + lane;
    int4 r = make_int4(0, 0, 0, 0);
    unsigned long long found = 0;
    int32_t pid = 0, u = 0;
    if (i < cnt) {
      const unsigned long long s = v0 + i;
      if (kBatch) {
        int32_t lo = 0, hi = A.npat - 1;  // the last pattern whose first vertex is at or before the chunk's
        while (lo < hi) {
          const int32_t mid = (lo + hi + 1) >> 1;
          if (__ldg(A.vert_n + mid) <= v0 + ch * 32) lo = mid; else hi = mid - 1;
        }
        pid = lo;
        while (__ldg(A.vert_n + pid + 1) <= s) ++pid;
        u = __ldg(A.vert_at[pid] + s);
      } else {
        u = __ldg(A.vert + s);
      }
      r = lv_range<kBatch, !kRows, kSym>(A, 1, make_int4(0, 0, 0, 0), nullptr, u, pid, found);
    }
    if (!kRows) lv_add_found<kBatch, kSym>(A, sm, found, pid, lane);
    const uint32_t bal = __ballot_sync(kFull, r.y > 0);
    if (r.y > 0) {
      const int at = n + __popc(bal & lt);
      fresh[at] = r;
      buf[at] = make_int2(0, u);
    }
    n += __popc(bal);
    __syncwarp();
    if (n >= 32) {  // one full group; the rest moves down
      if (!lv_append(A, sm, 1, fresh, buf, 32, lane)) break;
      const int4 f = fresh[32 + lane];
      const int2 v = buf[32 + lane];
      __syncwarp();
      n -= 32;
      if (lane < n) {
        fresh[lane] = f;
        buf[lane] = v;
      }
      __syncwarp();
    }
  }
  // the slice is so small that its groups fit
  if (n && !lv_append(A, sm, 1, fresh, buf, n, lane) && lane == 0) atomicCAS(&A.ctl->status, 0, kStatQueue);
}

// The group that chunk x of the level lies in: the last one whose first chunk
// is at or before x.  `gi` is the group of the chunk before x (or none, ~0u):
// mostly x lies in one of the 32 groups after it, which takes one load.
__device__ __forceinline__ uint32_t lv_locate(const LvGroup *grp, uint32_t ngroup, unsigned long long x, int lane,
                                              uint32_t gi) {
  if (gi != ~0u) {
    const uint32_t i = gi + 1 + lane;
    const uint32_t le = __ballot_sync(kFull, i < ngroup && grp[i].start <= x);
    if (le && le != kFull) return gi + 32 - __clz(le);
  }
  uint32_t a = 0, n = ngroup;  // groups [a, a + n); the first starts at or before x
  while (n > 1) {
    const uint32_t step = (n + 31) >> 5;
    const uint32_t i = (uint32_t)lane * step;
    const uint32_t at = (31 - __clz(__ballot_sync(kFull, i < n && grp[a + i].start <= x))) * step;
    a += at;
    n = min(step, n - at);
  }
  return a;
}

// The expansion of a level by this warp: its own first run of chunks and then
// runs claimed from the level's counter, or (resume) what it left when the next
// level was full.  Returns the number of chunks it took.
template <bool kRows, bool kBatch, bool kSym>
__device__ __forceinline__ uint32_t lv_expand(const LvArgs &A, LvShared &sm, int p, bool resume, uint32_t me) {
  Bytes none;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t lt = lanemask_lt();
  int4 *rec = sm.rec[warp];
  int2 *buf = sm.buf[warp];
  const LvGroup *grp = A.grp[p];
  uint32_t run = me, look = 0, left = 0;
  unsigned long long x = 0;
  int nbuf = 0, wait = 0;
  const bool inner = p + 1 < A.kmax;
  bool stop_here = false;  // another warp found the next level full
  unsigned int full = 0;
  if (resume) {
    LvPause &P = A.pause[p][me];
    if (!P.on) return 0;
    x = P.x;
    left = P.left;
    run = P.run;
    wait = P.nwait;
    nbuf = P.nbuf;
    for (int e = lane; e < wait + nbuf; e += 32) buf[e] = P.buf[e];
    __syncwarp();
    const int first = wait;
    wait = lv_drain<kRows, kBatch, kSym>(A, sm, p, buf, wait, true, lane);
    if (!wait) {
      int2 v = make_int2(0, 0);
      if (lane < nbuf) v = buf[first + lane];
      __syncwarp();
      if (lane < nbuf) buf[lane] = v;
      __syncwarp();
    }
  } else {
    if (run < sm.nrun) {
      x = (unsigned long long)run * sm.run_len;
      left = (uint32_t)min((unsigned long long)sm.run_len, sm.total - x);
      // the next run, claimed early so that its number is there when this one is done
      if (lane == 0) run = gridDim.x * kLvWarps + atomicAdd(sm.claim, 1u);
    }
  }
  uint32_t gi = ~0u;
  while (!wait && !stop_here) {
    if (!left) {
      run = __shfl_sync(kFull, run, 0);
      if (run >= sm.nrun) break;
      x = (unsigned long long)run * sm.run_len;
      left = (uint32_t)min((unsigned long long)sm.run_len, sm.total - x);
      if (lane == 0) run = gridDim.x * kLvWarps + atomicAdd(sm.claim, 1u);
      gi = ~0u;
    }
    gi = lv_locate(grp, sm.ngroup, x, lane, gi);
    // the group's states to shared memory
    const LvGroup G = grp[gi];
    int4 r = make_int4(0, 0, 0, 0);
    if (lane < (int)G.n) r = A.rng[p][(uint64_t)gi * 32 + lane];
    uint32_t incl = (uint32_t)r.y;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(kFull, incl, o);
      if (lane >= o) incl += y;
    }
    const uint32_t total = __shfl_sync(kFull, incl, 31);
    const uint32_t excl = r.y > 0 ? incl - (uint32_t)r.y : 0xffffffffu;
    if (r.y > 0) {
      const int32_t pid = lv_pid(r.z), drive = lv_drive(r.z), probe = drive == 0 ? 1 : 0;
      const LevelPlan &L = kBatch ? A.levels[(int64_t)pid * A.kmax + p] : A.level1[p];
      const int32_t *mp = A.base[p] + ((uint64_t)gi * 32 + lane) * (uint32_t)A.stride[p];
      const int4 m = lv_images(mp, p);
      uint64_t part = 0;
      bool to = false;
      if (probe < L.npos) {
        const LvCons cs = lv_cons<kBatch>(A, L, probe);
        to = cs.kind == kOut;
        const int32_t f = lv_image(m, mp, cs.q);
        part = (to ? kHashU : kHashV) * (uint32_t)f + cs.la;
        Region g{0, A.G.rf_nword};
        if (A.G.regions) {
          const int4 vi = __ldg(&A.G.vi[HM_AT(A.G, f, A.G.n, kChkVertex)]);
          const int2 off = __ldg(&A.G.off[HM_AT(A.G, f, A.G.n, kChkVertex)]);
          g = region_of(f, (uint32_t)(to ? off.x : off.y), (uint32_t)(to ? vi.y : vi.z));
        }
        sm.reg[warp][lane] = g;
      }
      rec[lane] = make_int4((int32_t)((uint32_t)r.x - excl), lv_flags(lv_list(r.z), probe < L.npos, to, drive, probe + 1),
                            (int32_t)(uint32_t)part, (int32_t)(part >> 32));
      sm.img[warp][lane] = m;
      if (kBatch) sm.pid[warp][lane] = pid;
    }
    __syncwarp();
    if (x < G.start || x - G.start >= ((unsigned long long)total + 31) >> 5) {
      // cannot happen (the group's chunks were counted from the same numbers, whose sum fits 32 bits); never spin
      if (lane == 0) atomicCAS(&A.ctl->status, 0, kStatQueue);
      return look;
    }
    uint32_t pos0 = (uint32_t)(x - G.start) << 5;
    uint32_t n = min(left, ((total - 1) >> 5) + 1 - (pos0 >> 5));  // chunks of this group
    for (; n && !wait && !stop_here; --n, --left, ++x, pos0 += 32) {
      // (read four chunks before it is asked, so that nothing waits for it)
      if (inner && (look & 7u) == 0 && lane == 0) full = *(volatile unsigned int *)sm.paused;
      if (inner && (look & 7u) == 4u) stop_here = __shfl_sync(kFull, full, 0) != 0;
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
      int32_t c = 0;
      if (total - pos0 > (uint32_t)lane) {
        const int4 o = rec[ow];
        const uint32_t at = (uint32_t)o.x + pos0 + lane;
        c = __ldg((o.y & 1 ? A.G.gin_adj : A.G.gout_adj) + HM_AT(A.G, at, A.G.m, kChkList));
        const LevelPlan &L = kBatch ? A.levels[(int64_t)sm.pid[warp][ow] * A.kmax + p] : A.level1[p];
        const int32_t *mp = A.base[p] + ((uint64_t)gi * 32 + ow) * (uint32_t)A.stride[p];
        ok = lv_first_checks<kBatch, kSym>(A, L, o, sm.img[warp][ow], sm.reg[warp][ow], mp, p, c, none);
      }
      const uint32_t bal = __ballot_sync(kFull, ok);
      if (ok) buf[nbuf + __popc(bal & lt)] = make_int2((int32_t)(gi * 32 + ow), c);
      nbuf += __popc(bal);
      __syncwarp();
      if (nbuf >= kLvDrain) {
        // the first 64; the rest moves down
        wait = lv_drain<kRows, kBatch, kSym>(A, sm, p, buf, kLvDrain, false, lane);
        const int more = nbuf - kLvDrain;
        int2 v = make_int2(0, 0);
        if (lane < more) v = buf[kLvDrain + lane];
        __syncwarp();
        if (lane < more) buf[wait + lane] = v;  // behind the states that wait for room, if any
        nbuf = more;
        __syncwarp();
      }
    }
    __syncwarp();  // every lane is done with rec
  }
  if (!wait && !stop_here && nbuf) {
    wait = lv_drain<kRows, kBatch, kSym>(A, sm, p, buf, nbuf, false, lane);
    nbuf = 0;
  }
  if (inner) {
    LvPause &P = A.pause[p][me];
    if (wait || stop_here) {
      for (int e = lane; e < wait + nbuf; e += 32) P.buf[e] = buf[e];
      if (lane == 0) {
        P.x = x;
        P.left = left;
        P.run = run;
        P.nwait = wait;
        P.nbuf = nbuf;
        atomicAdd(sm.paused, 1u);
      }
    }
    if (lane == 0) P.on = wait || stop_here ? 1 : 0;
  }
  return look;
}

template <bool kRows, bool kBatch, bool kSym>
__global__ void __launch_bounds__(kLvThreads, kLvMinBlocks) k_levels(const __grid_constant__ LvArgs A) {
  extern __shared__ __align__(16) unsigned char s_raw[];
  LvShared &sm = *reinterpret_cast<LvShared *>(s_raw);
  const uint32_t warps = gridDim.x * kLvWarps, me = blockIdx.x * kLvWarps + (threadIdx.x >> 5);
  const int last = A.kmax - 1;  // the deepest level
  if ((threadIdx.x & 31) == 0) sm.count[threadIdx.x >> 5] = sm.injected[threadIdx.x >> 5] = 0;
  if (threadIdx.x == 0) sm.deadline = globaltimer_ns() + A.budget_ns;
  unsigned long long my_chunks = 0, cursor = 0;
  unsigned int target = 0, phase = 0;
  // each level: which filling of it this is, its groups and chunks, whether warps paused in it
  uint32_t fill[kMaxK + 1];
  unsigned long long made[kMaxK + 1];
  bool open[kMaxK + 1], begun[kMaxK + 1];
  for (int i = 0; i <= kMaxK; ++i) {
    fill[i] = 0;
    open[i] = false;
  }
  int p = 0;
  for (;;) {
    // what this phase fills is level p + 1
    if (p == 0 && cursor >= A.nvert) break;
    if (p < last) ++fill[p + 1];
    __syncthreads();
    if (threadIdx.x == 0) {
      if (p < last) {
        sm.made = &A.ctl->made[p + 1][fill[p + 1] % 3];
        if (blockIdx.x == 0) {
          A.ctl->made[p + 1][(fill[p + 1] + 1) % 3] = 0;
          A.ctl->claim[p + 1][(fill[p + 1] + 1) % 3] = 0;
        }
      }
      if (p > 0) {
        sm.total = made[p] & kLvChunkMask;
        sm.ngroup = (uint32_t)(made[p] >> kLvChunkBits);
        sm.run_len = (uint32_t)min(max(sm.total / (warps * 8ull), 1ull), 1ull << 30);
        sm.nrun = (uint32_t)((sm.total + sm.run_len - 1) / sm.run_len);
        sm.claim = &A.ctl->claim[p][fill[p] % 3];
        sm.paused = &A.ctl->paused[phase % 3];
        if (blockIdx.x == 0) A.ctl->paused[(phase + 1) % 3] = 0;
      }
    }
    __syncthreads();
    if (p == 0) {
      const unsigned long long n = min(A.slice, A.nvert - cursor);
      lv_fill<kRows, kBatch, kSym>(A, sm, cursor, n, me);
      cursor += n;
    } else {
      my_chunks += lv_expand<kRows, kBatch, kSym>(A, sm, p, begun[p], me);
      begun[p] = true;
    }
    if (p == last) {  // does anything follow?
      bool more = cursor < A.nvert;
      for (int q = 1; q < last; ++q) more |= open[q];
      if (!more) break;
    }
    target += gridDim.x;
    if (!lv_barrier(A, sm, target)) break;
    if (p > 0) {
      open[p] = p < last && *(volatile unsigned int *)&A.ctl->paused[phase % 3] != 0;
      ++phase;
    }
    if (p < last) {
      const unsigned long long m = *(volatile unsigned long long *)&A.ctl->made[p + 1][fill[p + 1] % 3];
      if (m & kLvChunkMask) {
        ++p;
        made[p] = m;
        begun[p] = false;
        continue;
      }
    }
    while (p > 0 && !open[p]) --p;
  }
  if ((threadIdx.x & 31) == 0) {
    const unsigned long long count = sm.count[threadIdx.x >> 5];
    if (count) atomicAdd(&A.ctl->count, count);
    if (my_chunks) atomicAdd(&A.ctl->chunks, my_chunks);
    if (sm.injected[threadIdx.x >> 5]) atomicAdd(&A.ctl->injected, (unsigned long long)sm.injected[threadIdx.x >> 5]);
  }
}

using LvKernel = void (*)(LvArgs);

LvKernel lv_kernel(bool rows, bool batch, bool sym) {
  if (batch) {
    if (sym) return rows ? k_levels<true, true, true> : k_levels<false, true, true>;
    return rows ? k_levels<true, true, false> : k_levels<false, true, false>;
  }
  if (sym) return rows ? k_levels<true, false, true> : k_levels<false, false, true>;
  return rows ? k_levels<true, false, false> : k_levels<false, false, false>;
}

// Resident blocks of a variant (0: the device cannot run it).
// Asked once per device: each needs the opt-in to more than 48 KB of shared memory.
int lv_grid(LvKernel f, int slot) {
  static PerDevice<8> cache;
  int dev = 0;
  cudaGetDevice(&dev);
  const int v = cache.get(dev, slot, [&] {
    int per_sm = 0, coop = 0;
    if (cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess || !coop ||
        cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(LvShared)) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, f, kLvThreads, sizeof(LvShared)) != cudaSuccess)
      per_sm = 0;
    (void)cudaGetLastError();
    return per_sm > 0 ? per_sm * num_sms() : -1;
  });
  return std::max(v, 0);
}

int16_t lv_class(const hm_graph *g, int32_t alab, int32_t vlab) {
  const int64_t a = (int64_t)alab - g->al0, v = (int64_t)vlab - g->vl0;
  if (a < 0 || a >= g->nal || v < 0 || v >= g->nvl) return -1;
  return (int16_t)(a * g->nvl + v);
}

// The conditions of position p towards earlier positions, position 1 included
// (there the seeding arc and, if asked for, its opposite).
int lv_conditions(const Plan &P, int p, Cons *out, int *npos) {
  if (p > 1) {
    *npos = P.npos[p];
    for (int j = 0; j < P.ncons[p]; ++j) out[j] = P.cons[p][j];
    return P.ncons[p];
  }
  int n = 0;
  out[n++] = Cons{0, P.seed_rev ? kIn : kOut, 0, P.seed_lab};
  if (P.back_req) out[n++] = Cons{0, P.seed_rev ? kOut : kIn, 0, P.back_lab};
  *npos = n;
  if (P.back_forbid) out[n++] = Cons{0, P.seed_rev ? kNotOut : kNotIn, 0, 0};
  return n;
}

// The plan with position 1 matched last: position i > 1 becomes i - 1.  Only
// induced non-arcs and order constraints can name position 1 in a later
// position; they are read from the other side.
void lv_defer(Plan &P) {
  const Plan O = P;
  const int k = O.k, z = k - 1;
  auto pos = [&](int i) { return i == 0 ? 0 : i == 1 ? z : i - 1; };
  Cons tail[kMaxCons];
  int tpos = 0, tn = lv_conditions(O, 1, tail, &tpos);
  P.sym_gt[z] = O.sym_gt[1] & 1u;
  P.sym_lt[z] = O.sym_lt[1] & 1u;
  for (int p = 2; p < k; ++p) {
    const int q = p - 1;
    int c = 0;
    for (int j = 0; j < O.ncons[p]; ++j) {
      Cons cs = O.cons[p][j];
      if (cs.q == 1) {
        tail[tn++] = Cons{(int8_t)q, cs.kind == kNotOut ? kNotIn : kNotOut, 0, 0};
        continue;
      }
      cs.q = (int8_t)pos(cs.q);
      P.cons[q][c++] = cs;
    }
    P.ncons[q] = c;
    P.npos[q] = O.npos[p];
    uint32_t gt = 0, lt = 0;
    for (int i = 0; i < p; ++i) {
      if (i == 1) continue;
      gt |= (O.sym_gt[p] >> i & 1u) << pos(i);
      lt |= (O.sym_lt[p] >> i & 1u) << pos(i);
    }
    P.sym_gt[z] |= (O.sym_lt[p] >> 1 & 1u) << q;  // f(p) < f(1)
    P.sym_lt[z] |= (O.sym_gt[p] >> 1 & 1u) << q;  // f(p) > f(1)
    P.sym_gt[q] = gt;
    P.sym_lt[q] = lt;
    P.vlab[q] = O.vlab[p];
    P.orig[q] = O.orig[p];
    P.din[q] = O.din[p];
    P.dout[q] = O.dout[p];
  }
  for (int j = 0; j < tn; ++j) P.cons[z][j] = tail[j];
  P.ncons[z] = tn;
  P.npos[z] = tpos;
  P.vlab[z] = O.vlab[1];
  P.orig[z] = O.orig[1];
  P.din[z] = O.din[1];
  P.dout[z] = O.dout[1];
  for (int s = 0; s < O.naut && O.naut > 1; ++s)
    for (int v = 0; v < k; ++v) P.aut[s][v] = (int8_t)pos(O.aut[s][v]);
  if (O.root_pos >= 0) P.root_pos = pos(O.root_pos);
}

// `deferred`: lv_defer has been applied, position 1 is like any other.
void lv_level(const hm_graph *g, const Plan &P, bool deferred, int p, bool want_rows, LevelPlan &L, LvCons *out) {
  std::memset(&L, 0, sizeof(L));
  if (p >= P.k) return;
  Cons cons[kMaxCons];
  int npos = 0, n = 0;
  if (p == 1 && deferred) {
    npos = P.npos[1];
    n = P.ncons[1];
    for (int j = 0; j < n; ++j) cons[j] = P.cons[1][j];
  } else {
    n = lv_conditions(P, p, cons, &npos);
  }
  L.npos = (int16_t)npos;
  L.ncons = (int16_t)n;
  L.last = p == P.k - 1;
  L.root = P.root_pos == p;
  L.dout = P.dout[p];
  L.din = P.din[p];
  L.sym_gt = P.sym_gt[p];
  L.sym_lt = P.sym_lt[p];
  for (int j = 0; j < n; ++j) {
    const ArcKey l = j < npos ? labelled_key(ArcKey{0}, cons[j].lab) : ArcKey{0};
    out[j] = LvCons{cons[j].q, cons[j].kind, j < npos ? lv_class(g, cons[j].lab, P.vlab[p]) : (int16_t)0,
                       cons[j].lab, l.h};
  }
  // arcs to later positions: a single one is found missing with the new state's range anyway
  L.need_deg = !L.last && P.dout[p] + P.din[p] - npos >= 2;
  L.closed = L.last && !want_rows && npos == 1 && n == 1 && !L.root;
}

// The vertices the first level starts from: those with position 0's label and a
// group for a condition of position 1, the shortest such list.
const int32_t *lv_start(const hm_graph *g, const Plan &P, const LevelPlan &L, const LvCons *cons, int64_t *cnt) {
  const int64_t lab = (int64_t)P.vlab[0] - g->vl0;
  const int32_t *list = g->vby_out;
  *cnt = 0;
  if (lab < 0 || lab >= g->nvl) return list;
  *cnt = INT64_MAX;
  for (int j = 0; j < L.npos; ++j) {
    const bool in = cons[j].kind == kIn;
    const uint32_t *b = g->vstart + (in ? g->ncls * g->nvl + 1 : 0) + lab * g->ncls + std::max<int>(cons[j].cls, 0);
    const int64_t here = cons[j].cls < 0 ? 0 : (int64_t)b[1] - b[0];
    if (here < *cnt) {
      *cnt = here;
      list = (in ? g->vby_in : g->vby_out) + b[0];
    }
  }
  return list;
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

// A page-locked block for what a call reads back: a copy into ordinary memory is
// staged by the driver (1.5 to 2 us more per call).  The process keeps the blocks
// that were in use at one time, up to kMost (0.6 MB), for any thread's calls: a
// thread that makes a single call neither locks a block (0.1 ms) nor frees one,
// which would wait for the kernels of every stream.  A call that finds none left, or has more counts than
// a block holds, reads into ordinary memory.
struct Landing {
  static constexpr int32_t kCounts = 4096;
  static constexpr int kMost = 16;
  struct Block {
    LvCtl ctl;
    unsigned long long counts[kCounts];
  } *p = nullptr;
  struct Pool {
    std::mutex mu;
    Block *idle[kMost];
    int nidle = 0, made = 0;
  };
  // never destroyed: calls of other threads may outlast static objects
  static Pool &pool() {
    static Pool *q = new Pool;
    return *q;
  }
  explicit Landing(bool wanted) {
    if (!wanted) return;
    Pool &q = pool();
    {
      std::lock_guard<std::mutex> lk(q.mu);
      if (q.nidle) {
        p = q.idle[--q.nidle];
        return;
      }
      if (q.made == kMost) return;
      ++q.made;
    }
    if (cudaMallocHost((void **)&p, sizeof(Block)) != cudaSuccess) {
      (void)cudaGetLastError();
      p = nullptr;
      std::lock_guard<std::mutex> lk(q.mu);
      --q.made;
    }
  }
  ~Landing() {
    if (!p) return;
    Pool &q = pool();
    std::lock_guard<std::mutex> lk(q.mu);
    q.idle[q.nidle++] = p;
  }
  Landing(const Landing &) = delete;
  Landing &operator=(const Landing &) = delete;
};

hm_status levels_try(const LvLaunch &L, cudaStream_t s, bool *ran, LvCtl *result, int *grid_out, int *threads_out,
                     float *ms) {
  *ran = false;
  const hm_graph *g = L.g;
  const bool batch = L.npat > 0;
  bool sym = false;
  int kmax = 0;
  const int32_t np = batch ? L.npat : 1;
  for (int32_t i = 0; i < np; ++i) {
    const Plan &P = batch ? *L.plans[i] : *L.plan;
    sym |= P.naut > 1;
    kmax = std::max(kmax, (int)P.k);
  }
  const LvKernel f = lv_kernel(L.want_rows, batch, sym);
  int grid = lv_grid(f, (L.want_rows ? 4 : 0) + (batch ? 2 : 0) + (sym ? 1 : 0));
  if (grid <= 0 || np >= 1 << 24) return HM_OK;
  LvArgs A{};
  std::vector<int8_t> aut;
  std::vector<LevelPlan> levels(batch ? (size_t)np * kmax : 0);
  std::vector<LvCons> conds;
  std::vector<EmitPlan> emit(batch ? np : 0);
  std::vector<unsigned long long> vert_n(batch ? np + 1 : 0);
  std::vector<const int32_t *> vert_at(batch ? np : 0);
  std::vector<int2> deg0(batch ? np : 0);
  const int32_t *first_vertex = g->vby_out;
  // a guess at the candidates: every position multiplies the states by a group's mean length, and
  // every further condition keeps as many of them as a group holds of its label's vertices
  const double mean = (double)g->m / (double)std::max<int64_t>(1, std::min(g->ndir_out, g->ndir_in));
  const double keeps = std::min(1.0, mean * g->nvl / (double)std::max(g->n, 1));
  double guess = 0;
  for (int32_t i = 0; i < np; ++i) {
    const Plan &P0 = batch ? *L.plans[i] : *L.plan;
    const bool defer = P0.k > 2 && P0.defer1 && L.defer;
    Plan moved;
    if (defer) {
      moved = P0;
      lv_defer(moved);
    }
    const Plan &P = defer ? moved : P0;
    LevelPlan *lv = batch ? &levels[(size_t)i * kmax] : A.level1;
    const int32_t *list = g->vby_out;
    int64_t cnt = 0;
    for (int p = 1; p < std::min(kmax, (int)P.k); ++p) {
      LvCons c[kMaxCons];
      lv_level(g, P, defer, p, L.want_rows, lv[p], c);
      lv[p].cons = (int32_t)conds.size();
      conds.insert(conds.end(), c, c + lv[p].ncons);
      if (p == 1) list = lv_start(g, P, lv[1], c, &cnt);
    }
    lv[1].final = defer ? (int8_t)(P.k - 1) : 0;
    lv_emit(P, batch ? emit[i] : A.emit1, aut);
    if (batch) {
      vert_n[i] = A.nvert;
      vert_at[i] = list - (int64_t)A.nvert;
      deg0[i] = make_int2(P.dout[0], P.din[0]);
    } else {
      first_vertex = list;
      A.dout0 = P.dout[0];
      A.din0 = P.din[0];
      A.root0 = L.root_mask && P.root_pos == 0;
    }
    A.nvert += (unsigned long long)cnt;
    double states = (double)cnt, last = defer ? mean : 1;  // (lv_has_final drops the vertices without a last image)
    for (int j = 1; defer && j < lv[P.k - 1].npos; ++j) last *= keeps;
    states *= std::min(last, 1.0);
    for (int p = 1; p < P.k; ++p) {
      guess += states *= mean;
      for (int j = 1; j < lv[p].npos; ++j) states *= keeps;
    }
  }
  if (batch) vert_n[np] = A.nvert;
  // Barriers cost less with fewer blocks: on 5,000 arcs with four labels a 4-cycle takes 56 us with 20
  // blocks and 65 with all 304.  But the arcs do not bound the work (a tournament of five on 60
  // vertices: 3.06 ms with the 8 blocks that 1,800 arcs ask for, 1.50 depth first, 0.22 now), so there is
  // one block for every four chunks per warp of the guess (a 7-cycle on 5,000 unlabelled arcs: 20
  // blocks 666 us, 304 blocks 241), and for every 512 arcs (pendant triangles on 73,000 R-MAT arcs: 60
  // us, 68 with one for every 256); without hubs, where the mean says what a vertex has, 64 of
  // these are enough (an 8-vertex pattern on 400,000 arcs: 106 us, 118 with 304).
  const double by_guess = guess / (32.0 * 4 * kLvWarps) + 1;
  int64_t by_arcs = (g->m + 511) / 512;
  if ((int64_t)g->maxdeg * g->n <= 16 * g->m) by_arcs = std::min<int64_t>(by_arcs, 64);
  grid = (int)std::min<double>(grid, std::max((double)by_arcs, by_guess));

  // The workspace: a quarter for the warps' resume points (fewer blocks if they
  // do not fit), the rest for the levels' states, equal numbers of groups each.
  const int top = kmax - 1;  // deepest level
  if (top > 1)
    grid = (int)std::min<uint64_t>((uint64_t)grid, std::max<uint64_t>(1, L.workspace / 4 / ((uint64_t)(top - 1) * kLvWarps *
                                                                                           sizeof(LvPause))));
  const int64_t warps = (int64_t)grid * kLvWarps;
  auto stride_of = [&](int p) { return p <= 2 ? p : (p + 3) / 4 * 4; };
  auto group_bytes = [&](int p) { return sizeof(LvGroup) + 32 * (sizeof(int4) + 4 * (uint64_t)stride_of(p)); };
  uint64_t per_group = 0;
  for (int p = 2; p <= top; ++p) per_group += group_bytes(p);
  // No more groups than the graph has arcs, or as the guess asks for: short calls on small graphs
  // take a few MB, a batch of 64 six-vertex paths on 916 arcs (hundreds of millions of states) all.
  const uint64_t room = std::max<uint64_t>({(uint64_t)g->m, 8192, (uint64_t)std::min(guess / 32, (double)kLvMaxGroups)});
  const uint64_t most = std::min<uint64_t>({(uint64_t)kLvMaxGroups, room,
                                            (kLvChunkMask >> 1) / (uint64_t)std::max(g->maxdeg, 1)});
  // the first level holds all its vertices if they fit an eighth of the workspace
  const uint64_t first = std::min<uint64_t>({most, (A.nvert + 31) / 32 + (uint64_t)warps,
                                             L.workspace / 8 / group_bytes(1)});
  A.gcap[1] = (uint32_t)std::max<uint64_t>(first, 64);
  for (int p = 2; p <= top; ++p)
    A.gcap[p] = (uint32_t)std::max<uint64_t>(std::min(most, L.workspace / 8 * 5 / per_group), 64);
  A.fill_warps = std::min((uint32_t)warps, A.gcap[1] / 2);  // each may leave a group that is not full
  // a slice's states fit whatever their candidates: one group each where 32 lists could exceed a group's sum
  A.slice = (uint64_t)(A.gcap[1] - A.fill_warps) * (32ull * g->maxdeg >= kLvGroupCands ? 1 : 32);
  auto round = [](size_t b) { return (b + 255) / 256 * 256; };
  size_t bytes = round(sizeof(LvCtl));
  size_t at_rng[kMaxK + 1] = {}, at_grp[kMaxK + 1] = {}, at_ps[kMaxK + 1] = {}, at_st[kMaxK + 1] = {};
  auto reserve = [&](size_t n) {
    const size_t a = bytes;
    bytes += round(n);
    return a;
  };
  for (int p = 1; p <= top; ++p) {
    A.stride[p] = stride_of(p);
    at_rng[p] = reserve(sizeof(int4) * 32 * A.gcap[p]);
    at_grp[p] = reserve(sizeof(LvGroup) * A.gcap[p]);
    at_st[p] = reserve(4 * (size_t)A.stride[p] * 32 * A.gcap[p]);
    if (p < top) at_ps[p] = reserve(sizeof(LvPause) * (size_t)warps);
  }
  if (!batch) {
    std::copy(conds.begin(), conds.end(), A.cons1);
    conds.clear();
  }
  // a batch's tables, and the automorphisms of symmetric patterns, in one host block and one copy
  size_t at_tab = bytes, tab = 0;
  auto place = [&](size_t n) {
    const size_t a = tab;
    tab += round(n);
    return a;
  };
  const size_t t_levels = place(sizeof(LevelPlan) * levels.size()), t_cons = place(sizeof(LvCons) * conds.size()), t_emit = place(sizeof(EmitPlan) * emit.size()),
               t_vn = place(8 * vert_n.size()), t_va = place(8 * vert_at.size()), t_deg = place(8 * deg0.size()),
               t_aut = place(aut.size());
  std::vector<unsigned char> host(tab);
  auto put = [&](size_t a, const void *src, size_t n) {
    if (n) std::memcpy(host.data() + a, src, n);
  };
  put(t_levels, levels.data(), sizeof(LevelPlan) * levels.size());
  put(t_cons, conds.data(), sizeof(LvCons) * conds.size());
  put(t_emit, emit.data(), sizeof(EmitPlan) * emit.size());
  put(t_vn, vert_n.data(), 8 * vert_n.size());
  put(t_va, vert_at.data(), 8 * vert_at.size());
  put(t_deg, deg0.data(), 8 * deg0.size());
  put(t_aut, aut.data(), aut.size());
  bytes += tab;

  struct Space {
    unsigned char *p = nullptr;
    cudaStream_t s;
    ~Space() {
      if (p) cudaFreeAsync(p, s);
    }
  } ws{nullptr, s};
  HM_CUDA_TRY(cudaMallocAsync((void **)&ws.p, bytes, s));
  for (int p = 1; p <= top; ++p) {
    A.rng[p] = reinterpret_cast<int4 *>(ws.p + at_rng[p]);
    A.grp[p] = reinterpret_cast<LvGroup *>(ws.p + at_grp[p]);
    A.base[p] = reinterpret_cast<int32_t *>(ws.p + at_st[p]);
    if (p < top) A.pause[p] = reinterpret_cast<LvPause *>(ws.p + at_ps[p]);
  }
  A.vert = first_vertex;
  A.ctl = reinterpret_cast<LvCtl *>(ws.p);
  unsigned char *t = ws.p + at_tab;
  A.levels = reinterpret_cast<const LevelPlan *>(t + t_levels);
  A.cons = reinterpret_cast<const LvCons *>(t + t_cons);
  A.emit = reinterpret_cast<const EmitPlan *>(t + t_emit);
  A.vert_n = reinterpret_cast<const unsigned long long *>(t + t_vn);
  A.vert_at = reinterpret_cast<const int32_t *const *>(t + t_va);
  A.deg0 = reinterpret_cast<const int2 *>(t + t_deg);
  A.aut = reinterpret_cast<const int8_t *>(t + t_aut);
  A.G = g->dev();
  A.npat = L.npat;
  A.root_mask = L.root_mask;
  A.budget_ns = budget_ms() * 1000000ull;
  A.rows = L.rows;
  A.cap = L.cap;
  A.counts = L.counts;
  A.row_off = L.row_off;
  A.row_cap = L.row_cap;
  A.row_cursor = L.row_cursor;
  A.kmax = kmax;
  HM_CUDA_TRY(cudaMemsetAsync(A.ctl, 0, sizeof(LvCtl), s));
  if (tab) HM_CUDA_TRY(cudaMemcpyAsync(t, host.data(), tab, cudaMemcpyHostToDevice, s));
  cudaEvent_t ev[2] = {nullptr, nullptr};
  if (ms) {
    cudaEventCreate(&ev[0]);
    cudaEventCreate(&ev[1]);
    cudaEventRecord(ev[0], s);
  }
  void *args[] = {&A};
  const cudaError_t le = cudaLaunchCooperativeKernel((const void *)f, dim3(grid), dim3(kLvThreads), args,
                                                     sizeof(LvShared), s);
  hm_status st = HM_OK;
  if (le == cudaSuccess) {
    *ran = true;
    if (ms) cudaEventRecord(ev[1], s);
    Landing landing(L.npat <= Landing::kCounts);
    Landing::Block *l = landing.p;
    LvCtl *to = l ? &l->ctl : result;
    unsigned long long *counts = l ? l->counts : L.counts_host;
    const size_t nc = L.counts_host ? sizeof(unsigned long long) * L.npat : 0;
    if (cudaMemcpyAsync(to, A.ctl, sizeof(LvCtl), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        (nc && cudaMemcpyAsync(counts, L.counts, nc, cudaMemcpyDeviceToHost, s) != cudaSuccess) ||
        cudaStreamSynchronize(s) != cudaSuccess)
      st = HM_ERR_CUDA;
    if (l && st != HM_OK) {
      landing.p = nullptr;  // a copy into it may be under way: it is not given to another call
    } else if (l) {
      *result = l->ctl;
      if (nc) std::memcpy(L.counts_host, l->counts, nc);
    }
    if (ms && st == HM_OK) cudaEventElapsedTime(ms, ev[0], ev[1]);
  }
  (void)cudaGetLastError();  // a launch that was refused: the caller searches depth first
  if (ms) {
    cudaEventDestroy(ev[0]);
    cudaEventDestroy(ev[1]);
  }
  *grid_out = grid;
  *threads_out = kLvThreads;
  return st;
}

}  // namespace

hm_status levels_run(const LvLaunch &L, cudaStream_t s, bool *ran, LvCtl *result, int *grid, int *threads,
                     float *ms) {
  LvLaunch M = L;
  for (;;) {
    const hm_status st = levels_try(M, s, ran, result, grid, threads, ms);
    // a device that is nearly full: the levels in smaller parts
    if (st != HM_ERR_OOM || M.workspace <= kLevelWorkspaceMin) return st;
    M.workspace = std::max(M.workspace / 4, kLevelWorkspaceMin);
  }
}

}  // namespace hm
