// hm_internal.cuh -- types and device helpers shared by the library's sources.
//
// Layout of a loaded target graph in HBM (all arrays 256-byte aligned):
//   src      int32[m]  source of each arc, CSR order (the per-arc source array
//                      of the double-index storage, Sec. III-D)
//   out_adj  int32[m]  out-neighbours, sorted within each vertex
//   out_elab int32[m]  label of each out-arc, parallel to out_adj
//   in_adj   int32[m]  in-neighbours, sorted within each vertex (CSC)
//   in_elab  int32[m]  label of each in-arc, parallel to in_adj
//   vi       int4[n]   {vertex label, out-degree, in-degree, 0}
//   off      int2[n]   {first out-arc, first in-arc}   (m < 2^31, so 32-bit offsets)
//   afilt    uint2[W]  arc filter: W = 4 * ceil(m/8) words of 64 bits holding two
//                      keys per arc, (u, v) and (u, v, label), 16 bits per key
//                      (64 MB for 16M arcs, within the 129 MB L2)
//   ahash    int4[2*H] arc hash table: H = m buckets of two 16-byte slots
//                      {u, v, label, 0} (32 bytes per arc, half the slots used)
// A vertex's label and both degrees arrive in one 16-byte load, its list
// offsets in a second one.  The label-grouped lists, their directory and dense
// offsets (gout_adj, gin_adj, gdir_out, gdir_in, vdir, gofs_out, gofs_in) and the
// filter by endpoint (rfilt_out, rfilt_in) are described with DevGraph.
#pragma once

#include <cuda_runtime.h>
#include <nvtx3/nvToolsExt.h>
#include <stdint.h>

#include <atomic>

#include "hipermotif.h"

namespace hm {

constexpr int kMaxK = HM_MAX_K;
constexpr int kMaxCons = 2 * (HM_MAX_K - 1);
constexpr int kMaxAut = 64;  // symmetry breaking is used for patterns with at most this many automorphisms
static_assert(kMaxCons <= 64, "condition masks are 64-bit");
constexpr int kWarp = 32;

struct DevGraph {
  int32_t n;
  int64_t m;
  const int32_t *src;
  const int32_t *out_adj;
  const int32_t *out_elab;
  const int32_t *in_adj;
  const int32_t *in_elab;
  const int4 *vi;
  const int2 *off;
  // label-grouped copies of the lists: each vertex's list ordered by
  // (arc label, neighbour label, neighbour id); one directory entry per group
  const int32_t *gout_adj;
  const int32_t *gin_adj;
  const int4 *gdir_out;  // {arc label, neighbour label, first, end} (relative to the list start)
  const int4 *gdir_in;
  const int4 *vdir;      // {first out entry, out entries, first in entry, in entries}
  // Bloom filter over the arcs, one word per key, keyed by (u, v) and by (u, v,
  // label): a "no" is exact, a "maybe" needs the search.  Searches over more
  // than filt_min entries probe it first (filt_min < 0: never).
  const uint2 *afilt;
  uint32_t afilt_nword;
  int32_t filt_min;
  // exact arc lookup in one or two 32-byte reads, for what the filter lets through
  const int4 *ahash;
  uint32_t ahash_nbkt;
  // dense group offsets: the group of class c = (arc label - first arc label) *
  // vertex labels + (neighbour label - first vertex label) of vertex v is
  // [gofs[v * ncls + c], gofs[v * ncls + c + 1]) of the grouped lists; ncls = 0:
  // too many classes, only the directory
  const int32_t *gofs_out, *gofs_in;
  int32_t ncls;
  int32_t maxdeg;  // largest out- or in-degree
  // with regions: the arc filter once more, each vertex's out- (in-) arcs in words
  // of its own (see region_of).  Without: both are afilt.  rf_nword words each.
  const uint2 *rfilt_out, *rfilt_in;
  uint32_t rf_nword;
  int32_t regions;
  // directory lengths, and the violation word of bounds-checked builds (null otherwise)
  int64_t ndir_out, ndir_in;
  unsigned long long *check;
};

// Sites of the bounds checks (HM_CHECK builds): which array an index was meant for.
enum CheckSite : int {
  kChkVertex = 1,   // vi, off, vdir (vertex id < n)
  kChkDirOut = 2,   // gdir_out entry
  kChkDirIn = 3,    // gdir_in entry
  kChkList = 4,     // src, out/in adjacency and labels, grouped lists (position < m)
  kChkFilter = 5,   // arc filter word
  kChkHash = 6,     // arc hash bucket
  kChkGroup = 7,    // dense group offset
  kChkRegion = 8,   // word of the filter by endpoint
};

// One pairwise condition between the position being extended (p) and an
// earlier position q, on the candidate c for p:
enum ConsKind : int8_t {
  kOut = 0,     // arc f(q) -> c must exist with label `lab`   (pattern arc q->p)
  kIn = 1,      // arc c -> f(q) must exist with label `lab`   (pattern arc p->q)
  kNotOut = 2,  // no arc f(q) -> c                            (induced, non-arc q->p)
  kNotIn = 3,   // no arc c -> f(q)                            (induced, non-arc p->q)
};

struct Cons {
  int8_t q;
  int8_t kind;
  int16_t pad;
  int32_t lab;
};

// One look-ahead class of a position (see Plan::la).
struct LookClass {
  int8_t kind;   // kOut: arcs f(p) -> later positions; kIn: arcs from them
  int8_t need;   // later positions in the class
  int16_t pad;
  int32_t alab;  // arc label
  int32_t vlab;  // the later positions' vertex label
};

// Per-pattern, per-mode plan, indexed by position after Alg. 1.
struct Plan {
  int32_t k;
  int32_t induced;
  int32_t orig[kMaxK];  // position -> original pattern vertex
  int32_t vlab[kMaxK];  // label required at each position
  int32_t din[kMaxK];   // pattern in-degree at each position
  int32_t dout[kMaxK];  // pattern out-degree at each position
  // the seeding arc between positions 0 and 1
  int32_t seed_rev;     // 0: target arc (a,b) gives f(0)=a, f(1)=b; 1: f(0)=b, f(1)=a
  int32_t seed_lab;     // label of that pattern arc
  int32_t back_req;     // pattern also has 1->0: target arc f(1)->f(0) needed, label back_lab
  int32_t back_lab;
  int32_t back_forbid;  // induced, and the pattern lacks the opposite arc: forbid it in the target
  int32_t ov_need;      // |N(0) & N(1)| in the pattern (neighbour-overlap test)
  int32_t root_pos;     // position whose image must pass a root mask, or -1
  int32_t ncons[kMaxK]; // conditions for position p (positives first)
  int32_t npos[kMaxK];  // how many of them are kOut/kIn
  int32_t gbase[kMaxK]; // first group slot of position p (sum of npos before p)
  int32_t ngrp;         // group slots in total
  // Shared position-0 states: when no later position has a pattern arc to
  // position 1 (defer1), the seeds can be grouped by their position-0 image
  // and position 1 chosen last, from the group's seed list; the induced
  // non-arcs between position 1 and later positions are then checked for
  // each chosen image (defer, with q the later position and the kind read as
  // "f(q) -> v" for kNotOut, "v -> f(q)" for kNotIn).
  int32_t defer1;
  int32_t ndefer;
  Cons cons[kMaxK][kMaxCons];
  Cons defer[kMaxCons];
  // Symmetry breaking.  The matches of a pattern (Sec. II-A, Eqs. 1-3) fall
  // into orbits of |Aut| maps f o s, s an automorphism of the labelled
  // pattern.  The search keeps the one map per orbit that satisfies the order
  // constraints below (f(p) > f(q) for bit q of sym_gt[p], f(p) < f(q) for
  // bit q of sym_lt[p], q < p) and emits it with its |Aut| - 1 images: image
  // s of original vertex v is the vertex at position aut[s][v].  naut = 1:
  // no symmetry breaking (aut[0] maps each vertex to its own position).
  int32_t naut;
  uint32_t sym_gt[kMaxK];
  uint32_t sym_lt[kMaxK];
  int8_t aut[kMaxAut][kMaxK];
  // Look-ahead (a labelled form of VF2's terminal-set rules): a candidate for
  // position p needs, for each class (direction, arc label, neighbour label)
  // of the pattern arcs between p and later positions, at least `need`
  // neighbours of that class -- their images must be distinct.
  int32_t nla[kMaxK];
  LookClass la[kMaxK][kMaxCons];
};

// A plan without symmetry breaking: every map is searched for itself.
inline void strip_symmetry(Plan &P) {
  if (P.naut <= 1) return;
  P.naut = 1;  // aut[0] is the identity
  for (int i = 0; i < kMaxK; ++i) P.sym_gt[i] = P.sym_lt[i] = 0;
}

// Budget / status words shared by all warps of one call.
enum : int32_t { kStatOk = 0, kStatBudget = 1, kStatQueue = 2 };

// Byte tallies of the instrumented kernel variants (hm_set_counters): `req`,
// the bytes the kernel's accesses request at the granularity it reads them
// (an 8-byte word per filter probe, a 16-byte vertex record, ...);
// `model`, the method's algorithmic bytes under the survey's cost model: 12 B
// per arc scanned, 12 B per vertex record gathered (label and two degrees),
// 8 B per candidate read from an adjacency list (neighbour and arc label),
// ceil(log2(d+1)) x 4 B per membership or non-arc test (a binary search of
// the shorter list, d entries), 4 B per surviving candidate's label, 4 B per
// neighbour merged by the overlap test, 8 B per state and 4k B per row
// written.  `c += b` adds to req.
struct Bytes {
  uint64_t req = 0, model = 0;
  __host__ __device__ Bytes &operator+=(uint64_t b) {
    req += b;
    return *this;
  }
};

// ceil(log2(d + 1)) x 4: the bytes of a binary search over d sorted entries.
__host__ __device__ __forceinline__ uint64_t search_bytes(int64_t d) {
  uint64_t b = 0;
  while (d > 0) {
    d >>= 1;
    b += 4;
  }
  return b;
}

// ---------------------------------------------------------------------------
// device helpers
// ---------------------------------------------------------------------------
#ifdef __CUDACC__

// Is x in the sorted list a[lo, lo+len)?  Returns its index or -1.  Offsets are
// 32-bit (the loader caps m below 2^31).  kCount adds the bytes read to `bytes`.
template <bool kCount>
__device__ __forceinline__ int32_t search_c(const int32_t *__restrict__ a, int32_t lo, int32_t len,
                                            int32_t x, Bytes &bytes) {
  const int32_t end = lo + len;
  while (len > 0) {
    const int32_t half = len >> 1;
    const int32_t v = __ldg(a + lo + half);
    if (kCount) bytes += 4;
    if (v < x) {
      lo += half + 1;
      len -= half + 1;
    } else {
      len = half;
    }
  }
  if (lo >= end) return -1;
  if (kCount) bytes += 4;
  return __ldg(a + lo) == x ? lo : -1;
}

// ---- arc filter -------------------------------------------------------------
// Every arc (u, v) with label l enters the filter under two keys: the pair
// (u, v) -- "is there an arc at all", for induced non-arcs and the opposite-arc
// test -- and the triple (u, v, l) -- "is there an arc with this label", for
// the pattern's arcs.  A key's hash is the sum A u + B v (+ C (l + 1)) modulo
// 2^64 with fixed odd constants (multilinear hashing: the upper halves of such
// sums are pairwise independent over the choice of the constants;
// Dietzfelbinger, "Universal hashing and k-wise independent random variables
// via integer arithmetic without primes", STACS 1996).  The constants are the
// first three splitmix64 outputs from seed 0x243F6A8885A308D3, made odd.  The
// upper half chooses a 64-bit word, and both halves together four bits in it,
// two in each half.  At 16 bits per key a key that was never inserted passes
// with probability about 0.5 % (measured on R-MAT arcs; 0.8 % on a lattice);
// an inserted key always passes.  The sum is linear, so the part of an endpoint
// that stays the same over many probes is computed once; a probe is then about
// 20 instructions and one 8-byte load.  (A 256-bit block with one bit in each
// of eight words and a 64-bit finalizer as the hash passed 0.1 % but took about
// 60 instructions and two loads, and eight atomics per key to build: 286 us for
// 3.9M arcs, now 43.)
constexpr uint64_t kHashU = 0x2cb0f69f4abea221ull, kHashV = 0x9417034723148989ull, kHashL = 0xdd555950609dfe03ull;

struct ArcKey {
  uint64_t h;
};

__host__ __device__ __forceinline__ ArcKey pair_key(int32_t u, int32_t v) {
  return ArcKey{kHashU * (uint32_t)u + kHashV * (uint32_t)v};
}

__host__ __device__ __forceinline__ ArcKey labelled_key(ArcKey k, int32_t lab) {
  return ArcKey{k.h + kHashL * ((uint64_t)(uint32_t)lab + 1)};
}

__host__ __device__ __forceinline__ uint32_t filter_word(ArcKey k, uint32_t nword) {
  return (uint32_t)(((k.h >> 32) * (uint64_t)nword) >> 32);
}

// Both halves of the hash in one word: the bits in the filter word, the bucket of the table.
__host__ __device__ __forceinline__ uint32_t key_fold(ArcKey k) {
  return (uint32_t)(k.h >> 32) * 0x9e3779b1u ^ (uint32_t)k.h;
}

// The key's bits in its word: two in each 32-bit half.
__host__ __device__ __forceinline__ uint2 filter_bits(ArcKey k) {
  const uint32_t h = key_fold(k);
  uint2 m;
  m.x = (1u << (h >> 27)) | (1u << ((h >> 22) & 31u));
  m.y = (1u << ((h >> 17) & 31u)) | (1u << ((h >> 12) & 31u));
  return m;
}

// The same filter laid out by an endpoint: a vertex with d arcs whose list
// starts at `off` has d / 2 + 1 words of its own from off / 2 + v on (16 bits per
// key, two keys per arc, and the regions of different vertices never meet).
// The level-by-level search probes a state's candidates against one fixed vertex,
// and then stays in a few lines of L1 and L2 instead of the whole filter (64 MB for
// 16M arcs, 600 MB for 150M, more than L2 holds).
// kRegionArcs: from here on a graph gets them.  Measured with them against without:
// 150M arcs, five connectome motifs 3.09 against 4.26 ms; 16M arcs, bi-fan 4.40
// against 4.59, 4-cycles 2.67 against 2.76.  The line lies where a batch of 64
// cycles of three to five vertices crosses: 3.9M arcs 13.95 against 13.67 ms, 5.8M
// 43.2 / 42.5, 8.0M 49.1 / 48.6, 10.8M 124 / 127, 14.1M 126 / 133, 16.1M 186 / 199.
// Below, the filter is at home in L2 as it is, and what the region of a vertex
// costs to look up is not won back; loading takes 4 to 5 % longer with them.
constexpr int64_t kRegionArcs = (int64_t)1 << 23;

struct Region {
  uint32_t base, nword;
};

__host__ __device__ __forceinline__ Region region_of(int32_t v, uint32_t off, uint32_t deg) {
  return Region{(off >> 1) + (uint32_t)v, (deg >> 1) + 1};
}

// ---- bounds checks -------------------------------------------------------------
// Built with HM_CHECK=1 (a separate library, libhipermotif_check.so), every
// index into a graph array passes through HM_AT: one outside [0, n) is
// recorded in *G.check -- bit 63 set, the site in bits 48..55, the index's
// low 48 bits -- if no violation was recorded before, and replaced by 0, so
// the access stays inside the array and the kernel runs on.  The host reads
// and clears the word with hm_check_status.  In the default build HM_AT is
// the index itself.
#ifndef HM_CHECK
#define HM_CHECK 0
#endif
#if HM_CHECK
__device__ __forceinline__ int64_t checked_index(const DevGraph &G, int64_t i, int64_t n, int site) {
  if (i >= 0 && i < n) return i;
  if (G.check)
    atomicCAS(G.check, 0ull,
              (1ull << 63) | ((unsigned long long)(site & 0xff) << 48) | ((unsigned long long)i & 0xffffffffffffull));
  return 0;
}
#define HM_AT(G, i, n, site) ::hm::checked_index((G), (int64_t)(i), (int64_t)(n), (site))
#else
#define HM_AT(G, i, n, site) (i)
#endif

// search_c over one of the graph's lists (every list array has m entries); in
// check builds a span outside [0, m) is recorded and searched as empty
template <bool kCount>
__device__ __forceinline__ int32_t search_g(const DevGraph &G, const int32_t *__restrict__ a, int32_t lo,
                                            int32_t len, int32_t x, Bytes &bytes) {
#if HM_CHECK
  if (len > 0 && (lo < 0 || (int64_t)lo + len > G.m)) {
    checked_index(G, lo < 0 ? (int64_t)lo : (int64_t)lo + len - 1, G.m, kChkList);
    return -1;
  }
#endif
  return search_c<kCount>(a, lo, len, x, bytes);
}

template <bool kCount>
__device__ __forceinline__ bool filter_has(const DevGraph &G, ArcKey k, Bytes &bytes) {
  const uint2 w = __ldg(G.afilt + HM_AT(G, filter_word(k, G.afilt_nword), G.afilt_nword, kChkFilter));
  if (kCount) bytes += 8;
  const uint2 m = filter_bits(k);
  return ((m.x & ~w.x) | (m.y & ~w.y)) == 0;
}

// false: there is certainly no arc u -> v.  true: there may be.
template <bool kCount>
__device__ __forceinline__ bool arc_maybe(const DevGraph &G, int32_t u, int32_t v, Bytes &bytes) {
  return filter_has<kCount>(G, pair_key(u, v), bytes);
}

// ---- arc hash table -----------------------------------------------------------
// Open addressing over buckets of two 16-byte slots {u, v, label, 0}, one
// 32-byte sector per bucket, with linear probing over buckets from the one the
// pair's hash selects.  Slots fill in order and are never removed, so an empty
// slot (u = -1) ends a probe sequence.  There are as many buckets as arcs
// (half the slots used), so a lookup nearly always reads one sector.
__host__ __device__ __forceinline__ uint32_t hash_bucket(ArcKey pair, uint32_t nbkt) {
  return (uint32_t)((key_fold(pair) * (uint64_t)nbkt) >> 32);
}

// Is u -> v an arc?  If so, *lab is its label.
template <bool kCount>
__device__ __forceinline__ bool arc_find(const DevGraph &G, int32_t u, int32_t v, int32_t *lab,
                                         Bytes &bytes) {
  uint32_t b = hash_bucket(pair_key(u, v), G.ahash_nbkt);
  for (uint32_t it = 0; it < G.ahash_nbkt; ++it) {
    const size_t bk = (size_t)HM_AT(G, b, G.ahash_nbkt, kChkHash);
    const int4 s0 = __ldg(G.ahash + 2 * bk);
    const int4 s1 = __ldg(G.ahash + 2 * bk + 1);
    if (kCount) bytes += 32;
    if (s0.x == u && s0.y == v) {
      *lab = s0.z;
      return true;
    }
    if (s1.x == u && s1.y == v) {
      *lab = s1.z;
      return true;
    }
    if (s0.x < 0 || s1.x < 0) return false;
    b = b + 1 == G.ahash_nbkt ? 0 : b + 1;
  }
  return false;
}

// false: there is certainly no arc u -> v with label lab.  true: there may be.
template <bool kCount>
__device__ __forceinline__ bool arc_maybe_l(const DevGraph &G, int32_t u, int32_t v, int32_t lab,
                                            Bytes &bytes) {
  return filter_has<kCount>(G, labelled_key(pair_key(u, v), lab), bytes);
}

__device__ __forceinline__ uint64_t globaltimer_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ uint32_t lanemask_lt() {
  uint32_t m;
  asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
  return m;
}
#endif  // __CUDACC__

}  // namespace hm

// ---------------------------------------------------------------------------
// host-side objects
// ---------------------------------------------------------------------------

namespace hm {
int32_t filter_min();  // current search length above which the arc filter is probed first

// A named range on the host thread's timeline around the launches of one
// phase (NVTX): profilers can select a phase's kernels by it ("ncu --nvtx
// --nvtx-include hm.extend/"); without a tool attached it costs a few ns.
struct NvtxRange {
  explicit NvtxRange(const char *name) { nvtxRangePushA(name); }
  ~NvtxRange() { nvtxRangePop(); }
  NvtxRange(const NvtxRange &) = delete;
  NvtxRange &operator=(const NvtxRange &) = delete;
};
}

struct hm_graph {
  int device;
  int32_t n;
  int64_t m;
  int32_t *src, *out_adj, *out_elab, *in_adj, *in_elab;
  int4 *vi;
  int2 *off;
  int32_t *gout_adj, *gin_adj;
  int4 *gdir_out, *gdir_in, *vdir;
  uint2 *afilt;
  uint32_t afilt_nword;
  int4 *ahash;
  uint32_t ahash_nbkt;
  int64_t ndir_out, ndir_in;
  int32_t *gofs_out, *gofs_in;  // dense group offsets (null: ncls = 0)
  int32_t ncls, al0, vl0, nal, nvl;  // classes; first labels and label counts
  int32_t maxdeg;                    // largest out- or in-degree
  uint2 *rfilt_out, *rfilt_in;       // the arc filter by source and by target, or afilt
  uint32_t rf_nword;
  int32_t regions;
  // with ncls: the vertices of label vl0 + l that have an out- (in-) group of
  // class c are vby_out (vby_in) [vstart[b], vstart[b + 1]), b = l * ncls + c
  // (in: b = ncls * nvl + 1 + l * ncls + c); vstart is host memory
  int32_t *vby_out, *vby_in;
  uint32_t *vstart;
  unsigned long long *check;  // bounds-checked builds: the violation word (device)
  size_t bytes;
  void *owned[8];  // the device allocations behind the arrays
  int nowned;
  // multi-property graphs (hm_load_graph_props): the sorted distinct property
  // tuples of vertices and arcs (host, malloc'ed); a label is a tuple's rank
  int32_t nvp, nep;
  int64_t nvtab, netab;
  int32_t *vtab, *etab;
  hm::DevGraph dev() const {
    return hm::DevGraph{n,        m,        src,     out_adj,  out_elab, in_adj,     in_elab,
                        vi,       off,      gout_adj, gin_adj, gdir_out, gdir_in,    vdir,
                        afilt,    afilt_nword, hm::filter_min(), ahash, ahash_nbkt, gofs_out, gofs_in, ncls, maxdeg, rfilt_out,
                        rfilt_in, rf_nword, regions, ndir_out, ndir_in, check};
  }
};

struct hm_pattern {
  int32_t k, mp;
  int32_t order[HM_MAX_K];
  hm::Plan plan[2];  // [mode]
};

namespace hm {

// Thread-local record of the last call (hm_last_stats).
hm_stats &tls_stats();
bool timing_enabled();
bool counters_enabled();
hm_tuning tuning();  // current process-wide extension knobs (validated)
// log2 of the warps per depth-2 state; 0 (automatic) gives 4 warps to shared
// position-0 states (few, each standing for up to 32 states) and 1 otherwise.
inline int32_t wps_shift(const hm_tuning &t, bool shared = false) {
  if (t.warps_per_state == 0) return shared ? 2 : 0;
  return t.warps_per_state >= 4 ? 2 : t.warps_per_state >= 2 ? 1 : 0;
}
// All knobs at their defaults: the extension runs level by level (hm_levels.cu).
inline bool default_search(const hm_tuning &t) {
  return t.extend_min_blocks == 4 && t.split_min == 64 && t.pair_mode == 0 && t.seeds_per_fetch == 1 &&
         t.poll_every == 128 && t.leaf_flatten > 0 && t.arc_filter == 1 && t.warps_per_state == 0 && t.lookahead <= 0;
}
uint64_t budget_ms();
uint64_t budget_chunks();

// Sort rows of `width` int32 words lexicographically by the `nkey` columns
// listed in key_cols (most significant first); every key value must lie in
// [0, 2^bits).  `rows` and `tmp` hold nrows*width words each; the sorted rows
// end in `rows`.  Stable.  Launches on `stream`.
// *launches (if given) receives the number of kernels it launched.
hm_status radix_sort_rows(int32_t *rows, int32_t *tmp, int64_t nrows, int width,
                          const int *key_cols, int nkey, int bits, cudaStream_t stream,
                          int *launches = nullptr);

// As radix_sort_rows, with a bit width (1..32) and an xor mask per key column
// (the xor maps signed values to an unsigned order, e.g. 0x80000000).  With
// `err` (device, zero) the call does not wait: a barrier that gave up sets *err,
// and what is launched behind must look at it before it uses the rows.
hm_status radix_sort_rows_cols(int32_t *rows, int32_t *tmp, int64_t nrows, int width,
                               const int *key_cols, const int *key_bits, const uint32_t *key_xor,
                               int nkey, cudaStream_t stream, int *launches = nullptr, int *err = nullptr);

// Sorts of at most this many rows place each row by counting the rows before
// it (n^2 compares over the whole GPU) instead of by a radix sort.  The two
// cost the same at about 16,000 rows (155 us, hm_sort.cu); at 12,288 counting
// takes about 95 us.
constexpr int64_t kRankMaxRows = 12288;

// 64 rows, from row0 on, of a list of n rows of `width` words: the list starts
// at word `src` of the caller's rows, at word `dst` of the temporary and at
// key `key0` of the packed keys.
struct RankTile {
  int64_t src, dst;
  int32_t key0, n, width, row0;
};
constexpr int kRankTileRows = 64;

// Sorts many lists (nrows rows in all, at most `longest` in one), each
// lexicographically by all its columns (values below 2^bits), through `tmp`;
// `tiles` (device) lists every list's tiles.
hm_status rank_sort_tiles(int32_t *rows, int32_t *tmp, const RankTile *tiles, int ntiles, int64_t nrows,
                          int64_t longest, int width_max, int bits, cudaStream_t stream);

// out[i] = in[0] + ... + in[i-1] for i in [0, n); values and total below 2^32.
hm_status exclusive_scan_u32(const uint32_t *in, uint32_t *out, int64_t n, cudaStream_t stream);

// A batched call (hm_count_batch, hm_enumerate_batch) with a limit on the
// memory its extension takes for the levels' states.  With `fit` (the query
// server's single pass) it keeps what fits: every count, and for each pattern
// whose count fits its region [row_offsets[i], row_offsets[i+1]) its sorted
// rows there and fit[i] = 1; fit[i] = 0 otherwise.
hm_status batch_run(const hm_graph *g, const hm_pattern *const *patterns, const int32_t *modes, int32_t npat,
                    int32_t *rows_dev, const uint64_t *row_offsets, uint64_t *counts, uint8_t *fit,
                    uint64_t workspace, cudaStream_t stream);

int bits_for(int64_t n);  // bits needed for values in [0, n)
int num_sms();            // of the current device

// kSlots values per device, each found once on the first kDevices devices and every
// time on further ones (a process may hold graphs on several devices).  Zero-initialised,
// so for static objects; `find` must not give 0.
template <int kSlots>
struct PerDevice {
  static constexpr int kDevices = 64;
  std::atomic<int> v[kDevices][kSlots];
  template <typename F>
  int get(int dev, int slot, F find) {
    if (dev < 0 || dev >= kDevices) return find();
    int x = v[dev][slot].load(std::memory_order_relaxed);
    if (!x) {
      x = find();
      v[dev][slot].store(x, std::memory_order_relaxed);
    }
    return x;
  }
};

}  // namespace hm

#define HM_CUDA_TRY(expr)                                    \
  do {                                                       \
    cudaError_t e_ = (expr);                                 \
    if (e_ != cudaSuccess) {                                 \
      (void)cudaGetLastError();                              \
      return e_ == cudaErrorMemoryAllocation ? HM_ERR_OOM    \
                                             : HM_ERR_CUDA;  \
    }                                                        \
  } while (0)
