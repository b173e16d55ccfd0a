// hm_graph.cu -- building the device-resident target graph (hm_load_graph).
//
// The paper stores the target in a double-index format: CSR plus an
// arc-to-source array so that both endpoints of an arc are O(1) away, with
// attributes in contiguous arrays and O(log d) edge-attribute lookup in
// sorted adjacency (Sec. III-D).  Here the same storage is built on the GPU
// from an arc list, plus what the search kernels look up:
//   1. pack rows (src, dst, label, aux), check ids / self-loops, and find
//      the label ranges                                         (k_pack, k_bounds)
//   2. stable radix sort by (src, dst); split into src / out_adj / out_elab,
//      check repeated pairs, fill out-offsets                        (k_split)
//   3. the label-grouped out-lists: each list counted and placed by class
//      (arc label, neighbour label) on its own      (k_group_lists, k_group_hubs)
//   4. stable sort by dst alone (the rows are in source order), and steps 2-3
//      for the in-lists
//   5. a directory with one entry per (vertex, class) group, and the vertices
//      of each (vertex label, class)            (k_group_dirs, k_class_place)
//   6. per-vertex records {label, degrees}, {offsets}, {directory spans}
//   7. the arc filter: every arc sets its bits under two keys       (k_filter);
//      with at least 2^23 arcs also by source and by target         (k_regions)
//   8. the arc hash table: every arc claims a slot                  (k_hash)
// With more than 64 classes steps 3-5 sort the rows by (key, arc label,
// neighbour label) instead and read groups off the sorted rows (build_groups).
// The grouped lists let the extension kernel jump straight to the candidates
// whose arc label and vertex label already match (checkAttributes of Alg. 2
// and Alg. 3 applied as a range lookup instead of per candidate).
#include <algorithm>
#include <cstring>
#include <vector>

#include "hm_internal.cuh"

namespace hm {
namespace {

constexpr int kThreads = 256;
constexpr int64_t kMaxDense = 64;  // classes with dense group offsets (two per lane of a warp)
constexpr int kW = 4;  // row width: src, dst, arc label, aux

enum : uint32_t { kErrRange = 1, kErrSelf = 2, kErrDup = 4, kErrHash = 8 };

struct Bounds {
  int32_t emin, emax, vmin, vmax, maxdeg;
};

// Smallest and largest value of the block's threads: one atomic each (with one
// per thread, packing 3.9M arcs took 37 instead of 21 us).
__device__ __forceinline__ void block_bounds(int32_t lo, int32_t hi, int32_t *glo, int32_t *ghi) {
  __shared__ int32_t s_lo[kThreads / 32], s_hi[kThreads / 32];
  lo = __reduce_min_sync(0xffffffffu, lo);
  hi = __reduce_max_sync(0xffffffffu, hi);
  if ((threadIdx.x & 31) == 0) {
    s_lo[threadIdx.x >> 5] = lo;
    s_hi[threadIdx.x >> 5] = hi;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < kThreads / 32; ++w) {
      lo = min(lo, s_lo[w]);
      hi = max(hi, s_hi[w]);
    }
    atomicMin(glo, lo);
    atomicMax(ghi, hi);
  }
}

__global__ void k_begin(uint32_t *err, Bounds *bnd) {
  err[0] = err[1] = 0;
  *bnd = Bounds{INT32_MAX, INT32_MIN, INT32_MAX, INT32_MIN, 0};
}

__global__ void k_pack(const int32_t *__restrict__ src, const int32_t *__restrict__ dst,
                       const int32_t *__restrict__ elab, int64_t m, int32_t n,
                       int32_t *__restrict__ rows, uint32_t *__restrict__ err,
                       Bounds *__restrict__ bnd) {
  int32_t lo = INT32_MAX, hi = INT32_MIN;
  uint32_t bad = 0;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < m;
       e += (int64_t)gridDim.x * blockDim.x) {
    int32_t a = src[e], b = dst[e], l = elab[e];
    if (a < 0 || a >= n || b < 0 || b >= n) bad |= kErrRange;
    else if (a == b) bad |= kErrSelf;
    int4 r = make_int4(min(max(a, 0), max(n - 1, 0)), min(max(b, 0), max(n - 1, 0)), l, 0);
    reinterpret_cast<int4 *>(rows)[e] = r;
    lo = min(lo, l);
    hi = max(hi, l);
  }
  if (bad) atomicOr(err, bad);
  block_bounds(lo, hi, &bnd->emin, &bnd->emax);
}

__global__ void k_vbounds(const int32_t *__restrict__ vlab, int32_t n, Bounds *__restrict__ bnd) {
  int32_t lo = INT32_MAX, hi = INT32_MIN;
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n;
       v += (int64_t)gridDim.x * blockDim.x) {
    lo = min(lo, vlab[v]);
    hi = max(hi, vlab[v]);
  }
  block_bounds(lo, hi, &bnd->vmin, &bnd->vmax);
}

// off[v] = first row whose key column is >= v, for v in [0, n]; rows sorted by that column.
__device__ __forceinline__ void fill_gap(const int32_t *__restrict__ rows, int col, int64_t e,
                                         int64_t m, int32_t n, int64_t *__restrict__ off) {
  int32_t cur = rows[kW * e + col];
  int32_t prev = e ? rows[kW * (e - 1) + col] : -1;
  for (int32_t v = prev + 1; v <= cur; ++v) off[v] = e;
  if (e == m - 1)
    for (int64_t v = (int64_t)cur + 1; v <= n; ++v) off[v] = m;
}

// The sorts of a load whose barriers may give up (radix_sort_rows_cols with `err`)
// leave it to the host to ask once, behind all of them.  Until then the rows may be in
// any order, or partly not written at all, and so may what was made of them: every
// kernel that takes an index from either looks at the word first and does nothing
// once it is set (one load per thread; reading it back on the host after each sort
// would stop the launches twice).
__device__ __forceinline__ bool sort_failed(const int *err) { return *(const volatile int *)err != 0; }

// Split rows sorted by (key, other): adj = other column, lab = arc label, offsets on key.
__global__ void k_split(const int32_t *__restrict__ rows, int64_t m, int32_t n, int key, int other,
                        int32_t *__restrict__ src_out, int32_t *__restrict__ adj,
                        int32_t *__restrict__ lab, int64_t *__restrict__ off,
                        uint32_t *__restrict__ err, const int *sort_err) {
  if (sort_failed(sort_err)) return;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < m;
       e += (int64_t)gridDim.x * blockDim.x) {
    int32_t a = rows[kW * e + key], b = rows[kW * e + other];
    if (src_out) src_out[e] = a;
    adj[e] = b;
    lab[e] = rows[kW * e + 2];
    if (err && e && rows[kW * (e - 1) + key] == a && rows[kW * (e - 1) + other] == b)
      atomicOr(err, kErrDup);
    fill_gap(rows, key, e, m, n, off);
  }
}

// aux column = label of the neighbour (column `other`)
__global__ void k_set_aux(int32_t *__restrict__ rows, int64_t m, int other,
                          const int32_t *__restrict__ vlab) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < m;
       e += (int64_t)gridDim.x * blockDim.x)
    rows[kW * e + 3] = vlab[rows[kW * e + other]];
}

// Rows sorted by (key, arc label, neighbour label, neighbour): grouped list +
// group-start flags (flags[m] = 0 is the scan's sentinel).
__global__ void k_group_flags(const int32_t *__restrict__ rows, int64_t m, int key, int other,
                              int32_t *__restrict__ gadj, uint32_t *__restrict__ flags) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e <= m;
       e += (int64_t)gridDim.x * blockDim.x) {
    if (e == m) {
      flags[m] = 0;
      continue;
    }
    const int32_t *r = rows + kW * e;
    gadj[e] = r[other];
    uint32_t f = 1;
    if (e) {
      const int32_t *q = rows + kW * (e - 1);
      f = (q[key] != r[key] || q[2] != r[2] || q[3] != r[3]) ? 1u : 0u;
    }
    flags[e] = f;
  }
}

// One directory entry per group: {arc label, neighbour label, first, end} relative to the list.
__global__ void k_group_entries(const int32_t *__restrict__ rows, int64_t m, int key,
                                const uint32_t *__restrict__ flags, const uint32_t *__restrict__ idx,
                                const int64_t *__restrict__ off, int4 *__restrict__ dir) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < m;
       e += (int64_t)gridDim.x * blockDim.x) {
    if (!flags[e]) continue;
    const int32_t *r = rows + kW * e;
    const int32_t v = r[key];
    const int64_t base = off[v];
    // the group ends at the next group start of the same vertex, or at the list end
    int64_t end = e + 1;
    const int64_t vend = off[v + 1];
    while (end < vend && !flags[end]) ++end;
    dir[idx[e]] = make_int4(r[2], r[3], (int32_t)(e - base), (int32_t)(end - base));
  }
}

__global__ void k_zero_off(int64_t *__restrict__ off, int32_t n) {
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v <= n;
       v += (int64_t)gridDim.x * blockDim.x)
    off[v] = 0;
}

// Per-vertex records.  The directory indexes are per row (rows sorted by key:
// index of the group the row starts or continues) or, by_vertex, per vertex.
__global__ void k_vertex(const int32_t *__restrict__ vlab, const int64_t *__restrict__ out_off,
                         const int64_t *__restrict__ in_off, const uint32_t *__restrict__ oidx,
                         const uint32_t *__restrict__ iidx, bool by_vertex, int32_t n, int4 *__restrict__ vi,
                         int2 *__restrict__ voff, int4 *__restrict__ vdir, Bounds *__restrict__ bnd) {
  int32_t most = 0;
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n;
       v += (int64_t)gridDim.x * blockDim.x) {
    int64_t o0 = out_off[v], o1 = out_off[v + 1], i0 = in_off[v], i1 = in_off[v + 1];
    vi[v] = make_int4(vlab[v], (int32_t)(o1 - o0), (int32_t)(i1 - i0), 0);
    voff[v] = make_int2((int32_t)o0, (int32_t)i0);
    uint32_t os = oidx ? oidx[by_vertex ? v : o0] : 0, oe = oidx ? oidx[by_vertex ? v + 1 : o1] : 0;
    uint32_t is = iidx ? iidx[by_vertex ? v : i0] : 0, ie = iidx ? iidx[by_vertex ? v + 1 : i1] : 0;
    if (by_vertex) {  // one prefix sum runs over both directions
      is -= iidx[0];
      ie -= iidx[0];
    }
    vdir[v] = make_int4((int32_t)os, (int32_t)(oe - os), (int32_t)is, (int32_t)(ie - is));
    most = max(most, (int32_t)max(o1 - o0, i1 - i0));
  }
  most = __reduce_max_sync(0xffffffffu, most);
  if ((threadIdx.x & 31) == 0 && most) atomicMax(&bnd->maxdeg, most);
}

// ---- label-grouped lists, few classes ------------------------------------------
//
// One direction's lists (sorted by neighbour) regrouped by class, stably: each
// list is counted and placed on its own, one warp per vertex, and the dense
// group offsets are the counts' prefix sums.  (A radix sort of all rows by
// (key, arc label, neighbour label), flags, a scan and a walk to each group's
// end took 394 us per direction for 3.9M arcs, R-MAT scale 18; this takes 150
// with the directory.  Bound by the latency of the list and label loads: a
// warp has one list at a time, and most lists are short.)
struct Classes {
  int32_t ncls, nvl, al0, vl0;
};

constexpr int kHub = 1024;  // longer lists get a block of 32 warps

__device__ __forceinline__ int class_of(const Classes &C, int32_t alab, int32_t vlab) {
  return (alab - C.al0) * C.nvl + (vlab - C.vl0);
}

// Group starts from the counts of classes lane and lane + 32; the starts replace
// the counts in shared memory, relative to the list, and go to gofs.  Returns
// the number of groups.
__device__ __forceinline__ int class_starts(const Classes &C, uint32_t *cnt, int lane, int64_t base,
                                            int32_t *__restrict__ gofs) {
  const uint32_t c0 = cnt[lane], c1 = cnt[lane + 32];
  uint32_t x = c0, y = c1;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t a = __shfl_up_sync(0xffffffffu, x, o), b = __shfl_up_sync(0xffffffffu, y, o);
    if (lane >= o) {
      x += a;
      y += b;
    }
  }
  const uint32_t s0 = x - c0, s1 = __shfl_sync(0xffffffffu, x, 31) + y - c1;
  cnt[lane] = s0;
  cnt[lane + 32] = s1;
  if (lane < C.ncls) gofs[lane] = (int32_t)(base + s0);
  if (lane + 32 < C.ncls) gofs[lane + 32] = (int32_t)(base + s1);
  __syncwarp();
  return __popc(__ballot_sync(0xffffffffu, c0 > 0)) + __popc(__ballot_sync(0xffffffffu, c1 > 0));
}

__global__ void __launch_bounds__(kThreads)
k_group_lists(const int64_t *__restrict__ off, const int32_t *__restrict__ adj, const int32_t *__restrict__ elab,
              const int32_t *__restrict__ vlab, int32_t n, int64_t m, Classes C, int32_t *__restrict__ gadj,
              int32_t *__restrict__ gofs, uint32_t *__restrict__ ngroup, int32_t *__restrict__ hubs,
              uint32_t *__restrict__ nhub, const int *sort_err) {
  if (sort_failed(sort_err)) return;
  __shared__ uint32_t s_cnt[kThreads / 32][64];
  const int lane = threadIdx.x & 31;
  uint32_t *cnt = s_cnt[threadIdx.x >> 5];
  uint32_t lt;
  asm("mov.u32 %0, %%lanemask_lt;" : "=r"(lt));
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t v = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; v < n; v += nw) {
    const int64_t base = off[v], len = off[v + 1] - base;
    if (len > kHub) {
      if (lane == 0) hubs[atomicAdd(nhub, 1u)] = (int32_t)v;
      continue;
    }
    cnt[lane] = cnt[lane + 32] = 0;
    __syncwarp();
    int32_t id = 0;
    int c = 64;
    for (int64_t i = lane; i < len; i += 32) {
      id = adj[base + i];
      c = class_of(C, elab[base + i], vlab[id]);
      atomicAdd(&cnt[c], 1u);
    }
    __syncwarp();
    const int g = class_starts(C, cnt, lane, base, gofs + v * C.ncls);
    if (lane == 0) ngroup[v] = g;
    for (int64_t b = 0; b < len; b += 32) {
      const bool valid = b + lane < len;
      if (len > 32 && valid) {  // a list of one chunk is in registers
        id = adj[base + b + lane];
        c = class_of(C, elab[base + b + lane], vlab[id]);
      }
      const uint32_t peers = __match_any_sync(0xffffffffu, valid ? c : 64 + lane);
      const uint32_t at = valid ? cnt[c] : 0;
      __syncwarp();
      if (valid) {
        gadj[base + at + __popc(peers & lt)] = id;
        if ((peers & lt) == 0) cnt[c] = at + __popc(peers);
      }
      __syncwarp();
    }
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    gofs[(int64_t)n * C.ncls] = (int32_t)m;
    ngroup[n] = 0;
  }
}

// The lists left out above: 32 warps each count and place an equal piece.
__global__ void __launch_bounds__(1024)
k_group_hubs(const int64_t *__restrict__ off, const int32_t *__restrict__ adj, const int32_t *__restrict__ elab,
             const int32_t *__restrict__ vlab, Classes C, int32_t *__restrict__ gadj, int32_t *__restrict__ gofs,
             uint32_t *__restrict__ ngroup, const int32_t *__restrict__ hubs, const uint32_t *__restrict__ nhub,
             const int *sort_err) {
  if (sort_failed(sort_err)) return;
  __shared__ uint32_t s_cnt[32][64], s_all[64];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t *cnt = s_cnt[warp];
  uint32_t lt;
  asm("mov.u32 %0, %%lanemask_lt;" : "=r"(lt));
  for (uint32_t h = blockIdx.x; h < *nhub; h += gridDim.x) {
    const int32_t v = hubs[h];
    const int64_t base = off[v], len = off[v + 1] - base;
    const int64_t piece = ((len + 31) / 32 + 31) / 32 * 32;
    const int64_t a = base + min(len, warp * piece), z = base + min(len, (warp + 1) * piece);
    cnt[lane] = cnt[lane + 32] = 0;
    __syncwarp();
    for (int64_t i = a + lane; i < z; i += 32) atomicAdd(&cnt[class_of(C, elab[i], vlab[adj[i]])], 1u);
    __syncthreads();
    if (threadIdx.x < 64) {  // each warp's part of every class, and the classes' sizes
      uint32_t run = 0;
      for (int w = 0; w < 32; ++w) {
        const uint32_t t = s_cnt[w][threadIdx.x];
        s_cnt[w][threadIdx.x] = run;
        run += t;
      }
      s_all[threadIdx.x] = run;
    }
    __syncthreads();
    if (warp == 0) {
      const int g = class_starts(C, s_all, lane, base, gofs + (int64_t)v * C.ncls);
      if (lane == 0) ngroup[v] = g;
    }
    __syncthreads();
    cnt[lane] += s_all[lane];
    cnt[lane + 32] += s_all[lane + 32];
    __syncwarp();
    for (int64_t b = a; b < z; b += 32) {
      const bool valid = b + lane < z;
      int32_t id = 0;
      int c = 64 + lane;
      if (valid) {
        id = adj[b + lane];
        c = class_of(C, elab[b + lane], vlab[id]);
      }
      const uint32_t peers = __match_any_sync(0xffffffffu, c);
      const uint32_t at = valid ? cnt[c] : 0;
      __syncwarp();
      if (valid) {
        gadj[base + at + __popc(peers & lt)] = id;
        if ((peers & lt) == 0) cnt[c] = at + __popc(peers);
      }
      __syncwarp();
    }
    __syncthreads();
  }
}

// Entries of both directories and the sorts' status, in one place for one copy.
__global__ void k_dir_sizes(const uint32_t *oidx, const uint32_t *iidx, int32_t n, const int *sort_err, uint32_t *sizes) {
  sizes[0] = oidx[n];
  sizes[1] = iidx[n] - oidx[n];
  sizes[2] = sort_failed(sort_err) ? 1u : 0u;
}

// Both directions of the steps below run in one launch (blockIdx.y).
struct Direction {
  const int32_t *gofs;
  const uint32_t *didx;  // first directory entry of each vertex, counted from didx[0] on
  int4 *dir;
  uint32_t *cnt, *cur, *start;  // per (vertex label, class): groups, cursors, list starts
  int32_t *vby;
};

// The directory from the dense group offsets, one warp per vertex, classes on
// the lanes; counts the groups of each (vertex label, class) for k_class_place.
__global__ void __launch_bounds__(kThreads)
k_group_dirs(const __grid_constant__ Direction D0, const __grid_constant__ Direction D1,
             const int32_t *__restrict__ vlab, int32_t n, Classes C) {
  __shared__ uint32_t h[kMaxDense * kMaxDense];
  const Direction &D = blockIdx.y ? D1 : D0;
  const int32_t *gofs = D.gofs;
  const uint32_t *didx = D.didx, first = D.didx[0];
  int4 *dir = D.dir;
  uint32_t *cnt_of = D.cnt;
  const int nbin = C.ncls * C.nvl, lane = threadIdx.x & 31;
  for (int b = threadIdx.x; b < nbin; b += blockDim.x) h[b] = 0;
  __syncthreads();
  uint32_t lt;
  asm("mov.u32 %0, %%lanemask_lt;" : "=r"(lt));
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t v = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; v < n; v += nw) {
    const int32_t *o = gofs + v * C.ncls;
    const int32_t base = o[0];
    uint32_t at = didx[v];
    if (at == didx[v + 1]) continue;
    const int l = (vlab[v] - C.vl0) * C.ncls;
    for (int c0 = 0; c0 < C.ncls; c0 += 32) {
      const int c = c0 + lane;
      const int32_t a = c < C.ncls ? o[c] : 0, b = c < C.ncls ? o[c + 1] : 0;
      const uint32_t have = __ballot_sync(0xffffffffu, b > a);
      if (b > a) {
        dir[at - first + __popc(have & lt)] = make_int4(C.al0 + c / C.nvl, C.vl0 + c % C.nvl, a - base, b - base);
        atomicAdd(&h[l + c], 1u);
      }
      at += __popc(have);
    }
  }
  __syncthreads();
  for (int b = threadIdx.x; b < nbin; b += blockDim.x)
    if (h[b]) atomicAdd(cnt_of + b, h[b]);
}

// Exclusive prefix sums of the counts, one block per direction.
__global__ void __launch_bounds__(1024)
k_class_starts(const __grid_constant__ Direction D0, const __grid_constant__ Direction D1, int nbin) {
  const Direction &D = blockIdx.x ? D1 : D0;
  __shared__ uint32_t s_sum[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t run = 0;
  for (int b0 = 0; b0 <= nbin; b0 += 1024) {
    const int b = b0 + threadIdx.x;
    const uint32_t v = b < nbin ? D.cnt[b] : 0;
    uint32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) s_sum[warp] = x;
    __syncthreads();
    uint32_t before = run, all = 0;
    for (int w = 0; w < 32; ++w) {
      if (w < warp) before += s_sum[w];
      all += s_sum[w];
    }
    if (b <= nbin) D.start[b] = before + x - v;
    run += all;
    __syncthreads();
  }
}

// The vertices of each (vertex label, class) that have such a group: tiles of
// vertices, each reserving its part of every list, so that neighbours in a list
// stay neighbours in the graph.
constexpr int kClassTile = 256;

__global__ void __launch_bounds__(kThreads)
k_class_place(const __grid_constant__ Direction D0, const __grid_constant__ Direction D1,
              const int32_t *__restrict__ vlab, int32_t n, Classes C) {
  __shared__ uint32_t h[kMaxDense * kMaxDense];
  const Direction &D = blockIdx.y ? D1 : D0;
  const uint32_t first = D.didx[0];
  const int nbin = C.ncls * C.nvl, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = kThreads / 32;
  for (int64_t t0 = (int64_t)blockIdx.x * kClassTile; t0 < n; t0 += (int64_t)gridDim.x * kClassTile) {
    const int64_t t1 = min((int64_t)n, t0 + kClassTile);
    for (int b = threadIdx.x; b < nbin; b += kThreads) h[b] = 0;
    __syncthreads();
    for (int pass = 0; pass < 2; ++pass) {
      for (int64_t v = t0 + warp; v < t1; v += warps) {
        const int l = (vlab[v] - C.vl0) * C.ncls;
        const uint32_t end = D.didx[v + 1] - first;
        for (uint32_t e = D.didx[v] - first + lane; e < end; e += 32) {
          const int4 d = D.dir[e];
          const uint32_t at = atomicAdd(&h[l + class_of(C, d.x, d.y)], 1u);
          if (pass) D.vby[at] = (int32_t)v;
        }
      }
      __syncthreads();
      if (!pass) {
        for (int b = threadIdx.x; b < nbin; b += kThreads)
          if (h[b]) h[b] = D.start[b] + atomicAdd(D.cur + b, h[b]);
        __syncthreads();
      }
    }
  }
}

__device__ __forceinline__ void filter_insert(ArcKey k, uint32_t nword, unsigned long long *__restrict__ words) {
  const uint2 m = filter_bits(k);
  atomicOr(words + filter_word(k, nword), ((unsigned long long)m.y << 32) | m.x);
}

__global__ void k_filter(const int32_t *__restrict__ src, const int32_t *__restrict__ dst,
                         const int32_t *__restrict__ elab, int64_t m, uint32_t nword,
                         unsigned long long *__restrict__ words, const int *sort_err) {
  if (sort_failed(sort_err)) return;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < m;
       e += (int64_t)gridDim.x * blockDim.x) {
    const ArcKey h = pair_key(src[e], dst[e]);
    filter_insert(h, nword, words);
    filter_insert(labelled_key(h, elab[e]), nword, words);
  }
}

// The filter by endpoint, from rows sorted by that endpoint (column `key`): the
// words of consecutive rows lie together, so a block collects those of its tile in
// shared memory and writes the whole regions out; only the first and the last
// vertex may go on in another tile and take atomics.  A tile over more words than
// that (a hub, a run of isolated vertices) sets its bits in memory.  (All bits set
// in memory added 120 us to the load of 3.9M arcs; this way 16M arcs load in 5.04
// ms instead of 4.84 without the regions, 150M in 48.0 instead of 48.7.)
constexpr int kRegionTile = 2048, kRegionWords = 4096;

__global__ void __launch_bounds__(kThreads)
k_regions(const int4 *__restrict__ rows, int64_t m, int key, const int64_t *__restrict__ off,
          unsigned long long *__restrict__ words, const int *sort_err) {
  if (sort_failed(sort_err)) return;
  __shared__ uint2 s_word[kRegionWords];
  const int64_t ntile = (m + kRegionTile - 1) / kRegionTile;
  for (int64_t t = blockIdx.x; t < ntile; t += gridDim.x) {
    const int64_t first = t * kRegionTile, last = min(m, first + kRegionTile) - 1;
    const int32_t v0 = key ? rows[first].y : rows[first].x, v1 = key ? rows[last].y : rows[last].x;
    const Region g0 = region_of(v0, (uint32_t)off[v0], (uint32_t)(off[v0 + 1] - off[v0]));
    const Region g1 = region_of(v1, (uint32_t)off[v1], (uint32_t)(off[v1 + 1] - off[v1]));
    const uint32_t span = g1.base + g1.nword - g0.base;
    const bool local = span <= kRegionWords;
    if (local)
      for (uint32_t i = threadIdx.x; i < span; i += blockDim.x) s_word[i] = make_uint2(0, 0);
    __syncthreads();
    for (int64_t e = first + threadIdx.x; e <= last; e += blockDim.x) {
      const int4 r = rows[e];
      const int32_t v = key ? r.y : r.x;
      const int64_t o = off[v];
      const Region g = region_of(v, (uint32_t)o, (uint32_t)(off[v + 1] - o));
      const ArcKey pair = pair_key(r.x, r.y), both[2] = {pair, labelled_key(pair, r.z)};
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        if (local) {
          const uint2 b = filter_bits(both[k]);
          uint2 *w = &s_word[g.base - g0.base + filter_word(both[k], g.nword)];
          atomicOr(&w->x, b.x);
          atomicOr(&w->y, b.y);
        } else {
          filter_insert(both[k], g.nword, words + g.base);
        }
      }
    }
    __syncthreads();
    if (local)
      for (uint32_t i = threadIdx.x; i < span; i += blockDim.x) {
        const unsigned long long w = s_word[i].x | (unsigned long long)s_word[i].y << 32;
        unsigned long long *to = words + g0.base + i;
        if (i >= g0.nword && i < g1.base - g0.base) *to = w;
        else if (w) atomicOr(to, w);
      }
    __syncthreads();
  }
}

__global__ void k_hash(const int32_t *__restrict__ src, const int32_t *__restrict__ dst,
                       const int32_t *__restrict__ elab, int64_t m, uint32_t nbkt,
                       int4 *__restrict__ table, uint32_t *__restrict__ err, const int *sort_err) {
  if (sort_failed(sort_err)) return;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < m;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int32_t u = src[e], v = dst[e];
    const unsigned long long key = ((unsigned long long)(uint32_t)v << 32) | (uint32_t)u;
    uint32_t b = hash_bucket(pair_key(u, v), nbkt);
    bool placed = false;
    // at most every bucket once: the table has twice as many slots as arcs
    for (uint32_t it = 0; it < nbkt && !placed; ++it) {
      for (int s = 0; s < 2 && !placed; ++s) {
        int4 *slot = table + 2 * (size_t)b + s;
        const unsigned long long old =
            atomicCAS(reinterpret_cast<unsigned long long *>(slot), ~0ull, key);
        if (old == ~0ull) {
          slot->z = elab[e];
          placed = true;
        }
      }
      b = b + 1 == nbkt ? 0 : b + 1;
    }
    if (!placed) atomicOr(err, kErrHash);
  }
}

int grid_for(int64_t work) {
  int64_t g = (work + kThreads - 1) / kThreads;
  return (int)std::max<int64_t>(1, std::min<int64_t>(g, (int64_t)num_sms() * 16));
}

// An array of the graph's own (freed with it).
template <typename T>
cudaError_t own(hm_graph *g, T **p, int64_t count) {
  const cudaError_t e = cudaMalloc((void **)p, sizeof(T) * (size_t)std::max<int64_t>(count, 1));
  if (e == cudaSuccess) g->owned[g->nowned++] = *p;
  return e;
}

// Several arrays in one allocation, each on a 256-byte boundary: cudaMalloc and
// cudaFree cost 20 to 100 us each, and a graph has 19 arrays.
struct Arena {
  size_t bytes = 0;
  struct Part {
    void **p;
    size_t at;
  };
  std::vector<Part> parts;
  template <typename T>
  void add(T **p, int64_t count) {
    parts.push_back(Part{(void **)p, bytes});
    bytes += (sizeof(T) * (size_t)std::max<int64_t>(count, 1) + 255) / 256 * 256;
  }
  cudaError_t allocate(hm_graph *g) {
    unsigned char *base = nullptr;
    const cudaError_t e = own(g, &base, (int64_t)bytes);
    if (e == cudaSuccess)
      for (const Part &q : parts) *q.p = base + q.at;
    return e;
  }
};

void label_key(int32_t lo, int32_t hi, int *bits, uint32_t *xr) {
  if (lo >= 0 && hi < (1 << 24)) {
    *bits = bits_for((int64_t)hi + 1);
    *xr = 0;
  } else {
    *bits = 32;
    *xr = 0x80000000u;  // signed order as unsigned
  }
}

struct Temps {
  cudaStream_t s;
  std::vector<void *> p;
  explicit Temps(cudaStream_t st) : s(st) { p.reserve(16); }
  cudaError_t get(void **out, size_t bytes) {
    cudaError_t e = cudaMallocAsync(out, bytes ? bytes : 16, s);
    if (e == cudaSuccess) p.push_back(*out);
    return e;
  }
  ~Temps() {
    for (void *q : p) cudaFreeAsync(q, s);
  }
};

}  // namespace

void ensure_pool() {
  static thread_local int done_for = -1;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return;
  if (done_for == dev) return;
  cudaMemPool_t pool;
  if (cudaDeviceGetDefaultMemPool(&pool, dev) == cudaSuccess) {
    uint64_t thr = UINT64_MAX;
    cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &thr);
  }
  done_for = dev;
}

// Gives back what the current device's pool holds unused.
void trim_pool() {
  int dev = 0;
  cudaMemPool_t pool;
  if (cudaGetDevice(&dev) == cudaSuccess && cudaDeviceGetDefaultMemPool(&pool, dev) == cudaSuccess)
    cudaMemPoolTrimTo(pool, 0);
  (void)cudaGetLastError();
}

}  // namespace hm

using namespace hm;

namespace {

// Sort `rows` by (key column, arc label, neighbour label) -- rows arrive sorted by
// (key, neighbour), so stability keeps neighbours ascending inside each group --
// then write the grouped list and its directory.
hm_status build_groups(int32_t *rows, int32_t *tmp, int64_t m, int32_t n, int key, int other,
                       const int32_t *vlab, const int64_t *off, int nbits, int be, uint32_t xe,
                       int bv, uint32_t xv, cudaStream_t s, Temps &T, int32_t *gadj, hm_graph *g, int4 **dir,
                       int64_t *ndir, uint32_t **idx_out) {
  k_set_aux<<<grid_for(m), kThreads, 0, s>>>(rows, m, other, vlab);
  const int cols[3] = {key, 2, 3};
  const int bits[3] = {nbits, be, bv};
  const uint32_t xr[3] = {0u, xe, xv};
  hm_status st = radix_sort_rows_cols(rows, tmp, m, kW, cols, bits, xr, 3, s);
  if (st != HM_OK) return st;
  uint32_t *flags, *idx;
  HM_CUDA_TRY(T.get((void **)&flags, sizeof(uint32_t) * (size_t)(m + 1)));
  HM_CUDA_TRY(T.get((void **)&idx, sizeof(uint32_t) * (size_t)(m + 1)));
  k_group_flags<<<grid_for(m + 1), kThreads, 0, s>>>(rows, m, key, other, gadj, flags);
  st = exclusive_scan_u32(flags, idx, m + 1, s);
  if (st != HM_OK) return st;
  uint32_t total = 0;
  HM_CUDA_TRY(cudaMemcpyAsync(&total, idx + m, sizeof(uint32_t), cudaMemcpyDeviceToHost, s));
  HM_CUDA_TRY(cudaStreamSynchronize(s));
  *ndir = total;
  HM_CUDA_TRY(own(g, dir, (int64_t)total));
  k_group_entries<<<grid_for(m), kThreads, 0, s>>>(rows, m, key, flags, idx, off, *dir);
  *idx_out = idx;
  return HM_OK;
}

// What a graph gets beside the storage itself, as memory allows.
enum class Tables { kNone, kDense, kAll };  // kDense: without the filters by endpoint

hm_status load_graph_impl(int32_t n, int64_t m, const int32_t *src, const int32_t *dst,
                          const int32_t *vlab, const int32_t *elab, int device_ptrs,
                          cudaStream_t s, hm_graph *g, Tables tables) {
  Temps T(s);
#if HM_CHECK
  HM_CUDA_TRY(own(g, &g->check, 1));  // the bounds checks' violation word
  HM_CUDA_TRY(cudaMemsetAsync(g->check, 0, sizeof(unsigned long long), s));
#endif
  const int32_t *d_src = src, *d_dst = dst, *d_vlab = vlab, *d_elab = elab;
  if (!device_ptrs) {
    int32_t *t;
    HM_CUDA_TRY(T.get((void **)&t, sizeof(int32_t) * (size_t)(3 * m + n + 4)));
    if (m) {
      HM_CUDA_TRY(cudaMemcpyAsync(t, src, sizeof(int32_t) * m, cudaMemcpyHostToDevice, s));
      HM_CUDA_TRY(cudaMemcpyAsync(t + m, dst, sizeof(int32_t) * m, cudaMemcpyHostToDevice, s));
      HM_CUDA_TRY(cudaMemcpyAsync(t + 2 * m, elab, sizeof(int32_t) * m, cudaMemcpyHostToDevice, s));
    }
    if (n)
      HM_CUDA_TRY(cudaMemcpyAsync(t + 3 * m, vlab, sizeof(int32_t) * n, cudaMemcpyHostToDevice, s));
    d_src = t;
    d_dst = t + m;
    d_elab = t + 2 * m;
    d_vlab = t + 3 * m;
  }
  // working memory: rows and their copy, offsets, class counts, and if there may be dense offsets
  // groups per vertex and their prefix sums (both directions one after the other) and long lists
  int32_t *rows, *tmp, *hubs;
  int64_t *out_off, *in_off;
  uint32_t *err, *ngroup, *didx, *bins, *sizes;
  Bounds *bnd;
  {
    size_t at = 0;
    auto part = [&](size_t b) {
      const size_t a = at;
      at += (b + 255) / 256 * 256;
      return a;
    };
    const bool dense = tables != Tables::kNone;
    const size_t bin_words = 6 * (size_t)(kMaxDense * kMaxDense + 1);
    const size_t a_rows = part(sizeof(int32_t) * (size_t)(kW * m + kW)), a_tmp = part(sizeof(int32_t) * (size_t)(kW * m + kW)),
                 a_off = part(sizeof(int64_t) * 2 * (size_t)(n + 1)),
                 a_grp = part(dense ? sizeof(uint32_t) * 4 * (size_t)(n + 1) : 0),
                 a_hub = part(dense ? sizeof(int32_t) * 2 * (size_t)(m / kHub + 1) : 0),
                 a_zero = part(sizeof(uint32_t) * (bin_words + 4)), a_bnd = part(sizeof(Bounds)), a_sizes = part(sizeof(uint32_t) * 3);
    unsigned char *w;
    HM_CUDA_TRY(T.get((void **)&w, at));
    rows = reinterpret_cast<int32_t *>(w + a_rows);
    tmp = reinterpret_cast<int32_t *>(w + a_tmp);
    out_off = reinterpret_cast<int64_t *>(w + a_off);
    in_off = out_off + (n + 1);
    ngroup = reinterpret_cast<uint32_t *>(w + a_grp);
    didx = ngroup + 2 * (size_t)(n + 1);
    hubs = reinterpret_cast<int32_t *>(w + a_hub);
    err = reinterpret_cast<uint32_t *>(w + a_zero);  // {input errors, sort error}, then two list lengths, then the bins
    bins = err + 4;
    bnd = reinterpret_cast<Bounds *>(w + a_bnd);
    sizes = reinterpret_cast<uint32_t *>(w + a_sizes);
  }
  k_begin<<<1, 1, 0, s>>>(err, bnd);

  if (m) k_pack<<<grid_for(m), kThreads, 0, s>>>(d_src, d_dst, d_elab, m, n, rows, err, bnd);
  if (n) k_vbounds<<<grid_for(n), kThreads, 0, s>>>(d_vlab, n, bnd);
  uint32_t h_err = 0;
  Bounds hb;
  HM_CUDA_TRY(cudaMemcpyAsync(&h_err, err, sizeof(uint32_t), cudaMemcpyDeviceToHost, s));
  HM_CUDA_TRY(cudaMemcpyAsync(&hb, bnd, sizeof(Bounds), cudaMemcpyDeviceToHost, s));
  HM_CUDA_TRY(cudaStreamSynchronize(s));
  HM_CUDA_TRY(cudaGetLastError());
  if (h_err & kErrRange) return HM_ERR_ARG;
  if (h_err & kErrSelf) return HM_ERR_SELF_LOOP;

  // dense group offsets while there are few classes and the tables are no larger than the arcs' own data
  const int64_t nal = m ? (int64_t)hb.emax - hb.emin + 1 : 0, nvl = m ? (int64_t)hb.vmax - hb.vmin + 1 : 0;
  if (tables != Tables::kNone && m && nal <= kMaxDense && nvl <= kMaxDense && nal * nvl <= kMaxDense &&
      (int64_t)n * nal * nvl <= 8 * std::max<int64_t>(m, 1 << 16)) {
    g->nal = (int32_t)nal;
    g->nvl = (int32_t)nvl;
    g->al0 = hb.emin;
    g->vl0 = hb.vmin;
    g->ncls = (int32_t)(nal * nvl);
  }
  const Classes C{g->ncls, g->nvl, g->al0, g->vl0};
  g->afilt_nword = (uint32_t)(4 * std::max<int64_t>(1, (m + 7) / 8));
  g->ahash_nbkt = (uint32_t)std::max<int64_t>(1, m);
  const int64_t region_words = (m >> 1) + n + 1;
  g->regions = g->ncls && tables == Tables::kAll && m >= kRegionArcs;
  g->rf_nword = g->regions ? (uint32_t)region_words : g->afilt_nword;
  Arena A;
  A.add(&g->src, m);
  A.add(&g->out_adj, m);
  A.add(&g->out_elab, m);
  A.add(&g->in_adj, m);
  A.add(&g->in_elab, m);
  A.add(&g->gout_adj, m);
  A.add(&g->gin_adj, m);
  A.add(&g->vi, n);
  A.add(&g->off, n);
  A.add(&g->vdir, n);
  A.add(&g->afilt, (int64_t)g->afilt_nword);
  A.add(&g->ahash, 2 * (int64_t)g->ahash_nbkt);
  if (g->ncls) {
    A.add(&g->gofs_out, (int64_t)n * g->ncls + 1);
    A.add(&g->gofs_in, (int64_t)n * g->ncls + 1);
    if (g->regions) {
      A.add(&g->rfilt_out, region_words);
      A.add(&g->rfilt_in, region_words);
    }
  }
  HM_CUDA_TRY(A.allocate(g));
  if (!g->regions) g->rfilt_out = g->rfilt_in = g->afilt;
  HM_CUDA_TRY(cudaMemsetAsync(g->afilt, 0, 8 * (size_t)g->afilt_nword, s));
  HM_CUDA_TRY(cudaMemsetAsync(g->ahash, 0xff, 32 * (size_t)g->ahash_nbkt, s));

  const int nbits = bits_for(n);
  int be = 1, bv = 1;
  uint32_t xe = 0, xv = 0;
  if (m) label_key(hb.emin, hb.emax, &be, &xe);
  if (n) label_key(hb.vmin, hb.vmax, &bv, &xv);
  uint32_t *oidx = nullptr, *iidx = nullptr;
  std::vector<uint32_t> h_bins;
  const int nbin = g->ncls * g->nvl;
  int *sort_err = reinterpret_cast<int *>(err + 1);  // looked at by the kernels behind the sorts, then by the host
  if (m) {
    const int by_src[2] = {0, 1}, by_dst[2] = {1, 0}, bits[2] = {nbits, nbits};
    const uint32_t xr[2] = {0u, 0u};
    // (build_groups' kernels do not look at it: without dense offsets each sort is waited for)
    hm_status st = radix_sort_rows_cols(rows, tmp, m, kW, by_src, bits, xr, 2, s, nullptr, g->ncls ? sort_err : nullptr);
    if (st != HM_OK) return st;
    k_split<<<grid_for(m), kThreads, 0, s>>>(rows, m, n, 0, 1, g->src, g->out_adj, g->out_elab,
                                             out_off, err, sort_err);
    k_filter<<<grid_for(m), kThreads, 0, s>>>(g->src, g->out_adj, g->out_elab, m, g->afilt_nword,
                                              reinterpret_cast<unsigned long long *>(g->afilt), sort_err);
    k_hash<<<grid_for(m), kThreads, 0, s>>>(g->src, g->out_adj, g->out_elab, m, g->ahash_nbkt,
                                            g->ahash, err, sort_err);
    if (g->ncls) {
      // counts and cursors of both directions are zero; the starts follow them
      HM_CUDA_TRY(cudaMemsetAsync(err + 2, 0, sizeof(uint32_t) * (2 + 4 * (size_t)(nbin + 1)), s));
      uint32_t *nhub = err + 2;
      for (int in = 0; in < 2; ++in) {
        if (in) {
          // the rows are in (src, dst) order: sorted by dst alone they are in (dst, src) order
          st = radix_sort_rows_cols(rows, tmp, m, kW, by_dst, bits, xr, 1, s, nullptr, sort_err);
          if (st != HM_OK) return st;
          k_split<<<grid_for(m), kThreads, 0, s>>>(rows, m, n, 1, 0, nullptr, g->in_adj, g->in_elab, in_off, nullptr,
                                                   sort_err);
        }
        const int64_t *off = in ? in_off : out_off;
        if (g->regions) {
          uint2 *words = in ? g->rfilt_in : g->rfilt_out;
          HM_CUDA_TRY(cudaMemsetAsync(words, 0, sizeof(uint2) * (size_t)region_words, s));
          k_regions<<<grid_for(m), kThreads, 0, s>>>(reinterpret_cast<const int4 *>(rows), m, in, off,
                                                     reinterpret_cast<unsigned long long *>(words), sort_err);
        }
        const int32_t *adj = in ? g->in_adj : g->out_adj, *elab = in ? g->in_elab : g->out_elab;
        int32_t *gadj = in ? g->gin_adj : g->gout_adj, *gofs = in ? g->gofs_in : g->gofs_out;
        int32_t *list = hubs + (size_t)in * (m / kHub + 1);
        uint32_t *ng = ngroup + (size_t)in * (n + 1);
        k_group_lists<<<grid_for(32 * (int64_t)n), kThreads, 0, s>>>(off, adj, elab, d_vlab, n, m, C, gadj, gofs,
                                                                     ng, list, nhub + in, sort_err);
        k_group_hubs<<<(unsigned)std::min<int64_t>(m / kHub + 1, num_sms()), 1024, 0, s>>>(
            off, adj, elab, d_vlab, C, gadj, gofs, ng, list, nhub + in, sort_err);
      }
      st = exclusive_scan_u32(ngroup, didx, 2 * ((int64_t)n + 1), s);
      if (st != HM_OK) return st;
      oidx = didx;
      iidx = didx + (n + 1);
      k_dir_sizes<<<1, 1, 0, s>>>(oidx, iidx, n, sort_err, sizes);
      uint32_t h_sizes[3] = {0, 0, 0};
      HM_CUDA_TRY(cudaMemcpyAsync(h_sizes, sizes, sizeof(h_sizes), cudaMemcpyDeviceToHost, s));
      HM_CUDA_TRY(cudaStreamSynchronize(s));
      if (h_sizes[2]) return HM_ERR_CUDA;  // a sort failed: the sizes mean nothing
      g->ndir_out = h_sizes[0];
      g->ndir_in = h_sizes[1];
      Arena D;
      D.add(&g->gdir_out, g->ndir_out);
      D.add(&g->gdir_in, g->ndir_in);
      D.add(&g->vby_out, g->ndir_out);
      D.add(&g->vby_in, g->ndir_in);
      HM_CUDA_TRY(D.allocate(g));
    } else {
      st = build_groups(rows, tmp, m, n, 0, 1, d_vlab, out_off, nbits, be, xe, bv, xv, s, T,
                        g->gout_adj, g, &g->gdir_out, &g->ndir_out, &oidx);
      if (st != HM_OK) return st;
      st = radix_sort_rows(rows, tmp, m, kW, by_dst, 2, nbits, s);
      if (st != HM_OK) return st;
      k_split<<<grid_for(m), kThreads, 0, s>>>(rows, m, n, 1, 0, nullptr, g->in_adj, g->in_elab,
                                               in_off, nullptr, sort_err);
      st = build_groups(rows, tmp, m, n, 1, 0, d_vlab, in_off, nbits, be, xe, bv, xv, s, T,
                        g->gin_adj, g, &g->gdir_in, &g->ndir_in, &iidx);
      if (st != HM_OK) return st;
    }
  } else {
    k_zero_off<<<grid_for(n + 1), kThreads, 0, s>>>(out_off, n);
    k_zero_off<<<grid_for(n + 1), kThreads, 0, s>>>(in_off, n);
    HM_CUDA_TRY(own(g, &g->gdir_out, 1));
    HM_CUDA_TRY(own(g, &g->gdir_in, 1));
  }
  if (n)
    k_vertex<<<grid_for(n), kThreads, 0, s>>>(d_vlab, out_off, in_off, oidx, iidx, g->ncls > 0, n, g->vi, g->off,
                                              g->vdir, bnd);
  if (g->ncls) {
    h_bins.resize(2 * (size_t)(nbin + 1));
    Direction D[2];
    for (int in = 0; in < 2; ++in) {
      uint32_t *cnt = bins + in * (nbin + 1);
      D[in] = Direction{in ? g->gofs_in : g->gofs_out, in ? iidx : oidx, in ? g->gdir_in : g->gdir_out, cnt,
                        cnt + 2 * (nbin + 1), cnt + 4 * (nbin + 1), in ? g->vby_in : g->vby_out};
    }
    k_group_dirs<<<dim3(grid_for(16 * (int64_t)n), 2), kThreads, 0, s>>>(D[0], D[1], d_vlab, n, C);
    k_class_starts<<<2, 1024, 0, s>>>(D[0], D[1], nbin);
    k_class_place<<<dim3(grid_for((int64_t)n), 2), kThreads, 0, s>>>(D[0], D[1], d_vlab, n, C);
    HM_CUDA_TRY(cudaMemcpyAsync(h_bins.data(), bins + 4 * (nbin + 1), sizeof(uint32_t) * h_bins.size(),
                                cudaMemcpyDeviceToHost, s));
  }
  HM_CUDA_TRY(cudaMemcpyAsync(&h_err, err, sizeof(uint32_t), cudaMemcpyDeviceToHost, s));
  HM_CUDA_TRY(cudaMemcpyAsync(&hb, bnd, sizeof(Bounds), cudaMemcpyDeviceToHost, s));
  HM_CUDA_TRY(cudaStreamSynchronize(s));
  HM_CUDA_TRY(cudaGetLastError());
  g->maxdeg = hb.maxdeg;
  if (!h_bins.empty()) {
    g->vstart = (uint32_t *)malloc(sizeof(uint32_t) * h_bins.size());
    if (!g->vstart) return HM_ERR_OOM;
    std::memcpy(g->vstart, h_bins.data(), sizeof(uint32_t) * h_bins.size());
  }
  if (h_err & kErrDup) return HM_ERR_DUP_EDGE;
  if (h_err & kErrHash) return HM_ERR_CUDA;  // cannot happen (twice as many slots as arcs)
  g->bytes = sizeof(int32_t) * 7 * (size_t)m + (sizeof(int4) * 2 + sizeof(int2)) * (size_t)n +
             sizeof(int4) * (size_t)(g->ndir_out + g->ndir_in) + 8 * (size_t)g->afilt_nword +
             32 * (size_t)g->ahash_nbkt + (g->ncls ? sizeof(int32_t) * (2 * ((size_t)n * g->ncls + 1) + (size_t)(g->ndir_out + g->ndir_in)) +
                              (g->regions ? 2 * sizeof(uint2) * (size_t)region_words : 0)
                        : 0);
  return HM_OK;
}

void free_graph_arrays(hm_graph *g) {
  for (int i = 0; i < g->nowned; ++i) cudaFree(g->owned[i]);
}

}  // namespace

extern "C" hm_status hm_load_graph(int32_t n, int64_t m, const int32_t *src, const int32_t *dst,
                                   const int32_t *vlab, const int32_t *elab, int device_ptrs,
                                   void *stream, hm_graph **out) {
  if (!out || n < 0 || m < 0 || m > INT64_C(0x7FFFFFFF)) return HM_ERR_ARG;
  if (m > 0 && (!src || !dst || !elab)) return HM_ERR_ARG;
  if (n > 0 && !vlab) return HM_ERR_ARG;
  if (m > 0 && n == 0) return HM_ERR_ARG;
  int ndev = 0;
  if (cudaGetDeviceCount(&ndev) != cudaSuccess || ndev == 0) {
    (void)cudaGetLastError();
    return HM_ERR_NO_DEVICE;
  }
  ensure_pool();
  cudaStream_t s = (cudaStream_t)stream;
  hm_graph *g = new hm_graph();
  Tables tables = Tables::kAll;
  bool trimmed = false;
  for (;;) {
    std::memset(g, 0, sizeof(*g));
    cudaGetDevice(&g->device);
    g->n = n;
    g->m = m;
    hm_status st = load_graph_impl(n, m, src, dst, vlab, elab, device_ptrs, s, g, tables);
    if (st == HM_OK && cudaStreamSynchronize(s) != cudaSuccess) st = HM_ERR_CUDA;
    if (st == HM_OK) break;
    cudaStreamSynchronize(s);
    (void)cudaGetLastError();
    free_graph_arrays(g);
    free(g->vstart);
    // a device that is nearly full: once more with what the pool keeps given
    // back, then without the tables that only make searches faster (the dense
    // offsets and their vertex lists are up to 80 bytes per arc, the filters by
    // endpoint 8; without them calls search depth first)
    const bool regions = g->regions != 0;
    if (st == HM_ERR_OOM && !trimmed) {
      trimmed = true;
      trim_pool();
    } else if (st == HM_ERR_OOM && tables != Tables::kNone) {
      tables = regions ? Tables::kDense : Tables::kNone;
    } else {
      delete g;
      return st;
    }
  }
  *out = g;
  return HM_OK;
}

extern "C" void hm_free_graph(hm_graph *g) {
  if (!g) return;
  free_graph_arrays(g);
  free(g->vtab);
  free(g->etab);
  free(g->vstart);
  delete g;
}

extern "C" hm_status hm_check_status(const hm_graph *g, uint64_t *violation) {
  if (!g || !violation) return HM_ERR_ARG;
#if HM_CHECK
  unsigned long long w = 0;
  if (cudaMemcpy(&w, g->check, sizeof(w), cudaMemcpyDeviceToHost) != cudaSuccess ||
      cudaMemset(g->check, 0, sizeof(w)) != cudaSuccess)
    return HM_ERR_CUDA;
  *violation = w;
  return HM_OK;
#else
  *violation = 0;
  return HM_ERR_ARG;  // built without the bounds checks
#endif
}

extern "C" hm_status hm_graph_info(const hm_graph *g, int32_t *n, int64_t *m,
                                   size_t *device_bytes) {
  if (!g) return HM_ERR_ARG;
  if (n) *n = g->n;
  if (m) *m = g->m;
  if (device_bytes) *device_bytes = g->bytes;
  return HM_OK;
}

extern "C" hm_status hm_graph_export(const hm_graph *g, int64_t *out_off, int32_t *out_adj,
                                     int32_t *out_elab, int64_t *in_off, int32_t *in_adj,
                                     int32_t *in_elab) {
  if (!g) return HM_ERR_ARG;
  const size_t m = (size_t)g->m, n = (size_t)g->n;
  if (out_adj && m) HM_CUDA_TRY(cudaMemcpy(out_adj, g->out_adj, 4 * m, cudaMemcpyDeviceToHost));
  if (out_elab && m) HM_CUDA_TRY(cudaMemcpy(out_elab, g->out_elab, 4 * m, cudaMemcpyDeviceToHost));
  if (in_adj && m) HM_CUDA_TRY(cudaMemcpy(in_adj, g->in_adj, 4 * m, cudaMemcpyDeviceToHost));
  if (in_elab && m) HM_CUDA_TRY(cudaMemcpy(in_elab, g->in_elab, 4 * m, cudaMemcpyDeviceToHost));
  if (out_off || in_off) {
    int2 *h = (int2 *)malloc(sizeof(int2) * (n ? n : 1));
    if (!h) return HM_ERR_OOM;
    cudaError_t e = n ? cudaMemcpy(h, g->off, sizeof(int2) * n, cudaMemcpyDeviceToHost)
                      : cudaSuccess;
    if (e != cudaSuccess) {
      free(h);
      return HM_ERR_CUDA;
    }
    for (size_t v = 0; v < n; ++v) {
      if (out_off) out_off[v] = h[v].x;
      if (in_off) in_off[v] = h[v].y;
    }
    if (out_off) out_off[n] = (int64_t)m;
    if (in_off) in_off[n] = (int64_t)m;
    free(h);
  }
  return HM_OK;
}

extern "C" hm_status hm_graph_export_groups(const hm_graph *g, int32_t *gout_adj,
                                            int32_t *gin_adj, int32_t *vdir, int32_t *gdir_out,
                                            int32_t *gdir_in, int64_t *ndir) {
  if (!g) return HM_ERR_ARG;
  const size_t m = (size_t)g->m, n = (size_t)g->n;
  if (ndir) {
    ndir[0] = g->ndir_out;
    ndir[1] = g->ndir_in;
  }
  if (gout_adj && m) HM_CUDA_TRY(cudaMemcpy(gout_adj, g->gout_adj, 4 * m, cudaMemcpyDeviceToHost));
  if (gin_adj && m) HM_CUDA_TRY(cudaMemcpy(gin_adj, g->gin_adj, 4 * m, cudaMemcpyDeviceToHost));
  if (vdir && n) HM_CUDA_TRY(cudaMemcpy(vdir, g->vdir, sizeof(int4) * n, cudaMemcpyDeviceToHost));
  if (gdir_out && g->ndir_out)
    HM_CUDA_TRY(cudaMemcpy(gdir_out, g->gdir_out, sizeof(int4) * g->ndir_out, cudaMemcpyDeviceToHost));
  if (gdir_in && g->ndir_in)
    HM_CUDA_TRY(cudaMemcpy(gdir_in, g->gdir_in, sizeof(int4) * g->ndir_in, cudaMemcpyDeviceToHost));
  return HM_OK;
}
