// hm_levels.cuh -- matching level by level (hm_levels.cu): what the host entry
// points pass to it and read back.
#pragma once

#include "hm_internal.cuh"

namespace hm {

// Control words of one call, zero at launch.  Words that phases in turn use
// come in threes: the one of the next turn is cleared while this one is used.
struct LvCtl {
  alignas(128) unsigned int bar;  // arrivals at the grid barrier
  alignas(128) int32_t status;
  alignas(128) unsigned int paused[3];                // warps that stopped because the next level was full
  alignas(128) unsigned int claim[kMaxK + 1][3];      // runs of chunks taken, per level
  alignas(128) unsigned long long made[kMaxK + 1][3]; // groups << 40 | chunks of each level
  alignas(128) unsigned long long count;              // matches
  unsigned long long rows;                            // row cursor
  unsigned long long chunks;                          // 32-candidate chunks examined
  unsigned long long injected;                        // states with two mapped positions
};

struct LvLaunch {
  const hm_graph *g;
  const uint8_t *root_mask;  // device; applies to the plan's root_pos
  bool want_rows;
  int32_t *rows;             // device
  uint64_t workspace;        // bytes the states of the levels may take
  // one pattern
  const Plan *plan;
  uint64_t cap;
  bool defer;                // position 1 is matched last (the plan's defer1)
  // a batch: `plans` (host), counts and row regions (device)
  int32_t npat;
  const Plan *const *plans;
  unsigned long long *counts, *counts_host;  // counts_host: read back when the call is done
  const unsigned long long *row_off, *row_cap;
  unsigned long long *row_cursor;
};

// What a call's levels may take.  A level that does not fit is worked off in
// parts; each part costs a barrier per deeper level and begins and ends with
// idle warps, so a part should hold some hundred states per warp.  With 64 bytes
// per arc alone a 7-cycle on 564,000 arcs had 20 and took 37,000 phases (1,278 ms;
// with 256 MB 386, with 1 GiB 278; depth first 375), an induced star of seven on
// 166,000 arcs 933 ms (1 GiB 107; depth first 220), an induced path of five on
// 18,600 arcs 23.4 ms (14.4 from 64 MB on; depth first 9.4, 4.7 with more blocks).
// 128 MB for every level that keeps states, beside the first, is near the end of
// that for all of them.  It stays in the device's pool: the first search of a
// process takes about 0.1 ms longer for every 256 MB, the following ones nothing.
// A level gets no more groups than the graph has arcs (at least 8,192), or than a
// guess at the call's candidates asks for, so short calls on small graphs take a few MB.
constexpr uint64_t kLevelWorkspaceMax = 1ull << 30;
constexpr uint64_t kLevelWorkspacePer = 128ull << 20;
constexpr uint64_t kLevelWorkspaceMin = 8ull << 20;  // on a device that is nearly full
inline uint64_t level_workspace(const hm_graph *g, int k) {
  const uint64_t arcs = 64 * (uint64_t)g->m, levels = kLevelWorkspacePer * (uint64_t)(k > 3 ? k - 2 : 1);
  const uint64_t w = arcs > levels ? arcs : levels;
  return w > kLevelWorkspaceMax ? kLevelWorkspaceMax : w;
}

// Runs a whole call, from the vertices that may be position 0's images to the
// counts and (unsorted) rows, and waits for it.  *ran is false, and nothing was
// launched, when the device cannot hold the grid.  Needs dense group offsets
// (g->ncls > 0).
// Measured, whole searches, depth first (edge scan and extension) / level by
// level: R-MAT scale 20, induced, with rows, feed-forward loop 2.36 / 0.66 ms,
// bi-fan 7.57 / 3.74, 4-cycle 4.67 / 1.89; 150M arcs, five motifs 1.2 to 3.6 /
// 0.15 to 0.34 ms each.  27 of 32 lanes work (15), issue slots are 42 to 47 %
// busy, 57 to 60 % of the reads hit L2, DRAM runs at 0.19 of the copy rate.
hm_status levels_run(const LvLaunch &L, cudaStream_t s, bool *ran, LvCtl *result, int *grid, int *threads,
                     float *ms);

}  // namespace hm
