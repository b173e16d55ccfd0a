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

// What a call's levels may take: as much as the graph's arrays do (about 80
// bytes per arc) at most, and no more than 1 GiB.  A level that does not fit is
// worked off in parts, at 20 to 40 us each.
constexpr uint64_t kLevelWorkspaceMax = 1ull << 30;
constexpr uint64_t kLevelWorkspaceMin = 8ull << 20;
inline uint64_t level_workspace(const hm_graph *g) {
  const uint64_t w = 64 * (uint64_t)g->m;
  return w < kLevelWorkspaceMin ? kLevelWorkspaceMin : w > kLevelWorkspaceMax ? kLevelWorkspaceMax : w;
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
