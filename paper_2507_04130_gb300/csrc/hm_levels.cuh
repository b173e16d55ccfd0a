// hm_levels.cuh -- extension level by level (hm_levels.cu): what the host
// entry points pass to it and read back.
#pragma once

#include "hm_internal.cuh"

namespace hm {

// A condition of a level: Cons with the class (arc label, vertex label) whose
// group of f(q) holds the candidates, -1 if the graph has no such label.
struct LvCons {
  int8_t q, kind;
  int16_t cls;
  int32_t lab;
  uint64_t la, lb;  // the label's part of the two hashes of the arc filter
};

// What a candidate for one position must satisfy.
struct LevelPlan {
  int16_t npos, ncons;    // positive conditions first
  int8_t last;            // the position completes a match (but for a deferred position 1)
  int8_t need_deg;        // test the degrees: at least two pattern arcs lead to positions after the next
  int8_t root;            // the root mask applies to this position
  int8_t done;            // batch: the states of this level are matches already (two-vertex patterns)
  int32_t dout, din;
  uint32_t sym_gt, sym_lt;
  LvCons cons[kMaxCons];
};

// How a pattern's matches are written.
struct EmitPlan {
  int32_t k, naut;
  int32_t aut;            // first byte of its automorphisms in the table, kMaxK each
  int32_t orig[kMaxK];
};

// Control words of one call, zero at launch.
struct LvCtl {
  alignas(128) unsigned int bar;  // arrivals at the grid barrier
  alignas(128) int32_t status;
  alignas(128) unsigned int claim[3];                 // runs of chunks taken, one word per expansion in turn
  alignas(128) unsigned long long next_n[kMaxK + 2];  // states appended for each level
  alignas(128) unsigned long long count;              // matches
  unsigned long long rows;                            // row cursor
  unsigned long long chunks;                          // 32-candidate chunks examined
};

struct LvLaunch {
  const hm_graph *g;
  LvCtl *ctl;                        // device
  // depth-2 states: seeds, or (shared position-0 states) groups {u, first, end, 0} over sorted_seeds
  const int2 *seeds;
  const unsigned long long *nseeds;  // device
  int64_t max_seeds;
  const int4 *groups;
  const int2 *sorted_seeds;
  const uint8_t *root_mask;
  // one pattern: its plan (shared_plan's for shared states)
  const Plan *plan;
  int32_t *rows;
  unsigned long long cap;
  // a batch: `plans` (host) and, on the device, the pattern of each seed, counts and row regions
  int32_t npat;
  const Plan *plans;
  const int32_t *seed_pid;
  unsigned long long *counts;
  const unsigned long long *row_off, *row_cap;
  unsigned long long *row_cursor;
  bool want_rows;
  uint64_t workspace;                // bytes it may take for the levels
};

constexpr uint64_t kLevelWorkspace = 256ull << 20;

// Runs the extension of a call.  *ran is false, and nothing was launched, when
// the graph has no dense group offsets or the device cannot hold the grid.
hm_status levels_run(const LvLaunch &L, cudaStream_t s, bool *ran, int *grid, int *threads);

}  // namespace hm
