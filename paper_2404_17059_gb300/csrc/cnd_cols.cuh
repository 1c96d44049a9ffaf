// Column engine for graphs whose per-trial state fits shared memory (cnd_cols.cu).
#pragma once

#include <vector>

#include "cnd_common.cuh"

namespace cnd {

// One simulation problem: a seed set, a trial count and a Philox key.
struct ItemDesc {
    int64_t seed_begin, seed_end;  // range in the seed array
    int64_t trials;
    int64_t out0;                  // position of its first trial in the spread output
    uint64_t key;
};

// What a call reads back from the device beside its outputs.
struct CallFlags {
    int32_t bad_seed, limit, timed_out;
    int32_t next_column;    // columns handed out (column engine)
    unsigned long long t0;  // global timer (ns) of the call's first step
    unsigned long long checks;
};

// A call of the column engine: its items as the device reads them, and the scratch it needs.
struct ColPlan {
    std::vector<unsigned char> items;
    size_t scratch = 0;  // bytes
    int32_t n_items = 0, bits = 0, cols = 0, blocks = 0, threads = 0, cap = 0;
    size_t dyn = 0, over = 0;
};

// True if a call of `trials` trials in all, in `words` words of 64 of the same item, runs in the column engine.
bool columns_fit(int model, const cnd_graph_dev &G, const cnd_sim_opts &o, int64_t trials, int64_t words);

// The trials of a column of such a call.
int32_t column_bits(int model, const cnd_graph_dev &G, int64_t trials);

cnd_status plan_columns(int model, const cnd_graph_dev &G, const std::vector<ItemDesc> &items, ColPlan &plan);

// Runs the items' trials.  items: plan.items on the device; scratch: plan.scratch bytes, 16-byte aligned.
// spread (null: not wanted), count (rows of n, zeroed, or null), checks and level_counts (zeroed) and flags
// (zeroed) are device memory.  Every trial's spread is written.  The caller synchronises and reads flags.
cnd_status run_columns(int model, const cnd_graph_dev &G, const ColPlan &plan, const void *items, void *scratch,
                       const int32_t *seeds_dev, int32_t *spread, int32_t *count, unsigned long long *checks,
                       unsigned long long *level_counts, CallFlags *flags, const cnd_sim_opts &o, cudaStream_t st);

}  // namespace cnd
