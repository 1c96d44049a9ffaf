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

// Flags a call reads back from the device.
struct CallFlags {
    int32_t bad_seed, limit, timed_out, pad;
    unsigned long long t0;  // global timer (ns) of the call's first step
};

// True if a call of `trials` trials in all runs in the column engine.
bool columns_fit(int model, const cnd_graph_dev &G, const cnd_sim_opts &o, int64_t trials);

// Runs the items' trials.  spread (null: not wanted), count (rows of n, zeroed, or null), checks and
// level_counts (zeroed) and flags (zeroed) are device memory; temporaries come from the stream-ordered
// pool and are freed on the stream.  The caller synchronises and reads flags.
cnd_status run_columns(int model, const cnd_graph_dev &G, const std::vector<ItemDesc> &items, const int32_t *seeds_dev,
                       int32_t *spread, int32_t *count, unsigned long long *checks, unsigned long long *level_counts,
                       CallFlags *flags, const cnd_sim_opts &o, cudaStream_t st);

}  // namespace cnd
