// Launch plans of the attention calls: which kernel takes which sequences of a batch, how their KV is split and how the splits are merged.
// Host code without CUDA calls.
#pragma once
#include <vector>

#include "agx.h"
#include "agx_internal.cuh"

namespace agx {

// What the planner needs to know, and its knobs (environment variables, read when a handle is created).
struct PlanConfig {
    int num_q_heads, num_kv_heads, head_dim, dtype;
    int sm_count;
    int (*max_clusters)(int mt, int kw, int cluster);   // attn_small_max_clusters
    int small_min_split;    // tokens (env AGX_SMALL_MIN_SPLIT)
    int force_mma_sync;     // route large q through the mma.sync kernel (env AGX_FORCE_MMA_SYNC)
    int debug_plan;         // print launch plans to stderr (env AGX_DEBUG_PLAN)
    int small_kw;           // pages per pipeline stage of the warp-MMA kernel: 4, 8, or 0 = chosen per batch (env AGX_SMALL_KW)
    int batch_stream_tokens; // total tokens of a batch's small blocks from which they all take the stream schedule (env AGX_BATCH_STREAM_TOKENS)
    bool longest_first;     // sequences of a launch ordered by decreasing context length (env AGX_LONGEST_FIRST=0: batch order)
    bool merge_sms;         // one-wave small-q launches leave SMs free for their merge kernel (env AGX_MERGE_SMS=0 turns it off)
    int cluster_merge;      // KV splits of the small-q kernel merged inside thread-block clusters: 1 = where the batch allows and it is the faster merge,
                            // 2 = wherever the batch allows (env AGX_CLUSTER_MERGE=1), 0 = never (AGX_CLUSTER_MERGE=0)
    int stream_max_rows;    // blocks of up to this many rows per KV head may take the one-Q-tile schedule in 128-row chunks (env AGX_STREAM_MAX_ROWS)
    bool stream_rows_estimated;   // (that variable not set) one block of more than 64 rows only where the estimates of both schedules say so
    int stream_min_tokens;  // context length from which blocks of <= 32 rows take the tensor-core stream schedule (env AGX_STREAM_MIN_TOKENS; -1 = by
                            // the estimates of both kernels)
};
PlanConfig plan_config(const agx_config& cfg, int sm_count, int (*max_clusters)(int mt, int kw, int cluster));

enum Kind { KIND_SMALL1 = 0, KIND_SMALL2, KIND_SMALL4, KIND_STREAM, KIND_TILE, KIND_SIMT, KIND_COUNT };

struct Launch {
    Kind kind;
    int total_rows;  // sum of q_len over the launch's sequences
    int num_items;
    int kw;          // small-q kernel: pages per pipeline stage (KV groups), 4 or 8
    int cluster;     // > 1: CTAs per cluster = KV splits of every sequence of the launch, merged in-kernel (no partials)
    bool lean_merge; // small-q kernel or one-Q-tile schedule: one wave, its merge on SMs left out of the attention grid
    bool f32_partials = false;   // 256-row schedule: fp32 partials
    std::vector<SeqPlan> seqs;
};

struct Plan {
    std::vector<Launch> launches;
    long long part_entries = 0;  // (row, head, split) partial slots
    bool any_split = false;
    bool tensor_core = false;    // a launch of the tensor-core kernel is among them
    long long total_rows = 0;    // block rows of the whole batch
};

// Decide kernel kind, KV splits and partial slots for every sequence (host lengths only; pt_stride < 0: the page table is not known yet).
// On failure a text for the caller is left in `err`.
agx_status build_plan(const PlanConfig& c, int B, const int32_t* P, const int32_t* Q, int pt_stride, Plan& plan, char* err, size_t err_bytes);

}  // namespace agx
