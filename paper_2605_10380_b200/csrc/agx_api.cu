// C ABI of the agx library: argument checks, dispatch.  No kernel lives here; what is launched is planned in agx_plan.cu.
#include <stdarg.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <exception>
#include <new>
#include <vector>

#include <nvtx3/nvToolsExt.h>

#include "agx_internal.cuh"
#include "agx_plan.cuh"

namespace {
// An NVTX range around every call that enqueues work: a timeline tool shows the library's calls by name; with no tool
// attached a range costs a few nanoseconds.
struct CallRange {
    explicit CallRange(const char* name) { nvtxRangePushA(name); }
    ~CallRange() { nvtxRangePop(); }
};
}  // namespace

struct agx_handle {
    agx_config cfg;
    float scale;
    int device;
    int sm_count;
    int* d_status;          // device status word
    unsigned int* d_ticket; // ticket counter of the accept kernel (self-resetting)
    unsigned long long* d_row_keys;   // one argmax key per logits row of the accept kernel (all zero between launches)
    int last_launches;
    int zero_copy;          // host steps: bit 0 = kernels read small pinned inputs, bit 1 = kernels write `out` into a pinned buffer (env AGX_ZERO_COPY, default 3)
    agx::PlanConfig plan;   // what the planner needs to know, and its knobs
    long long wait_limit_cycles;   // AGX_OPT_WAIT_LIMIT_CYCLES
    int early_prefix;       // AGX_OPT_EARLY_PREFIX_LOADS
    int drop_stage;         // AGX_OPT_TEST_DROP_STAGE (-1 = none)
    std::vector<int32_t> cu_host;  // staging for agx_verify_step_host (lives until its final sync)
    // Large attention-only host steps run as a pipeline of row chunks: uploads on one stream of the handle's own, the
    // attention calls on the caller's stream, downloads on a third (env AGX_HOST_PIPELINE_ROWS: rows per chunk, 0 = off).
    int pipe_rows;
    cudaStream_t pipe_in, pipe_out;
    std::vector<cudaEvent_t> pipe_events;
    // The launch plans of the last batches seen: the layers of a model step all ask for the same one, those of a pipelined host step for one per chunk.
    static constexpr int kPlans = 16;
    struct CachedPlan {
        agx::Plan plan;
        std::vector<int32_t> P, Q;   // empty: no plan
    } plans[kPlans];
    int plan_last;                   // the one used last
    char err[512];
};

namespace {

using namespace agx;

agx_status fail(agx_handle* h, agx_status code, const char* fmt, ...) {
    if (h) {
        va_list ap;
        va_start(ap, fmt);
        vsnprintf(h->err, sizeof h->err, fmt, ap);
        va_end(ap);
    }
    return code;
}

agx_status cuda_fail(agx_handle* h, cudaError_t e, const char* what) {
    return fail(h, AGX_E_CUDA, "%s: %s", what, cudaGetErrorString(e));
}

inline bool aligned(const void* p, size_t a) { return ((uintptr_t)p % a) == 0; }

inline int elem_size(int dtype) { return dtype == AGX_BF16 ? 2 : 4; }

// The plan for this batch: a cached one when the lengths are those of one of the last calls on the handle.
agx_status make_plan(agx_handle* h, int B, const int32_t* P, const int32_t* Q, int pt_stride, const Plan*& out) {
    for (int i = 0; i < agx_handle::kPlans; ++i) {
        const int at = (h->plan_last + agx_handle::kPlans - i) % agx_handle::kPlans;
        const agx_handle::CachedPlan& e = h->plans[at];
        if ((int)e.P.size() != B || memcmp(e.P.data(), P, sizeof(int32_t) * B) != 0 || memcmp(e.Q.data(), Q, sizeof(int32_t) * B) != 0) continue;
        if (pt_stride >= 0)
            for (int s = 0; s < B; ++s)
                if ((long long)P[s] + Q[s] > (long long)pt_stride * kPage)
                    return fail(h, AGX_E_RANGE, "sequence %d: %d + %d tokens exceed the page table (%d pages)", s, P[s], Q[s], pt_stride);
        h->plan_last = at;
        out = &e.plan;
        return AGX_OK;
    }
    const int at = (h->plan_last + 1) % agx_handle::kPlans;   // (round robin)
    agx_handle::CachedPlan& e = h->plans[at];
    e.P.clear();   // (invalid while it is rebuilt)
    try {
        e.plan = Plan();
        agx_status st = build_plan(h->plan, B, P, Q, pt_stride, e.plan, h->err, sizeof h->err);
        if (st != AGX_OK) return st;
        e.Q.assign(Q, Q + B);
        e.P.assign(P, P + B);
    } catch (const std::exception&) {   // (no exception leaves a C entry)
        e.P.clear();
        return fail(h, AGX_E_NOMEM, "out of host memory for the plan of %d sequences", B);
    }
    h->plan_last = at;
    out = &e.plan;
    return AGX_OK;
}

// Split partials: (max, sum) of every entry, the rows, and the exponents of rows beyond fp16's range.
inline size_t part_ml_bytes(long long entries) { return (size_t)((entries * sizeof(float2) + 255) / 256 * 256); }
inline size_t part_bytes(long long entries, int head_dim) {
    return entries == 0 ? 0 : part_ml_bytes(entries) + (size_t)entries * head_dim * sizeof(float) + (size_t)(entries + 255) / 256 * 256;
}

}  // namespace

extern "C" {

const char* agx_status_string(agx_status s) {
    switch (s) {
        case AGX_OK: return "ok";
        case AGX_E_INVAL: return "invalid argument";
        case AGX_E_RANGE: return "argument out of range";
        case AGX_E_UNSUPPORTED: return "unsupported configuration";
        case AGX_E_CUDA: return "CUDA error";
        case AGX_E_DEVICE: return "device status word set";
        case AGX_E_NOMEM: return "out of memory";
        default: return "unknown status";
    }
}

const char* agx_last_error(const agx_handle* h) { return h ? h->err : "null handle"; }

agx_status agx_create(const agx_config* cfg, agx_handle** out) {
    if (!cfg || !out) return AGX_E_INVAL;
    *out = nullptr;
    if (cfg->num_q_heads < 1 || cfg->num_kv_heads < 1 || cfg->num_q_heads % cfg->num_kv_heads != 0) return AGX_E_INVAL;
    if (cfg->page_size != kPage) return AGX_E_UNSUPPORTED;
    if (cfg->dtype != AGX_BF16 && cfg->dtype != AGX_F32) return AGX_E_UNSUPPORTED;
    if (cfg->dtype == AGX_BF16 && cfg->head_dim != 128 && cfg->head_dim != 64) return AGX_E_UNSUPPORTED;
    if (cfg->dtype == AGX_F32 && cfg->head_dim != 64 && cfg->head_dim != 128) return AGX_E_UNSUPPORTED;
    if (!(cfg->scale >= 0.f)) return AGX_E_INVAL;
    agx_handle* h = new (std::nothrow) agx_handle();
    if (!h) return AGX_E_NOMEM;
    h->cfg = *cfg;
    h->scale = cfg->scale > 0.f ? cfg->scale : 1.0f / sqrtf((float)cfg->head_dim);
    h->err[0] = 0;
    h->last_launches = 0;
    const char* env;
    env = getenv("AGX_HOST_PIPELINE_ROWS");
    h->pipe_rows = env ? std::max(0, atoi(env)) : 384;   // measured on the long-context step: 256 / 384 / 512 / 768 / 1024 rows -> 1.54 / 1.43 / 1.57 / 1.56 / 1.72 ms
    h->pipe_in = h->pipe_out = nullptr;
    env = getenv("AGX_ZERO_COPY");
    h->zero_copy = env ? atoi(env) : 3;
    h->wait_limit_cycles = kWaitLimitCycles;
    env = getenv("AGX_EARLY_PREFIX");
    h->early_prefix = env ? atoi(env) : 0;
    h->drop_stage = -1;
    cudaError_t e = cudaGetDevice(&h->device);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&h->sm_count, cudaDevAttrMultiProcessorCount, h->device);
    int major = 0;
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, h->device);
    if (e == cudaSuccess && major != 10) { delete h; return AGX_E_UNSUPPORTED; }
    constexpr size_t kStateBytes = 256 + 65536 * 8;   // status word and accept ticket | one key per logits row (at most 65535)
    if (e == cudaSuccess) e = cudaMalloc((void**)&h->d_status, kStateBytes);
    if (e != cudaSuccess) { delete h; return e == cudaErrorMemoryAllocation ? AGX_E_NOMEM : AGX_E_CUDA; }
    e = cudaMemset(h->d_status, 0, kStateBytes);
    if (e != cudaSuccess) { cudaFree(h->d_status); delete h; return AGX_E_CUDA; }
    h->plan = plan_config(h->cfg, h->sm_count, attn_small_max_clusters);
    h->d_ticket = (unsigned int*)(h->d_status + 16);
    h->d_row_keys = (unsigned long long*)(h->d_status + 64);
    *out = h;
    return AGX_OK;
}

agx_status agx_destroy(agx_handle* h) {
    if (!h) return AGX_E_INVAL;
    cudaFree(h->d_status);
    if (h->pipe_in) cudaStreamDestroy(h->pipe_in);
    if (h->pipe_out) cudaStreamDestroy(h->pipe_out);
    for (cudaEvent_t ev : h->pipe_events) cudaEventDestroy(ev);
    delete h;
    return AGX_OK;
}

agx_status agx_kv_append(agx_handle* h, void* k_pool, void* v_pool, int64_t num_pages, const void* k_new,
                         const void* v_new, const int32_t* page_table, int32_t pt_stride, const int32_t* prefix_len,
                         const int32_t* cu_q, int32_t B, int32_t total_q, void* stream) {
    CallRange range_("agx_kv_append");
    if (!h) return AGX_E_INVAL;
    h->last_launches = 0;
    if (B < 0 || total_q < 0) return fail(h, AGX_E_INVAL, "negative B or total_q");
    if (B == 0 || total_q == 0) return AGX_OK;
    if (!k_pool || !v_pool || !k_new || !v_new || !page_table || !prefix_len || !cu_q)
        return fail(h, AGX_E_INVAL, "null pointer");
    if (!aligned(k_pool, 16) || !aligned(v_pool, 16) || !aligned(k_new, 16) || !aligned(v_new, 16))
        return fail(h, AGX_E_INVAL, "K/V buffers must be 16-byte aligned");
    if (num_pages < 1 || pt_stride < 1) return fail(h, AGX_E_INVAL, "num_pages and page_table_stride must be >= 1");
    cudaError_t e = launch_kv_append(h->cfg.dtype, k_pool, v_pool, num_pages, k_new, v_new, page_table, pt_stride,
                                     prefix_len, cu_q, B, total_q, h->cfg.num_kv_heads, h->cfg.head_dim, h->d_status,
                                     (cudaStream_t)stream);
    if (e != cudaSuccess) return cuda_fail(h, e, "kv_append launch");
    h->last_launches = 1;
    return AGX_OK;
}

int64_t agx_attn_workspace_bytes(agx_handle* h, int32_t B, const int32_t* P, const int32_t* Q) {
    if (!h) return AGX_E_INVAL;
    if (B < 0) return fail(h, AGX_E_INVAL, "negative B");
    if (B == 0) return 0;
    if (!P || !Q) return fail(h, AGX_E_INVAL, "null pointer");
    const Plan* plan_ptr = nullptr;
    agx_status st = make_plan(h, B, P, Q, -1, plan_ptr);
    if (st != AGX_OK) return st;
    const Plan& plan = *plan_ptr;
    if (plan.part_entries == 0) return 0;
    return (int64_t)part_bytes(plan.part_entries, h->cfg.head_dim);
}

// Attention, optionally with the append of the block's own K/V rows (k_new != NULL): the attention kernels take the block's rows from
// k_new / v_new and store them into the pages on the side.  Launches of the warp-MMA kernel with more than one row chunk, which only
// AGX_FORCE_MMA_SYNC makes, get a separate append launch in front.
static agx_status attn_impl(agx_handle* h, const void* q_block, const void* k_new, const void* v_new, const void* k_pool,
                            const void* v_pool, int64_t num_pages, const int32_t* page_table, int32_t pt_stride,
                            const int32_t* P, const int32_t* Q, int32_t B, void* out, float* lse, void* workspace,
                            size_t workspace_bytes, void* stream_v, bool early_prefix) {
    CallRange range_("agx_attn_prefixed");
    if (!h) return AGX_E_INVAL;
    h->last_launches = 0;
    if (B < 0) return fail(h, AGX_E_INVAL, "negative B");
    if (B == 0) return AGX_OK;
    if (!q_block || !k_pool || !v_pool || !page_table || !P || !Q || !out) return fail(h, AGX_E_INVAL, "null pointer");
    if (k_new && (!v_new || !aligned(k_new, 16) || !aligned(v_new, 16)))
        return fail(h, AGX_E_INVAL, "k_new/v_new must both be given and 16-byte aligned");
    if (!aligned(q_block, 16) || !aligned(out, 16) || !aligned(k_pool, 256) || !aligned(v_pool, 256))
        return fail(h, AGX_E_INVAL, "q_block/out must be 16-byte and pools 256-byte aligned");
    if (num_pages < 1 || pt_stride < 1) return fail(h, AGX_E_INVAL, "num_pages and page_table_stride must be >= 1");
    const Plan* plan_ptr = nullptr;
    agx_status st = make_plan(h, B, P, Q, pt_stride, plan_ptr);
    if (st != AGX_OK) return st;
    const Plan& plan = *plan_ptr;
    const size_t need = part_bytes(plan.part_entries, h->cfg.head_dim);
    if (need > 0) {
        if (!workspace || !aligned(workspace, 256)) return fail(h, AGX_E_INVAL, "workspace missing or not 256-byte aligned");
        if (workspace_bytes < need) return fail(h, AGX_E_INVAL, "workspace too small: %zu < %zu", workspace_bytes, need);
    }
    cudaStream_t stream = (cudaStream_t)stream_v;
    AttnParams p;
    memset(&p, 0, sizeof p);
    p.q = q_block; p.k_pool = k_pool; p.v_pool = v_pool; p.page_table = page_table;
    p.out = out; p.lse = lse;
    p.part_ml = (float2*)workspace;
    p.part_o = need ? (float*)((char*)workspace + part_ml_bytes(plan.part_entries)) : nullptr;
    p.part_exp = need ? (signed char*)(p.part_o + plan.part_entries * h->cfg.head_dim) : nullptr;
    p.status = h->d_status;
    p.num_pages = num_pages;
    p.total_rows = (int)plan.total_rows;
    p.pt_stride = pt_stride;
    p.hq = h->cfg.num_q_heads; p.hkv = h->cfg.num_kv_heads; p.head_dim = h->cfg.head_dim;
    p.scale_log2 = h->scale * 1.4426950408889634f;
    p.gqa = p.hq / p.hkv;
    p.row_div_magic = (0x100000000ull + (unsigned)p.gqa - 1) / (unsigned)p.gqa;
    p.row_div_shift = 31;
    while ((1ll << (p.row_div_shift - 31)) < p.gqa) ++p.row_div_shift;
    p.row_div31 = (unsigned)(((1ull << p.row_div_shift) + (unsigned)p.gqa - 1) / (unsigned)p.gqa);
    p.wait_limit_cycles = h->wait_limit_cycles;
    p.early_prefix = early_prefix;
    p.drop_stage = h->drop_stage;
    alignas(64) CUtensorMap map_k, map_v;   // (encoding one takes 0.05 us)
    RowsMaps maps_new;
    if (h->cfg.dtype == AGX_BF16 && h->cfg.head_dim == 128) {
        if ((long long)num_pages * p.hkv * kPage > 0x7FFFFFFFll) return fail(h, AGX_E_RANGE, "pool too large for one tensor map");
        bool ok = make_pool_map(&map_k, k_pool, num_pages, p.hkv) && make_pool_map(&map_v, v_pool, num_pages, p.hkv);
        if (ok && k_new && plan.tensor_core) ok = make_rows_maps(&maps_new, k_new, v_new, plan.total_rows, k_pool, v_pool, num_pages, p.hkv);
        else if (plan.tensor_core) memset(&maps_new, 0, sizeof maps_new);
        if (!ok) return fail(h, AGX_E_CUDA, "cuTensorMapEncodeTiled failed");
    }
    for (const Launch& ln : plan.launches) {
        p.num_seqs = (int)ln.seqs.size();
        p.num_items = ln.num_items;
        bool split = false;
        bool one_chunk = true;
        for (int i = 0; i < p.num_seqs; ++i) {
            p.seq[i] = ln.seqs[i];
            split |= ln.seqs[i].nsplit > 1 && !ln.cluster;
            one_chunk &= ln.seqs[i].row_chunks == 1;
        }
        cudaError_t e;
        p.cluster_size = ln.cluster;
        p.part_half = ln.kind != KIND_TILE ? PART_F32 : ln.f32_partials ? PART_F32_TILES : PART_HALF_TILES;
        p.k_new = p.v_new = nullptr;
        if (k_new) {
            p.k_new = k_new; p.v_new = v_new;
            if (!one_chunk && ln.kind != KIND_TILE && ln.kind != KIND_STREAM && ln.kind != KIND_SIMT) {
                e = launch_kv_append_plan(p, h->cfg.dtype, ln.total_rows, stream);
                if (e != cudaSuccess) return cuda_fail(h, e, "append launch");
                h->last_launches++;
                p.k_new = p.v_new = nullptr;
            }
        }
        switch (ln.kind) {
            case KIND_SMALL1: e = launch_attn_small_bf16(p, 1, ln.kw, map_k, map_v, stream); break;
            case KIND_SMALL2: e = launch_attn_small_bf16(p, 2, ln.kw, map_k, map_v, stream); break;
            case KIND_SMALL4: e = launch_attn_small_bf16(p, 4, 4, map_k, map_v, stream); break;
            case KIND_SIMT: e = launch_attn_simt(p, h->cfg.dtype, stream); break;
            case KIND_TILE:
            case KIND_STREAM: {
                // Q boxes: as many tokens as a 128-row tile holds from any row on, and no more than a block of the launch has
                int longest = 1;
                for (const SeqPlan& sp : ln.seqs) longest = std::max(longest, sp.q_len);
                const int fit = p.gqa > 128 ? 0 : 128 % p.gqa == 0 ? 128 / p.gqa : (129 - p.gqa) / p.gqa;
                if (!make_q_maps(&maps_new, p.q, plan.total_rows, p.hq, p.hkv, std::min(fit, longest)))
                    return fail(h, AGX_E_CUDA, "cuTensorMapEncodeTiled failed");
                e = launch_attn_tile_bf16(p, ln.kind == KIND_STREAM, map_k, map_v, maps_new, stream);
                break;
            }
            default: return fail(h, AGX_E_UNSUPPORTED, "unknown kernel kind");
        }
        if (e != cudaSuccess) return cuda_fail(h, e, "attention launch");
        h->last_launches++;
        if (split) {
            e = launch_attn_combine(p, h->cfg.dtype, ln.total_rows, stream);
            if (e != cudaSuccess) return cuda_fail(h, e, "combine launch");
            h->last_launches++;
        }
    }
    return AGX_OK;
}

agx_status agx_attn_prefixed(agx_handle* h, const void* q_block, const void* k_pool, const void* v_pool,
                             int64_t num_pages, const int32_t* page_table, int32_t pt_stride, const int32_t* P,
                             const int32_t* Q, int32_t B, void* out, float* lse, void* workspace,
                             size_t workspace_bytes, void* stream) {
    return attn_impl(h, q_block, nullptr, nullptr, k_pool, v_pool, num_pages, page_table, pt_stride, P, Q, B, out, lse,
                     workspace, workspace_bytes, stream, h && h->early_prefix);
}

agx_status agx_attn_prefixed_append(agx_handle* h, const void* q_block, const void* k_new, const void* v_new, void* k_pool,
                                    void* v_pool, int64_t num_pages, const int32_t* page_table, int32_t pt_stride,
                                    const int32_t* P, const int32_t* Q, int32_t B, void* out, float* lse,
                                    void* workspace, size_t workspace_bytes, void* stream) {
    if (h && B > 0 && (!k_new || !v_new)) return fail(h, AGX_E_INVAL, "null pointer");
    return attn_impl(h, q_block, k_new, v_new, k_pool, v_pool, num_pages, page_table, pt_stride, P, Q, B, out, lse,
                     workspace, workspace_bytes, stream, h && h->early_prefix);
}

int64_t agx_accept_workspace_bytes(agx_handle* h, int32_t total_q, int32_t vocab) {
    if (!h) return AGX_E_INVAL;
    if (total_q < 0 || vocab < 1) return fail(h, AGX_E_RANGE, "total_q < 0 or vocab < 1");
    // the rows' winners when they do not fit the kernel's shared memory (more than 2048 rows); the rows' keys live in the handle
    return (int64_t)total_q * 4 + 256;
}

agx_status agx_accept_greedy(agx_handle* h, const void* logits, int32_t logits_dtype, int64_t row_stride,
                             int32_t vocab, const int32_t* drafts, const int32_t* cu_q, int32_t B, int32_t total_q,
                             int32_t* accept_len, int32_t* next_token, int32_t* argmax, int32_t* seq_lens,
                             void* workspace, size_t workspace_bytes, void* stream) {
    CallRange range_("agx_accept_greedy");
    if (!h) return AGX_E_INVAL;
    h->last_launches = 0;
    if (B < 0 || total_q < 0) return fail(h, AGX_E_INVAL, "negative B or total_q");
    if (B == 0) return AGX_OK;
    if (total_q < B) return fail(h, AGX_E_INVAL, "total_q < B (every sequence has at least one row)");
    if (logits_dtype != AGX_BF16 && logits_dtype != AGX_F32) return fail(h, AGX_E_UNSUPPORTED, "logits dtype");
    if (vocab < 1 || row_stride < vocab) return fail(h, AGX_E_RANGE, "vocab < 1 or row_stride < vocab");
    if (total_q > 65535) return fail(h, AGX_E_RANGE, "more than 65535 logits rows in one call");
    if (!logits || !cu_q || !accept_len || !next_token || (!drafts && total_q > B)) return fail(h, AGX_E_INVAL, "null pointer");
    if (!aligned(logits, elem_size(logits_dtype))) return fail(h, AGX_E_INVAL, "logits misaligned");
    const int64_t need = agx_accept_workspace_bytes(h, total_q, vocab);
    if (!workspace || !aligned(workspace, 8) || (int64_t)workspace_bytes < need)
        return fail(h, AGX_E_INVAL, "accept workspace missing, misaligned or too small (%lld needed)", (long long)need);
    cudaError_t e = launch_accept(logits, logits_dtype, row_stride, vocab, drafts, cu_q, B, total_q, accept_len,
                                  next_token, argmax, seq_lens, h->d_row_keys, (int*)workspace, h->sm_count, h->d_ticket,
                                  (cudaStream_t)stream);
    if (e != cudaSuccess) return cuda_fail(h, e, "accept launch");
    h->last_launches = 1;
    return AGX_OK;
}

agx_status agx_get_status(agx_handle* h, void* stream, int32_t* device_status) {
    if (!h || !device_status) return AGX_E_INVAL;
    int v = 0;
    cudaError_t e = cudaMemcpyAsync(&v, h->d_status, sizeof v, cudaMemcpyDeviceToHost, (cudaStream_t)stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize((cudaStream_t)stream);
    if (e != cudaSuccess) return cuda_fail(h, e, "status read");
    *device_status = v;
    if (v != 0) {
        e = cudaMemsetAsync(h->d_status, 0, sizeof(int), (cudaStream_t)stream);
        if (e != cudaSuccess) return cuda_fail(h, e, "status clear");
        return fail(h, AGX_E_DEVICE, "device status 0x%x", v);
    }
    return AGX_OK;
}

int32_t agx_last_launch_count(const agx_handle* h) { return h ? h->last_launches : 0; }

agx_status agx_set_option(agx_handle* h, int32_t option, int64_t value) {
    if (!h) return AGX_E_INVAL;
    switch (option) {
        case AGX_OPT_EARLY_PREFIX_LOADS:
            h->early_prefix = value != 0;
            return AGX_OK;
        case AGX_OPT_WAIT_LIMIT_CYCLES:
            if (value < 1000) return fail(h, AGX_E_RANGE, "wait limit below 1000 cycles");
            h->wait_limit_cycles = value;
            return AGX_OK;
        case AGX_OPT_ZERO_COPY:
            if (value < 0 || value > 3) return fail(h, AGX_E_RANGE, "zero-copy bits");
            h->zero_copy = (int)value;
            return AGX_OK;
        case AGX_OPT_TEST_DROP_STAGE:
            if (value < -1 || value > 0x7FFFFFFF) return fail(h, AGX_E_RANGE, "stage index");
            h->drop_stage = (int)value;
            return AGX_OK;
        default:
            return fail(h, AGX_E_INVAL, "unknown option %d", option);
    }
}

}  // extern "C"

namespace {
constexpr size_t kZeroCopyMaxBytes = 1u << 20;

// Device-side address of a 16-byte-aligned host buffer that is pinned and mapped (cudaHostAlloc / cudaHostRegister
// under unified addressing), else NULL.
void* mapped_alias(const void* host) {
    if (!host || ((uintptr_t)host & 15)) return nullptr;
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, host) != cudaSuccess) { (void)cudaGetLastError(); return nullptr; }
    return at.type == cudaMemoryTypeHost ? at.devicePointer : nullptr;
}

// Attention-only host steps that move a few megabytes or more are cut into row chunks whose transfers overlap the
// attention calls of the other chunks (chunked prefill: rows [r0, r1) of a block are a block of their own behind a prefix
// longer by r0, since the chunks before them have appended their K/V by then).
bool host_step_pipelined(const agx_handle* h, int B, const int32_t* Q, int vocab) {
    if (vocab > 0 || h->pipe_rows <= 0) return false;
    long long tq = 0;
    for (int s = 0; s < B; ++s) tq += Q[s];
    const long long in_bytes = tq * (h->cfg.num_q_heads + 2 * h->cfg.num_kv_heads) * h->cfg.head_dim * elem_size(h->cfg.dtype);
    return in_bytes >= (4ll << 20) && tq > h->pipe_rows;
}

// The attention calls of a pipelined host step: runs of whole blocks that together have about a thousand rows, and
// blocks longer than that in row chunks of pipe_rows rows.
struct HostChunk {
    int s0, nseq;      // sequences [s0, s0 + nseq)
    int r0, rows;      // nseq == 1: rows [r0, r0 + rows) of the block; otherwise r0 = 0 and rows = all rows of the run
    size_t row_begin;  // first row of the chunk in the step's row order
};
void host_step_chunks(const agx_handle* h, int B, const int32_t* Q, std::vector<HostChunk>& out) {
    // Runs of whole blocks of about a thousand rows (measured on the ragged prefill blocks of c4, runs of 384 / 512 / 768 / 1024 rows:
    // 1.94 / 1.97 / 1.81 / 1.77 ms per step).  When that gives fewer than three calls there is nothing to overlap: blocks on their
    // own are then cut into row chunks (the 512-row block of c3 as one call 1.68 ms per 8 layers, as 384 + 128 rows 1.54 ms; with
    // many runs the cut only adds calls: c4 1.93 ms).
    const int run_rows = std::max(1024, 2 * h->pipe_rows);
    std::vector<HostChunk> runs;
    size_t row = 0;
    int s = 0;
    while (s < B) {
        HostChunk c = {s, 0, 0, 0, row};
        while (s < B && c.nseq < kMaxSeqs && (c.nseq == 0 || c.rows + Q[s] <= run_rows)) {
            c.rows += Q[s]; row += Q[s]; ++c.nseq; ++s;
        }
        runs.push_back(c);
    }
    out.clear();
    for (const HostChunk& c : runs) {
        if (runs.size() < 3 && c.nseq == 1 && c.rows > h->pipe_rows) {
            for (int r0 = 0; r0 < c.rows; r0 += h->pipe_rows)
                out.push_back({c.s0, 1, r0, std::min(h->pipe_rows, c.rows - r0), c.row_begin + (size_t)r0});
        } else {
            out.push_back(c);
        }
    }
}

struct HostStepLayout {
    size_t q, k, v, out, logits, drafts, prefix, cu, acc, next, seqlen, attn_ws, accept_ws, total;
    size_t q_bytes, kv_bytes, logits_bytes, attn_ws_bytes, accept_ws_bytes;
    int total_q;
};
agx_status host_step_layout(agx_handle* h, int B, const int32_t* P, const int32_t* Q, int logits_dtype,
                            int64_t row_stride, int vocab, HostStepLayout& L) {
    if (B < 1 || !P || !Q) return fail(h, AGX_E_INVAL, "B < 1 or null lengths");
    const bool with_accept = vocab > 0;  // vocab == 0: attention only
    if (with_accept) {
        if (logits_dtype != AGX_BF16 && logits_dtype != AGX_F32) return fail(h, AGX_E_UNSUPPORTED, "logits dtype");
        if (row_stride < vocab) return fail(h, AGX_E_RANGE, "row_stride < vocab");
    } else if (vocab < 0) {
        return fail(h, AGX_E_RANGE, "vocab < 0");
    }
    long long tq = 0;
    for (int s = 0; s < B; ++s) {
        if (Q[s] < 1) return fail(h, AGX_E_INVAL, "q_len[%d] = %d < 1", s, Q[s]);
        tq += Q[s];
    }
    if (tq > 65535) return fail(h, AGX_E_RANGE, "more than 65535 rows in one host step");
    int64_t aws = 0;
    if (host_step_pipelined(h, B, Q, vocab)) {
        // one attention call per chunk, one after the other on the caller's stream: the largest workspace of them
        std::vector<HostChunk> chunks;
        host_step_chunks(h, B, Q, chunks);
        for (const HostChunk& c : chunks) {
            const int32_t pc = P[c.s0] + c.r0, qc = c.rows;
            const int64_t w = c.nseq == 1 ? agx_attn_workspace_bytes(h, 1, &pc, &qc) : agx_attn_workspace_bytes(h, c.nseq, P + c.s0, Q + c.s0);
            if (w < 0) return (agx_status)w;
            aws = std::max(aws, w);
        }
    } else {
        aws = agx_attn_workspace_bytes(h, B, P, Q);
        if (aws < 0) return (agx_status)aws;
    }
    const int64_t cws = with_accept ? agx_accept_workspace_bytes(h, (int)tq, vocab) : 0;
    if (cws < 0) return (agx_status)cws;
    const size_t es = elem_size(h->cfg.dtype);
    L.total_q = (int)tq;
    L.q_bytes = (size_t)tq * h->cfg.num_q_heads * h->cfg.head_dim * es;
    L.kv_bytes = (size_t)tq * h->cfg.num_kv_heads * h->cfg.head_dim * es;
    L.logits_bytes = with_accept ? (size_t)tq * row_stride * elem_size(logits_dtype) : 0;
    L.attn_ws_bytes = (size_t)aws;
    L.accept_ws_bytes = (size_t)cws;
    size_t off = 0;
    auto take = [&](size_t bytes) { size_t o = off; off += (bytes + 255) / 256 * 256; return o; };
    L.q = take(L.q_bytes); L.k = take(L.kv_bytes); L.v = take(L.kv_bytes); L.out = take(L.q_bytes);
    L.logits = take(L.logits_bytes); L.drafts = take((size_t)(tq - B) * 4 + 4);
    L.prefix = take((size_t)B * 4); L.cu = take((size_t)(B + 1) * 4);
    L.acc = take((size_t)B * 4); L.next = take((size_t)B * 4); L.seqlen = take((size_t)B * 4);
    L.attn_ws = take(L.attn_ws_bytes); L.accept_ws = take(L.accept_ws_bytes);
    L.total = off;
    return AGX_OK;
}
}  // namespace

extern "C" {

int64_t agx_verify_step_host_workspace_bytes(agx_handle* h, int32_t B, const int32_t* P, const int32_t* Q,
                                             int32_t logits_dtype, int64_t row_stride, int32_t vocab) {
    if (!h) return AGX_E_INVAL;
    HostStepLayout L;
    agx_status st = host_step_layout(h, B, P, Q, logits_dtype, row_stride, vocab, L);
    return st != AGX_OK ? (int64_t)st : (int64_t)L.total;
}

static agx_status verify_step_host_impl(agx_handle* h, void* k_pool, void* v_pool, int64_t num_pages,
                                const int32_t* page_table, int32_t pt_stride, const int32_t* P, const int32_t* Q,
                                int32_t B, const void* h_q, const void* h_k, const void* h_v, const void* h_logits,
                                int32_t logits_dtype, int64_t row_stride, int32_t vocab, const int32_t* h_drafts,
                                void* h_out, int32_t* h_accept, int32_t* h_next, int32_t* h_seq_lens, void* workspace,
                                size_t workspace_bytes, void* stream_v, bool sync) {
    CallRange range_("agx_verify_step_host");
    if (!h) return AGX_E_INVAL;
    HostStepLayout L;
    agx_status st = host_step_layout(h, B, P, Q, logits_dtype, row_stride, vocab, L);
    if (st != AGX_OK) return st;
    const bool with_accept = vocab > 0;
    if (!k_pool || !v_pool || !page_table || !h_q || !h_k || !h_v || !h_out) return fail(h, AGX_E_INVAL, "null pointer");
    if (with_accept && (!h_logits || !h_accept || !h_next || !h_seq_lens || (!h_drafts && L.total_q > B)))
        return fail(h, AGX_E_INVAL, "null pointer (accept arguments)");
    if (!workspace || !aligned(workspace, 256) || workspace_bytes < L.total)
        return fail(h, AGX_E_INVAL, "host-step workspace missing, misaligned or too small (%zu needed)", L.total);
    cudaStream_t stream = (cudaStream_t)stream_v;
    char* ws = (char*)workspace;
    if (host_step_pipelined(h, B, Q, vocab)) {
        cudaError_t pe = cudaSuccess;
        if (!h->pipe_in) pe = cudaStreamCreateWithFlags(&h->pipe_in, cudaStreamNonBlocking);
        if (pe == cudaSuccess && !h->pipe_out) pe = cudaStreamCreateWithFlags(&h->pipe_out, cudaStreamNonBlocking);
        std::vector<HostChunk> list;
        host_step_chunks(h, B, Q, list);
        const size_t chunks = list.size();
        while (pe == cudaSuccess && h->pipe_events.size() < 2 * chunks + 2) {
            cudaEvent_t ev;
            pe = cudaEventCreateWithFlags(&ev, cudaEventDisableTiming);
            if (pe == cudaSuccess) h->pipe_events.push_back(ev);
        }
        if (pe != cudaSuccess) return cuda_fail(h, pe, "host step: pipeline set-up");
        const size_t es = elem_size(h->cfg.dtype);
        const size_t q_row = (size_t)h->cfg.num_q_heads * h->cfg.head_dim * es, kv_row = (size_t)h->cfg.num_kv_heads * h->cfg.head_dim * es;
        cudaEvent_t fork = h->pipe_events[2 * chunks], join = h->pipe_events[2 * chunks + 1];
        // the side streams start behind whatever the caller has already put on its stream ...
        pe = cudaEventRecord(fork, stream);
        if (pe == cudaSuccess) pe = cudaStreamWaitEvent(h->pipe_in, fork, 0);
        if (pe == cudaSuccess) pe = cudaStreamWaitEvent(h->pipe_out, fork, 0);
        int launches = 0;
        for (size_t i = 0; i < chunks && pe == cudaSuccess; ++i) {
            const HostChunk& c = list[i];
            const int32_t pc = P[c.s0] + c.r0, qc = c.rows;
            const size_t r = c.row_begin, n = (size_t)c.rows;
            cudaEvent_t in_done = h->pipe_events[2 * i], out_ready = h->pipe_events[2 * i + 1];
            pe = cudaMemcpyAsync(ws + L.q + r * q_row, (const char*)h_q + r * q_row, n * q_row, cudaMemcpyHostToDevice, h->pipe_in);
            if (pe == cudaSuccess) pe = cudaMemcpyAsync(ws + L.k + r * kv_row, (const char*)h_k + r * kv_row, n * kv_row, cudaMemcpyHostToDevice, h->pipe_in);
            if (pe == cudaSuccess) pe = cudaMemcpyAsync(ws + L.v + r * kv_row, (const char*)h_v + r * kv_row, n * kv_row, cudaMemcpyHostToDevice, h->pipe_in);
            if (pe == cudaSuccess) pe = cudaEventRecord(in_done, h->pipe_in);
            if (pe == cudaSuccess) pe = cudaStreamWaitEvent(stream, in_done, 0);
            if (pe != cudaSuccess) break;
            st = agx_attn_prefixed_append(h, ws + L.q + r * q_row, ws + L.k + r * kv_row, ws + L.v + r * kv_row, k_pool, v_pool, num_pages,
                                          page_table + (size_t)c.s0 * pt_stride, pt_stride, c.nseq == 1 ? &pc : P + c.s0,
                                          c.nseq == 1 ? &qc : Q + c.s0, c.nseq, ws + L.out + r * q_row, nullptr,
                                          L.attn_ws_bytes ? ws + L.attn_ws : nullptr, L.attn_ws_bytes, stream);
            if (st != AGX_OK) break;
            launches += h->last_launches;
            pe = cudaEventRecord(out_ready, stream);
            if (pe == cudaSuccess) pe = cudaStreamWaitEvent(h->pipe_out, out_ready, 0);
            if (pe == cudaSuccess) pe = cudaMemcpyAsync((char*)h_out + r * q_row, ws + L.out + r * q_row, n * q_row, cudaMemcpyDeviceToHost, h->pipe_out);
        }
        // ... and the caller's stream ends behind the last download (also when a call in the middle failed: the join still
        // has to bring the side streams back, or a stream capture of the caller's would be left forked)
        cudaError_t je = cudaEventRecord(join, h->pipe_out);
        if (je == cudaSuccess) je = cudaStreamWaitEvent(stream, join, 0);
        if (st != AGX_OK) return st;
        if (pe == cudaSuccess) pe = je;
        if (pe == cudaSuccess && sync) pe = cudaStreamSynchronize(stream);
        if (pe != cudaSuccess) return cuda_fail(h, pe, "host step: pipelined transfers");
        h->last_launches = launches;
        return AGX_OK;
    }
    std::vector<int32_t>& cu = h->cu_host;  // outlives the asynchronous copy (the call ends with a sync)
    cu.assign(B + 1, 0);
    for (int s = 0; s < B; ++s) cu[s + 1] = cu[s] + Q[s];
    cudaError_t e = cudaSuccess;
    int launches = 0;
    auto h2d = [&](size_t off, const void* src, size_t bytes) {
        if (e == cudaSuccess && bytes) e = cudaMemcpyAsync(ws + off, src, bytes, cudaMemcpyHostToDevice, stream);
    };
    // Small blocks in pinned, device-mapped host memory cross by one kernel that reads the host buffers and, on the
    // way back, by the attention kernels writing `out` straight into the host buffer: each copy-engine transfer on
    // the stream costs several microseconds whatever its size.  Anything else goes through cudaMemcpyAsync.
    const size_t in_bytes = L.q_bytes + 2 * L.kv_bytes;
    const void* mq = (h->zero_copy & 1) && in_bytes <= kZeroCopyMaxBytes ? mapped_alias(h_q) : nullptr;
    const void* mk = mq ? mapped_alias(h_k) : nullptr;
    const void* mv = mk ? mapped_alias(h_v) : nullptr;
    void* out_dev = ws + L.out;
    if ((h->zero_copy & 2) && L.q_bytes <= kZeroCopyMaxBytes)
        if (void* mo = mapped_alias(h_out)) out_dev = mo;
    if (mv) {
        StageCopies sc;
        sc.src[0] = (const uint4*)mq; sc.src[1] = (const uint4*)mk; sc.src[2] = (const uint4*)mv;
        sc.dst[0] = (uint4*)(ws + L.q); sc.dst[1] = (uint4*)(ws + L.k); sc.dst[2] = (uint4*)(ws + L.v);
        sc.units[0] = (unsigned)(L.q_bytes / 16); sc.units[1] = sc.units[2] = (unsigned)(L.kv_bytes / 16);
        e = launch_stage_in(sc, stream);
        if (e == cudaSuccess) ++launches;
    } else {
        h2d(L.q, h_q, L.q_bytes); h2d(L.k, h_k, L.kv_bytes); h2d(L.v, h_v, L.kv_bytes);
    }
    // The logits are needed by the accept step only: a megabyte or more of them crosses on a stream of the handle's own,
    // beside the attention kernels, and the caller's stream waits for that copy just before the accept launch.
    cudaEvent_t logits_done = nullptr;
    if (with_accept && L.logits_bytes >= (1u << 20) && h->pipe_rows > 0 && e == cudaSuccess) {
        if (!h->pipe_in) e = cudaStreamCreateWithFlags(&h->pipe_in, cudaStreamNonBlocking);
        while (e == cudaSuccess && h->pipe_events.size() < 2) {
            cudaEvent_t ev;
            e = cudaEventCreateWithFlags(&ev, cudaEventDisableTiming);
            if (e == cudaSuccess) h->pipe_events.push_back(ev);
        }
        if (e == cudaSuccess) e = cudaEventRecord(h->pipe_events[0], stream);   // behind whatever last used the workspace
        if (e == cudaSuccess) e = cudaStreamWaitEvent(h->pipe_in, h->pipe_events[0], 0);
        if (e == cudaSuccess) e = cudaMemcpyAsync(ws + L.logits, h_logits, L.logits_bytes, cudaMemcpyHostToDevice, h->pipe_in);
        if (e == cudaSuccess && L.total_q > B)
            e = cudaMemcpyAsync(ws + L.drafts, h_drafts, (size_t)(L.total_q - B) * 4, cudaMemcpyHostToDevice, h->pipe_in);
        if (e == cudaSuccess) e = cudaEventRecord(h->pipe_events[1], h->pipe_in);
        if (e == cudaSuccess) logits_done = h->pipe_events[1];
    } else if (with_accept) {
        h2d(L.logits, h_logits, L.logits_bytes);
        h2d(L.drafts, h_drafts, (size_t)(L.total_q - B) * 4);
    }
    if (!with_accept) {
        // lengths are needed on the device by the accept step only
    } else if (B <= kMaxSeqs) {   // as kernel arguments: no pageable copies, which would each synchronise the stream first
        StepMeta meta;
        meta.B = B;
        for (int s = 0; s < B; ++s) { meta.prefix[s] = P[s]; meta.cu[s] = cu[s]; }
        meta.cu[B] = cu[B];
        if (e == cudaSuccess)
            e = launch_write_meta(meta, (int*)(ws + L.prefix), (int*)(ws + L.seqlen), (int*)(ws + L.cu), stream);
        if (e == cudaSuccess) ++launches;
    } else {
        h2d(L.prefix, P, (size_t)B * 4);
        h2d(L.seqlen, P, (size_t)B * 4);
        h2d(L.cu, cu.data(), (size_t)(B + 1) * 4);
    }
    if (e != cudaSuccess) return cuda_fail(h, e, "host step: upload");
    // behind the stage-in kernel, which lets this launch start only when everything before it is complete, cached-prefix pages may
    // always be fetched early
    st = attn_impl(h, ws + L.q, ws + L.k, ws + L.v, k_pool, v_pool, num_pages, page_table, pt_stride, P, Q, B, out_dev, nullptr,
                   L.attn_ws_bytes ? ws + L.attn_ws : nullptr, L.attn_ws_bytes, stream, mv || h->early_prefix);
    if (st == AGX_OK) launches += h->last_launches;
    if (logits_done) {   // (also when the attention call failed: the side stream is brought back before the call returns)
        e = cudaStreamWaitEvent(stream, logits_done, 0);
        if (e != cudaSuccess) return cuda_fail(h, e, "host step: logits upload");
    }
    if (st != AGX_OK) return st;
    if (with_accept) {
        st = agx_accept_greedy(h, ws + L.logits, logits_dtype, row_stride, vocab, (const int32_t*)(ws + L.drafts),
                               (const int32_t*)(ws + L.cu), B, L.total_q, (int32_t*)(ws + L.acc),
                               (int32_t*)(ws + L.next), nullptr, (int32_t*)(ws + L.seqlen), ws + L.accept_ws,
                               L.accept_ws_bytes, stream);
        if (st != AGX_OK) return st;
        launches += h->last_launches;
    }
    auto d2h = [&](void* dst, size_t off, size_t bytes) {
        if (e == cudaSuccess && bytes) e = cudaMemcpyAsync(dst, ws + off, bytes, cudaMemcpyDeviceToHost, stream);
    };
    if (out_dev == ws + L.out) d2h(h_out, L.out, L.q_bytes);
    if (with_accept) {
        d2h(h_accept, L.acc, (size_t)B * 4); d2h(h_next, L.next, (size_t)B * 4); d2h(h_seq_lens, L.seqlen, (size_t)B * 4);
    }
    if (e == cudaSuccess && sync) e = cudaStreamSynchronize(stream);
    if (e != cudaSuccess) return cuda_fail(h, e, "host step: download");
    h->last_launches = launches;
    return AGX_OK;
}

agx_status agx_verify_step_host(agx_handle* h, void* k_pool, void* v_pool, int64_t num_pages,
                                const int32_t* page_table, int32_t pt_stride, const int32_t* P, const int32_t* Q,
                                int32_t B, const void* h_q, const void* h_k, const void* h_v, const void* h_logits,
                                int32_t logits_dtype, int64_t row_stride, int32_t vocab, const int32_t* h_drafts,
                                void* h_out, int32_t* h_accept, int32_t* h_next, int32_t* h_seq_lens, void* workspace,
                                size_t workspace_bytes, void* stream) {
    return verify_step_host_impl(h, k_pool, v_pool, num_pages, page_table, pt_stride, P, Q, B, h_q, h_k, h_v, h_logits,
                                 logits_dtype, row_stride, vocab, h_drafts, h_out, h_accept, h_next, h_seq_lens, workspace,
                                 workspace_bytes, stream, true);
}

agx_status agx_verify_step_host_enqueue(agx_handle* h, void* k_pool, void* v_pool, int64_t num_pages,
                                        const int32_t* page_table, int32_t pt_stride, const int32_t* P, const int32_t* Q,
                                        int32_t B, const void* h_q, const void* h_k, const void* h_v,
                                        const void* h_logits, int32_t logits_dtype, int64_t row_stride, int32_t vocab,
                                        const int32_t* h_drafts, void* h_out, int32_t* h_accept, int32_t* h_next,
                                        int32_t* h_seq_lens, void* workspace, size_t workspace_bytes, void* stream) {
    return verify_step_host_impl(h, k_pool, v_pool, num_pages, page_table, pt_stride, P, Q, B, h_q, h_k, h_v, h_logits,
                                 logits_dtype, row_stride, vocab, h_drafts, h_out, h_accept, h_next, h_seq_lens, workspace,
                                 workspace_bytes, stream, false);
}

int64_t agx_ngram_lut_bytes(int32_t max_stream_tokens) {
    if (max_stream_tokens < 0 || max_stream_tokens > (1 << 24)) return AGX_E_RANGE;
    return (int64_t)ngram_lut_bytes(max_stream_tokens);
}

int64_t agx_ngram_workspace_bytes(int32_t stream_tokens) {
    if (stream_tokens < 0 || stream_tokens > (1 << 24)) return AGX_E_RANGE;
    return (int64_t)ngram_workspace_bytes(stream_tokens);
}

agx_status agx_ngram_build(agx_handle* h, const int32_t* stream_tokens, int32_t num_tokens, int32_t n, void* lut,
                           size_t lut_bytes, void* workspace, size_t workspace_bytes, void* stream) {
    CallRange range_("agx_ngram_build");
    if (!h) return AGX_E_INVAL;
    h->last_launches = 0;
    if (n != 2 && n != 3) return fail(h, AGX_E_UNSUPPORTED, "n-gram order %d (2 and 3 are built)", n);
    if (num_tokens < 0) return fail(h, AGX_E_INVAL, "negative num_tokens");
    if (num_tokens > (1 << 24)) return fail(h, AGX_E_RANGE, "more than 2^24 stream tokens");
    if (!lut || !workspace || (!stream_tokens && num_tokens > 0)) return fail(h, AGX_E_INVAL, "null pointer");
    if (!aligned(lut, 16) || !aligned(workspace, 16)) return fail(h, AGX_E_INVAL, "lut/workspace must be 16-byte aligned");
    if ((long long)lut_bytes < ngram_lut_bytes(num_tokens) || (long long)workspace_bytes < ngram_workspace_bytes(num_tokens))
        return fail(h, AGX_E_INVAL, "lut (%lld needed) or workspace (%lld needed) too small", ngram_lut_bytes(num_tokens),
                    ngram_workspace_bytes(num_tokens));
    cudaError_t e = launch_ngram_build(stream_tokens, num_tokens, n, lut, workspace, h->d_status, (cudaStream_t)stream);
    if (e != cudaSuccess) return cuda_fail(h, e, "n-gram build");
    h->last_launches = ngram_build_launches(num_tokens, n);
    return AGX_OK;
}

agx_status agx_ngram_draft(agx_handle* h, const void* lut, const int32_t* context, const int32_t* fill, int32_t B, int32_t k,
                           int32_t* drafts, int32_t* has_draft, void* stream) {
    CallRange range_("agx_ngram_draft");
    if (!h) return AGX_E_INVAL;
    h->last_launches = 0;
    if (B < 0 || k < 0) return fail(h, AGX_E_INVAL, "negative B or k");
    if (B == 0) return AGX_OK;
    if (!lut || !context || !has_draft || (k > 0 && (!fill || !drafts))) return fail(h, AGX_E_INVAL, "null pointer");
    cudaError_t e = launch_ngram_draft(lut, context, fill, B, k, drafts, has_draft, (cudaStream_t)stream);
    if (e != cudaSuccess) return cuda_fail(h, e, "n-gram draft");
    h->last_launches = 1;
    return AGX_OK;
}

agx_status agx_kv_copy_pages(agx_handle* h, void* k_pool, void* v_pool, int64_t num_pages, const int32_t* src,
                             const int32_t* dst, int32_t count, void* stream) {
    CallRange range_("agx_kv_copy_pages");
    if (!h) return AGX_E_INVAL;
    h->last_launches = 0;
    if (count < 0) return fail(h, AGX_E_INVAL, "negative count");
    if (count == 0) return AGX_OK;
    if (!k_pool || !v_pool || !src || !dst || num_pages < 1) return fail(h, AGX_E_INVAL, "null pointer or no pages");
    if (!aligned(k_pool, 16) || !aligned(v_pool, 16)) return fail(h, AGX_E_INVAL, "pools must be 16-byte aligned");
    cudaError_t e = launch_copy_pages(h->cfg.dtype, k_pool, v_pool, num_pages, src, dst, count, h->cfg.num_kv_heads,
                                      h->cfg.head_dim, h->d_status, (cudaStream_t)stream);
    if (e != cudaSuccess) return cuda_fail(h, e, "page copy");
    h->last_launches = 1;
    return AGX_OK;
}

int64_t agx_kv_import_staging_bytes(const agx_handle* h, int32_t count) {
    if (!h || count < 0) return AGX_E_INVAL;
    return 2ll * count * h->cfg.num_kv_heads * kPage * h->cfg.head_dim * elem_size(h->cfg.dtype);
}

agx_status agx_kv_import_pages(agx_handle* h, void* k_pool, void* v_pool, int64_t num_pages, const void* h_k, const void* h_v,
                               const int32_t* dst_pages, int32_t count, void* staging, size_t staging_bytes, void* stream_v) {
    CallRange range_("agx_kv_import_pages");
    if (!h) return AGX_E_INVAL;
    h->last_launches = 0;
    if (count < 0) return fail(h, AGX_E_INVAL, "negative count");
    if (count == 0) return AGX_OK;
    if (!k_pool || !v_pool || !h_k || !h_v || !dst_pages || !staging || num_pages < 1) return fail(h, AGX_E_INVAL, "null pointer or no pages");
    if (!aligned(k_pool, 16) || !aligned(v_pool, 16) || !aligned(staging, 16)) return fail(h, AGX_E_INVAL, "pools and staging must be 16-byte aligned");
    const size_t half = (size_t)agx_kv_import_staging_bytes(h, count) / 2;
    if (staging_bytes < 2 * half) return fail(h, AGX_E_INVAL, "staging too small: %zu < %zu", staging_bytes, 2 * half);
    cudaStream_t stream = (cudaStream_t)stream_v;
    char* st = (char*)staging;
    // Stored pages in pinned, device-mapped host memory are read across the bus by the scatter kernel itself (one pass,
    // no staging); anything else is copied into the staging area first.
    const void* mk = (h->zero_copy & 1) ? mapped_alias(h_k) : nullptr;
    const void* mv = mk ? mapped_alias(h_v) : nullptr;
    cudaError_t e = cudaSuccess;
    if (mv) {
        e = launch_scatter_pages(h->cfg.dtype, k_pool, v_pool, num_pages, mk, mv, dst_pages, count, h->cfg.num_kv_heads,
                                 h->cfg.head_dim, h->d_status, stream);
    } else {
        e = cudaMemcpyAsync(st, h_k, half, cudaMemcpyHostToDevice, stream);
        if (e == cudaSuccess) e = cudaMemcpyAsync(st + half, h_v, half, cudaMemcpyHostToDevice, stream);
        if (e == cudaSuccess)
            e = launch_scatter_pages(h->cfg.dtype, k_pool, v_pool, num_pages, st, st + half, dst_pages, count, h->cfg.num_kv_heads,
                                     h->cfg.head_dim, h->d_status, stream);
    }
    if (e != cudaSuccess) return cuda_fail(h, e, "page import");
    h->last_launches = 1;
    return AGX_OK;
}

}  // extern "C"
