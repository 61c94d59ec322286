// Small-q attention over short KV splits on tcgen05 with the operands swapped (bf16, d = 128): decode and verify blocks of at most 32
// query rows per KV head whose splits hold at most NT * 128 tokens.
//
// Such a launch is bound by latency: a CTA brings in its split (at most 24 pages of K and of V) while the launch before it
// drains, and then everything between the arrival of Q and the last store is a chain.  With query rows as the M side of the MMAs
// (mma.sync over 16-row tiles, or tcgen05 over 128 mostly empty rows) that chain is the matrix instructions.  Here the tokens take the M
// side, S^T = K Q^T, and the head dimension in the second product, O^T = V^T P^T: the query rows are the N side, 16 or 32 columns, so
// that both products of a split are some 25 to 50 instructions of one thread.  TMEM then holds a token per lane and a query row per
// column: every thread owns one token's scores (RH = 2: those of half of the rows), row maxima are one instruction each, row sums butterflies over lanes
// that leave row r in lane r, and P goes back through shared memory (dead K) as the B operand.  All of a split's K, V and scores are on the SM at once: one
// softmax, no rescaling.
// A CTA of one verify layer (8 rows, 32/8 heads), from Q's arrival: over 2000 tokens (two tiles, two threads a token) first scores 0.4 us behind it, maxima 0.9,
// P 1.4, O 2.0, stored 2.3; over 4096 (three tiles) 0.45, 1.2, 2.0, 3.0, 3.3.
// What is left is the chain itself: three barriers, two MMA round trips (a 128 x 16 operand tile takes the MMA unit about 64 clocks to
// read whatever N is), and around it the launch, the dependency waits and the merge of the splits.

#include <algorithm>

#include "agx_internal.cuh"
#include "agx_sm100.cuh"

namespace agx {
namespace {

constexpr int kTileTok = 128;
constexpr unsigned kSuspendNs = 20000;   // see mbar_try_wait
constexpr uint32_t kTile = 128 * 256;   // 8 pages of K or V
constexpr uint32_t kCols = 128;         // TMEM: O^T at column 0, S^T of tile t at 32 + 32 t

// NR query rows that a CTA works on (4, 8, 16 or 32), NC columns of the MMAs (the rows behind NR are zeros nobody reads); RH threads a token, each
// with NR / RH of its rows
template <int NR, int NT, int RH>
struct Lay {
    static constexpr int NC = NR < 16 ? 16 : NR;
    static constexpr uint32_t kK = 0, kV = NT * kTile, kQ = 2 * NT * kTile, kBar = kQ + NC * 256;
    static constexpr uint32_t kMax = kBar + 128;                       // [token warp][NR] row maxima
    static constexpr uint32_t kRef = kMax + NT * 4 * NR * 4;           // [warp][NR / RH] the row references, a copy per warp
    static constexpr uint32_t kSum = kRef + NT * 4 * NR * 4;           // [token warp][NR]
    static constexpr uint32_t kDst = kSum + NT * 4 * NR * 4;           // [warp][NR / RH] where the rows go
    static constexpr uint32_t kBytes = kDst + NT * 4 * NR * 8 + 1024;  // + alignment slack
    static constexpr uint32_t kP = kK;                                 // P: [64-token block][NC rows][128 B], 128-byte swizzle
    static constexpr uint32_t kO = kV;                                 // cluster merge: [NR][128] floats, then [NR] (m, l)
    static_assert(kBytes <= 232448, "one CTA's shared memory");
};

// v[r] of every lane -> lane l holds the sum over all lanes of row l % NR.  The lanes meet in the same order for every NR.
template <int NR>
__device__ __forceinline__ float sum_across_lanes(float (&v)[NR]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int d = 16; d >= NR; d >>= 1) {
#pragma unroll
        for (int i = 0; i < NR; ++i) v[i] += __shfl_xor_sync(0xFFFFFFFFu, v[i], d);
    }
#pragma unroll
    for (int d = NR / 2; d >= 1; d >>= 1) {
        const bool up = lane & d;
#pragma unroll
        for (int i = 0; i < d; ++i) {
            const float keep = up ? v[i + d] : v[i], send = up ? v[i] : v[i + d];
            v[i] = keep + __shfl_xor_sync(0xFFFFFFFFu, send, d);
        }
    }
    return v[0];
}

}  // namespace

template <int NR, int NT, int RH>
__global__ void __launch_bounds__(NT * 128 * RH + 32, 1)
attn_swap_bf16_kernel(const __grid_constant__ AttnParams p, const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v) {
    using S = Lay<NR, NT, RH>;
    constexpr int NC = S::NC, NH = NR / RH;   // NH: rows of a softmax warp
    constexpr int kTokenWarps = NT * 4, kWarps = kTokenWarps * RH, kThreads = kWarps * 32;   // of the softmax warps; one more warp issues the copies and the MMAs
    extern __shared__ unsigned char smem_raw[];
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    unsigned char* smem = smem_raw + (base - smem_u32(smem_raw));
    auto k_bar = [&](int t) { return base + S::kBar + 8u * t; };
    auto v_bar = [&](int t) { return base + S::kBar + 8u * (NT + t); };
    auto s_bar = [&](int t) { return base + S::kBar + 8u * (2 * NT + t); };
    const uint32_t o_bar = base + S::kBar + 8u * (3 * NT);
    volatile int* abort_flag = (volatile int*)(smem + S::kBar + 8 * (3 * NT + 1));
    uint32_t* tmem_slot = (uint32_t*)(smem + S::kBar + 8 * (3 * NT + 2));

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int part = RH == 1 ? 0 : warp / kTokenWarps, tw = warp - part * kTokenWarps, tile = tw >> 2, row_off = part * NH;   // (issuer: not used)
    const bool issuer = warp == kWarps;
    const SeqPlan& sp = p.seq[find_seq(p, blockIdx.x)];
    // Items are ((g * row_chunks) + rc) * nsplit + split.  The planner sends blocks of one row chunk only, but the kernel keeps the general form:
    // with the chunk's first row a constant 0 the compiler's schedule costs a verify layer over 4096 tokens 0.16 us (9.1 -> 9.3 us with its append,
    // three forms of it tried) and gives a decode layer 0.04 us.
    const unsigned item = blockIdx.x - sp.item0;
    const unsigned chunk = item / (unsigned)sp.nsplit;
    const int split = (int)(item - chunk * sp.nsplit);
    const int g = sp.row_chunks == 1 ? (int)chunk : (int)(chunk / (unsigned)sp.row_chunks);
    const int rc = (int)chunk - g * sp.row_chunks;
    const int G = p.gqa, P = sp.prefix_len, q = sp.q_len, L = P + q;
    const int rows = q * G, row0 = rc * NC, n_rows = min(NR, rows - row0);   // query rows of this KV head, r = i * G + (h % G)
    auto div_g = [&](int r) { return (int)(((uint64_t)(uint32_t)r * p.row_div_magic) >> 32); };   // r / G without the division
    const int vis_end = P + min(q - 1, div_g(row0 + NC - 1)) + 1;   // tokens the chunk's last row sees
    const int tok_begin = split * sp.split_tokens, tok_end = min(vis_end, tok_begin + sp.split_tokens);
    const int n_pages = max(0, (tok_end - tok_begin + kPage - 1) / kPage), n_tiles = (n_pages + 7) >> 3;

    // ---- setup.  With p.early_prefix (the caller vouches that the page table and the pages below the cached-prefix length are not written by a
    // launch still in flight) page ids and pool pages are fetched before the dependency wait; with a fused append only pages below the block
    // come from the pool.  Pages from own_pg on are put together by hand beside Q: block rows come from k_new / v_new and go into the pool on
    // the way, and a last page that is only partly valid gets zeros behind the last token (V must not hold a NaN there).
    const int* pt_row = p.page_table + (long long)sp.seq_index * p.pt_stride;
    const int page0 = tok_begin / kPage;
    const bool pre = p.early_prefix;
    const int pool_end = p.k_new ? P : L;
    const int own_pg = min(n_pages, max(0, (pool_end >> 4) - page0));
    const int own_units = (n_pages - own_pg) * 512;   // 16-byte units, [page][K, V][16 rows][16 units]
    // a thread's units of the first own page, and of the second where there is one (with the second page behind the first one's trip to
    // memory 8 rows from token 2750 on took 10.0 us a layer, from 2752 on 8.1).  A block of 18 to 32 rows (one head a group) may lie in three
    // pages: units from 1024 on have an id of their own and come behind the others.
    constexpr int kOwn1 = (512 + kThreads - 1) / kThreads, kOwn = (1024 + kThreads - 1) / kThreads;
    const bool more_own = own_units > kOwn1 * kThreads;
    const int two_pages = min(own_units, 1024);
    // A unit's place in the pool but for its page, and its source where it is a block row's (held in registers for the first two pages).
    auto own_tok = [&](int u) { return tok_begin + (own_pg + (u >> 9)) * kPage + ((u >> 4) & 15); };
    auto own_pool = [&](int u) {
        return (unsigned char*)(((u >> 8) & 1) ? p.v_pool : p.k_pool) + (g * kPage + (own_tok(u) & 15)) * 256 + (u & 15) * 16;
    };
    auto own_new = [&](int u) {
        const int tok = own_tok(u);
        return (const unsigned char*)(((u >> 8) & 1) ? p.v_new : p.k_new) + ((long long)(sp.q_row0 + tok - P) * p.hkv + g) * 256 + (u & 15) * 16;
    };
    int num_pages = (int)min(p.num_pages, 0x7FFFFFFFll), page_bytes = p.hkv * kPage * 256;
    auto own_id = [&](int u) { const int slot = page0 + own_pg + (u >> 9); return slot < p.pt_stride ? __ldg(pt_row + slot) : -1; };
    auto own_load = [&](int u, int id, unsigned char* in_pool, const unsigned char* in_new) {
        const int tok = own_tok(u);
        uint4 v = make_uint4(0, 0, 0, 0);
        if (tok < pool_end) v = __ldcg((const uint4*)(in_pool + (long long)((id < 0 || id >= num_pages) ? 0 : id) * page_bytes));   // (reported below)
        else if (tok < L) v = __ldg((const uint4*)in_new);
        return v;
    };
    auto own_store = [&](int u, int id, unsigned char* in_pool, const uint4 v) {
        const int pg = own_pg + (u >> 9), r = (u >> 4) & 15, is_v = (u >> 8) & 1, ch = u & 15, tok = own_tok(u);
        *(uint4*)(smem + (is_v ? S::kV : S::kK) + pg * 4096 + (r >> 3) * 2048 + (ch >> 3) * 1024 + (r & 7) * 128 + (((ch & 7) ^ (r & 7)) << 4)) = v;
        if (tok >= pool_end && tok < L && id >= 0 && id < num_pages) *(uint4*)(in_pool + (long long)id * page_bytes) = v;
    };
    int first_id = 0, second_id = 0;   // of the own pages; issuer: first_id is that of page `lane`
    auto fetch_ids = [&]() {
        if (issuer) { if (lane < n_pages) first_id = __ldg(pt_row + page0 + lane); }
        else if (own_units) {
            first_id = own_id(0);
            if (own_units > 512) second_id = own_id(512);
        }
    };
    if (pre) fetch_ids();
    // what the parameters are needed for behind the wait, worked out before it: sources of Q and of the own page, destinations of the result rows
    constexpr int kUnits = NC * 16, kPer = (kUnits + kThreads - 1) / kThreads;
    const uint4* q_at[kPer];
    unsigned char* own_pool_at[kOwn];
    const unsigned char* own_new_at[kOwn];
    float2* ml_at = nullptr;
    float* lse_at = nullptr;
    float scale = p.scale_log2;
    int whole_rows = sp.nsplit == 1;   // results, not partials
    const int my_row = lane & (NH - 1), my_r = row_off + my_row;
    const bool merged_here = RH == 1 && p.cluster_size > 1 && sp.nsplit > 1;
    unsigned long long* const row_dst = (unsigned long long*)(smem + S::kDst) + warp * NH;
    if (!issuer) {
#pragma unroll
        for (int j = 0; j < kPer; ++j) {
            const int c = tid + j * kThreads, r = c >> 4;
            q_at[j] = nullptr;
            if (c < kUnits && r < n_rows) {
                const int i = div_g(row0 + r), hd = g * G + (row0 + r) - i * G;
                q_at[j] = (const uint4*)((const unsigned char*)p.q + ((long long)(sp.q_row0 + i) * p.hq + hd) * 256 + (c & 15) * 16);
            }
            hold(q_at[j]);
            // (8 rows over 1000 / 4096 tokens with Q in memory 7.17 / 7.77 -> 6.70 / 7.68 us a layer; a line of 128 bytes each: by every thread 3 x 700 tokens 6.30 -> 6.22)
            if (q_at[j] && (tid & 7) == 0) prefetch_l2(q_at[j]);
        }
#pragma unroll
        for (int j = 0; j < kOwn; ++j)
            if (j < kOwn1 || more_own) {
                own_pool_at[j] = own_pool(tid + j * kThreads); own_new_at[j] = own_new(tid + j * kThreads);
                hold(own_pool_at[j]); hold(own_new_at[j]);
                const int u = tid + j * kThreads, tok = own_tok(u);
                if ((tid & 7) == 0 && u < two_pages && tok < L) {
                    if (tok >= pool_end) prefetch_l2(own_new_at[j]);
                    else if (pre) {
                        const int id = u < 512 ? first_id : second_id;
                        if (id >= 0 && id < num_pages) prefetch_l2(own_pool_at[j] + (long long)id * page_bytes);
                    }
                }
            }
        if (tile < 2) {   // row my_row's, for all lanes of the warp through shared memory
            unsigned long long dst = 0;
            if (my_r < n_rows && !merged_here) {
                const int i = div_g(row0 + my_r), hd = g * G + (row0 + my_r) - i * G;
                if (sp.nsplit == 1) {
                    const long long at = (long long)(sp.q_row0 + i) * p.hq + hd;
                    dst = (unsigned long long)((unsigned char*)p.out + at * 256);
                    if (p.lse && tw == 0 && lane < NH) lse_at = p.lse + at;
                } else {
                    const long long e = (long long)sp.part_base + ((long long)i * p.hq + hd) * sp.nsplit + split;
                    dst = (unsigned long long)(p.part_o + e * 128);
                    if (tw == 0 && lane < NH) ml_at = p.part_ml + e;
                }
            }
            row_dst[my_row] = dst;
        }
    }
    hold(ml_at); hold(lse_at); hold(scale); hold(whole_rows); hold(num_pages); hold(page_bytes);
    if (issuer && lane == 0) {
        for (int i = 0; i < 3 * NT + 1; ++i) mbar_init(base + S::kBar + 8u * i, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        asm volatile("prefetch.tensormap [%0];\n" ::"l"(&map_k) : "memory");
        asm volatile("prefetch.tensormap [%0];\n" ::"l"(&map_v) : "memory");
    }
    pdl_launch_dependents();
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(tmem_slot)), "r"(kCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    if (!(issuer && pre)) pdl_wait();   // from here on global memory written by the launch before this one is read
    if (!pre) fetch_ids();
    if (issuer) {
        __syncwarp();
        int id = first_id;
        if (lane < n_pages && (id < 0 || id >= p.num_pages)) { id = 0; atomicOr(p.status, AGX_DEV_BAD_PAGE); }
        bool waited = !pre;
        if (!waited && !p.k_new && tok_end > (P & ~(kPage - 1))) { pdl_wait(); waited = true; }
        if (lane < n_tiles && lane != p.drop_stage) {   // (drop_stage, a test hook: this tile never arrives, its consumers' waits run out)
            const uint32_t bytes = 4096u * min(8, max(0, own_pg - lane * 8));
            mbar_arrive_expect_tx(k_bar(lane), bytes);
            mbar_arrive_expect_tx(v_bar(lane), bytes);
        }
        __syncwarp();   // the barriers are armed before any copy can complete on them
        const bool copies = lane < own_pg && (lane >> 3) != p.drop_stage;   // lane l copies page l, all of K first
        const int group = (id * p.hkv + g) * (kPage / 8);
        if (copies) tma_load_page(base + S::kK + lane * 4096, &map_k, group, k_bar(lane >> 3));
        __syncwarp();
        if (copies) tma_load_page(base + S::kV + lane * 4096, &map_v, group, v_bar(lane >> 3));
        __syncwarp();
        if (!waited) pdl_wait();
    } else {
        // Q: [half of 64 dims][NC rows][128 B], 128-byte swizzle; rows past q * G are zeros.  (All loads are issued before the first store.)
        uint4 v[kPer], w[kOwn];
#pragma unroll
        for (int j = 0; j < kPer; ++j) {
            v[j] = make_uint4(0, 0, 0, 0);
            if (q_at[j]) v[j] = __ldg(q_at[j]);
        }
#pragma unroll
        for (int j = 0; j < kOwn1; ++j)
            if (tid + j * kThreads < two_pages) w[j] = own_load(tid + j * kThreads, tid + j * kThreads < 512 ? first_id : second_id, own_pool_at[j], own_new_at[j]);
        if (more_own)
#pragma unroll
        for (int j = kOwn1; j < kOwn; ++j)
            if (tid + j * kThreads < two_pages) w[j] = own_load(tid + j * kThreads, tid + j * kThreads < 512 ? first_id : second_id, own_pool_at[j], own_new_at[j]);
#pragma unroll
        for (int j = 0; j < kPer; ++j) {
            const int c = tid + j * kThreads, r = c >> 4, ch = c & 15;
            if (c < kUnits) *(uint4*)(smem + S::kQ + (ch >> 3) * (NC * 128) + r * 128 + (((ch & 7) ^ (r & 7)) << 4)) = v[j];
        }
#pragma unroll
        for (int j = 0; j < kOwn1; ++j)
            if (tid + j * kThreads < two_pages) own_store(tid + j * kThreads, tid + j * kThreads < 512 ? first_id : second_id, own_pool_at[j], w[j]);
        if (more_own)
#pragma unroll
        for (int j = kOwn1; j < kOwn; ++j)
            if (tid + j * kThreads < two_pages) own_store(tid + j * kThreads, tid + j * kThreads < 512 ? first_id : second_id, own_pool_at[j], w[j]);
        for (int u = tid + 1024; u < own_units; u += kThreads) {
            const int id = own_id(u);
            own_store(u, id, own_pool(u), own_load(u, id, own_pool(u), own_new(u)));
        }
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();   // barriers, TMEM address, Q and the own pages are in place
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    // ---- S^T = K Q^T: tokens x rows, a tile at a time
    constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(NC >> 3) << 17) | ((128u >> 4) << 24);   // f32 += bf16 x bf16, M = 128, N = NC
    if (issuer) {
        if (elect_one()) {
            bool ok = true;
            for (int t = 0; t < n_tiles && ok; ++t) {
                ok = mbar_wait<kSuspendNs>(k_bar(t), 0, abort_flag, p.status, p.wait_limit_cycles);
                if (!ok) break;
                tc_fence_after();
                const uint64_t kd = make_desc(base + S::kK + t * kTile, 16, 2048), qd = make_desc(base + S::kQ, 16, 1024);
#pragma unroll
                for (int s = 0; s < 8; ++s)   // 8 k-steps of 16 dims
                    umma_ss(tmem + 32 + 32 * t, kd + (uint64_t)(((s >> 2) * 1024 + (s & 3) * 32) >> 4),
                            qd + (uint64_t)(((s >> 2) * (NC * 128) + (s & 3) * 32) >> 4), kIdesc, s > 0);
                umma_commit(s_bar(t));
            }
        }
        __syncwarp();
        asm volatile("bar.sync 1, %0;\n" ::"n"(kThreads + 32) : "memory");   // P is in place
        tc_fence_after();
        // ---- O^T = V^T P^T: head dims x rows, one k-step per page
        if (elect_one()) {
            bool ok = !*abort_flag;
            for (int t = 0; t < n_tiles && ok; ++t) {
                ok = mbar_wait<kSuspendNs>(v_bar(t), 0, abort_flag, p.status, p.wait_limit_cycles);
                if (!ok) break;
                tc_fence_after();
                const uint64_t vd = make_desc(base + S::kV + t * kTile, 1024, 2048), pd = make_desc(base + S::kP + t * (2 * NC * 128), 16, 1024);
                auto step = [&](int pg) {
                    umma_ss(tmem, vd + (uint64_t)((pg * 4096) >> 4), pd + (uint64_t)(((pg >> 2) * (NC * 128) + (pg & 3) * 32) >> 4),
                            kIdesc | (1u << 15), t > 0 || pg > 0);   // (bit 15: A = V is MN-major)
                };
                const int npg = n_pages - t * 8;
                if (npg >= 8) {
#pragma unroll
                    for (int pg = 0; pg < 8; ++pg) step(pg);
                } else {
                    for (int pg = 0; pg < npg; ++pg) step(pg);
                }
            }
            umma_commit(o_bar);   // (arrives at once where nothing was issued)
        }
        __syncwarp();
    }

    float* cl_o = (float*)(smem + S::kO);
    float2* cl_ml = (float2*)(smem + S::kO + NR * 512);
    if (!issuer) {
    // ---- one token per thread: mask, row maxima, P = 2^(S * scale - m)
    const uint32_t lanes = (uint32_t)((warp & 3) << 5) << 16;
    const int t_warp = tw * 32, tok = tok_begin + t_warp + lane;   // (t_warp: first token of the warp, from tok_begin)
    bool live = tile < n_tiles && __all_sync(0xFFFFFFFFu, mbar_wait<kSuspendNs>(s_bar(min(tile, NT - 1)), 0, abort_flag, p.status, p.wait_limit_cycles));
    float s[NH], x[NH];
    if (live) {
        tc_fence_after();
        tmem_ld<NH>(tmem + lanes + 32 + 32 * tile + row_off, (uint32_t*)s);
        tmem_wait_ld();
        if (tok_begin + t_warp + 31 > P || tok_begin + t_warp + 32 > tok_end) {   // rows below `lo` do not see this token
            const int lo = tok >= tok_end ? NR : (tok - P) * G - row0 - row_off;
#pragma unroll
            for (int r = 0; r < NH; ++r) if (r < lo) s[r] = -INFINITY;
        }
    } else {
#pragma unroll
        for (int r = 0; r < NH; ++r) s[r] = -INFINITY;
    }
    float* x_max = (float*)(smem + S::kMax);
    float* x_sum = (float*)(smem + S::kSum);
    float w_max = 0.f;   // (by shuffles as the sums are: one row / 8 rows over 4096 tokens 6.01 / 7.74 us a layer, with the merges' maxima, instead of 5.85 / 7.49)
#pragma unroll
    for (int r = 0; r < NH; ++r) { const float m = warp_max(s[r]); if (my_row == r) w_max = m; }
    x_max[tw * NR + my_r] = w_max * scale;   // (NH < 32: several lanes write the same)
    tc_fence_before();
    asm volatile("bar.sync 2, %0;\n" ::"n"(kThreads) : "memory");   // every warp's maxima; all scores are in registers, so K is dead
    tc_fence_after();
    float m_row = -INFINITY;   // of row my_row
#pragma unroll
    for (int w = 0; w < kTokenWarps; ++w) m_row = fmaxf(m_row, x_max[w * NR + my_r]);
    float* ref = (float*)(smem + S::kRef) + warp * NH;
    ref[my_row] = (m_row == -INFINITY) ? 0.f : -m_row;
    __syncwarp();
    if (tile < n_tiles) {
        const int t = t_warp + lane, c = (t & 63) >> 3;
        unsigned char* pt = smem + S::kP + (t >> 6) * (NC * 128) + row_off * 128 + (t & 7) * 2;
#pragma unroll
        for (int r4 = 0; r4 < NH; r4 += 4) {
            if (row_off + r4 >= n_rows) {   // (padding: the columns of O^T that come of it are not stored, whatever P holds)
                x[r4] = x[r4 + 1] = x[r4 + 2] = x[r4 + 3] = 0.f;
                continue;
            }
            const float4 nm = *(const float4*)(ref + r4);
            const float n[4] = {nm.x, nm.y, nm.z, nm.w};
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int r = r4 + k;
                x[r] = ex2(fmaf(s[r], scale, n[k]));
                *(__nv_bfloat16*)(pt + r * 128 + ((c ^ ((row_off + r) & 7)) << 4)) = __float2bfloat16_rn(x[r]);
            }
        }
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    } else {
#pragma unroll
        for (int r = 0; r < NH; ++r) x[r] = 0.f;
    }
    tc_fence_before();
    asm volatile("bar.arrive 1, %0;\n" ::"n"(kThreads + 32) : "memory");   // P is in place

    // ---- row sums, while O^T is under way
    const float w_sum = sum_across_lanes(x);
    x_sum[tw * NR + my_r] = w_sum;
    asm volatile("bar.sync 2, %0;\n" ::"n"(kThreads) : "memory");   // every warp's sums
    float l_row = 0.f;
#pragma unroll
    for (int w = 0; w < kTokenWarps; ++w) l_row += x_sum[w * NR + my_r];

    // ---- epilogue: lane = head dim, column = row; the warpgroups of the first two tiles take half of their rows each
    constexpr int kHalf = NH / 2;
    // weight of row my_row, for all lanes of the warp through shared memory (its copy of the row references is dead)
    if (tile < 2) {
        if (lse_at) *lse_at = (m_row + log2f(l_row)) * 0.6931471805599453f;
        if (ml_at) *ml_at = make_float2(m_row, l_row);
        ref[my_row] = (l_row > 0.f) ? 1.f / l_row : 0.f;
        __syncwarp();
    }
    const bool done = __all_sync(0xFFFFFFFFu, mbar_wait<kSuspendNs>(o_bar, 0, abort_flag, p.status, p.wait_limit_cycles));
    if (tile < 2) {
        float o[kHalf];
        if (done && n_tiles > 0) {
            tc_fence_after();
            tmem_ld<kHalf>(tmem + lanes + row_off + tile * kHalf, (uint32_t*)o);
            tmem_wait_ld();
        } else {
#pragma unroll
            for (int j = 0; j < kHalf; ++j) o[j] = 0.f;
        }
        const int d = (warp & 3) * 32 + lane;
        if (merged_here) {
            if (tw == 0 && lane < NH) cl_ml[my_r] = make_float2(m_row, l_row);
#pragma unroll
            for (int j = 0; j < kHalf; ++j) cl_o[(row_off + tile * kHalf + j) * 128 + d] = o[j];
        } else if (!whole_rows) {   // the un-normalised fp32 rows
#pragma unroll
            for (int j = 0; j < kHalf; ++j) {
                const unsigned long long at = row_dst[tile * kHalf + j];
                if (at) __stcg((float*)at + d, o[j]);
            }
        } else {
            // bf16 results: lane pairs swap so that the even lane stores two columns of the first
            // row of a pair, the odd lane two of the second
            const bool odd = lane & 1;
#pragma unroll
            for (int j = 0; j < kHalf; j += 2) {
                const float a = o[j] * ref[tile * kHalf + j], b = o[j + 1] * ref[tile * kHalf + j + 1];
                const float got = __shfl_xor_sync(0xFFFFFFFFu, odd ? a : b, 1);
                const float lo = odd ? got : a, hi = odd ? b : got;
                unsigned char* const at = (unsigned char*)row_dst[tile * kHalf + j + odd];
                if (at) *(uint32_t*)(at + (d & ~1) * 2) = pack_bf16(lo, hi);
            }
        }
    }
    }
    // After a wait gave up, copies armed above may still be on their way into shared memory: they land (bounded by the clock alone)
    // before the CTA reuses or releases it.
    if (issuer && lane == 0 && *abort_flag)
        for (int t = 0; t < n_tiles; ++t)
            if (t != p.drop_stage) { mbar_drain(k_bar(t), 0, p.wait_limit_cycles); mbar_drain(v_bar(t), 0, p.wait_limit_cycles); }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(kCols) : "memory");
    }
    if constexpr (RH == 1)
        if (merged_here) merge_cluster_rows<kWarps + 1>(p, sp, cl_o, cl_ml, g, split, row0, n_rows);   // (uniform over the cluster)
}

namespace {
template <int NR, int NT, int RH>
cudaError_t launch_swap(const AttnParams& p, const CUtensorMap& map_k, const CUtensorMap& map_v, cudaStream_t stream) {
    constexpr int kSmem = (int)Lay<NR, NT, RH>::kBytes;
    // the attribute is per device: remember which devices have it (a process normally drives one GPU)
    static bool configured_on[64] = {false};
    int device = 0;
    if (cudaGetDevice(&device) != cudaSuccess || device < 0 || device >= 64) return cudaErrorInvalidDevice;
    if (!configured_on[device]) {
        cudaError_t e = cudaFuncSetAttribute(attn_swap_bf16_kernel<NR, NT, RH>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
        if (e != cudaSuccess) return e;
        e = cudaFuncSetAttribute(attn_swap_bf16_kernel<NR, NT, RH>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);   // clusters of up to 16
        if (e != cudaSuccess) return e;
        configured_on[device] = true;
    }
    if (p.cluster_size > 1)
        return launch_chained_cluster(attn_swap_bf16_kernel<NR, NT, RH>, dim3(p.num_items), dim3(NT * 128 * RH + 32), kSmem, (unsigned)p.cluster_size, stream, p, map_k, map_v);
    return launch_chained(attn_swap_bf16_kernel<NR, NT, RH>, dim3(p.num_items), dim3(NT * 128 * RH + 32), kSmem, stream, p, map_k, map_v);
}

template <int NT>
cudaError_t launch_rows(const AttnParams& p, int rows, const CUtensorMap& map_k, const CUtensorMap& map_v, cudaStream_t stream) {
    if (rows <= 4) return launch_swap<4, NT, 1>(p, map_k, map_v, stream);
    // More than four rows and two tiles: two threads a token, each with half of its rows, so that butterflies, exponentials and stores are half as long.  One
    // layer, one thread a token / two: 8 rows of 32/8 heads over 3 x 700 tokens 8.46 / 6.80 us, 5 over 2 x 1500 8.47 / 7.04, 4 over 8 x 300 7.49 / 6.60, 8 over
    // 3000 7.64 / 7.01, 2 over 1000 7.08 / 6.48 (with Q on its way to L2 ahead of the wait, below).  Not for three tiles, whose 800 threads are slower (8 rows
    // over 4096 tokens 7.84 / 8.38: the third tile's scores, a third of a microsecond behind the first's, set the pace), nor for splits merged in
    // clusters (one row or two; not compiled: the merge's loads want 64 registers).
    if constexpr (NT == 2) {
        if (p.cluster_size <= 1)
            return rows <= 8 ? launch_swap<8, NT, 2>(p, map_k, map_v, stream)
                             : rows <= 16 ? launch_swap<16, NT, 2>(p, map_k, map_v, stream) : launch_swap<32, NT, 2>(p, map_k, map_v, stream);
    }
    return rows <= 8 ? launch_swap<8, NT, 1>(p, map_k, map_v, stream) : rows <= 16 ? launch_swap<16, NT, 1>(p, map_k, map_v, stream) : launch_swap<32, NT, 1>(p, map_k, map_v, stream);
}
}  // namespace

// One layer of one sequence, GQA 32/8, mma.sync kernel with the same splits -> this one: 8-row verify over 4096 / 1024 tokens 9.07 -> 8.08 / 7.77 ->
// 7.12 us, one row over 300 / 1500 / 4096 / 7000 tokens 5.08 -> 4.93 / 6.28 -> 6.01 / 6.78 -> 6.49 / 9.40 -> 9.37.  Only the rows that exist are
// worked on (one row with the softmax of 16: 7.01 us over 4096 tokens instead of 6.49).
// In 32 layers launched eagerly over 4096 tokens, with the merge, since then: one row 7.7 -> 6.3 us a layer, 8 rows 9.1 -> 8.0 (parameters held ahead of the
// dependency wait, own pages in one trip, a shorter last split, long suspensions).
cudaError_t launch_attn_swap(const AttnParams& p, int rows, int longest, const CUtensorMap& map_k, const CUtensorMap& map_v, cudaStream_t stream) {
    return longest <= 2 * kTileTok ? launch_rows<2>(p, rows, map_k, map_v, stream) : launch_rows<3>(p, rows, map_k, map_v, stream);
}

}  // namespace agx
