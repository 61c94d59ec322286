// Small-q attention over a paged KV cache: the verify block of speculative decoding (q = N + 1
// rows, Sec. 2.3) and plain decode (q = 1, the selective fallback of Sec. 4.3).
//
// The step is HBM-bound: every K and V byte of the sequence is read once and meets only q * G
// query rows (G = Hq / Hkv), i.e. q * G flop per KV byte.  That is above what the fp32 FMA pipes
// sustain at HBM speed once q * G > ~8, so the q * G rows of one KV head are packed into the M
// dimension of warp-level bf16 tensor-core MMAs (m16n8k16, fp32 accumulate): the kernel stays
// bandwidth-bound and verifying 8 tokens costs the same bytes as decoding 1.
//
// Work item = (sequence, KV head, KV split).  A CTA of KW * MT warps (KW = 4 or 8 KV groups): warp (mt, kg)
// owns query rows [16 mt, 16 mt + 16) and, in every stage of KW pages, page kg.  K/V pages stream through a
// 3-stage ring filled by TMA (per page one 4 KB box for K and one for V, SWIZZLE_128B so
// ldmatrix is conflict-free; page ids come from the page table, prefetched 32 at a time) and handed over
// with full/empty mbarriers, so no thread spends instructions on addresses.  Per stage the KV groups of an
// m-tile meet twice at a named barrier: once to agree on the rows' running maximum (page maxima through
// shared memory), once to hand round the pages' P (as MMA A fragments, 512 bytes per page).  Each warp
// then accumulates O over all pages of the stage, but only for the 128 / KW output columns it owns, so
// the accumulators never have to be merged: at the end only the row sums are added up.  KW = 8 (16 warps
// for a 32-row verify block, one CTA per SM) halves the number of page steps per warp.  Splits write
// fp32 (m, l, O) partials; a combine kernel merges them in fixed order, so results are bit-reproducible
// run to run.
#include <cuda_fp16.h>
#include <math.h>

#include <type_traits>

#include "agx_internal.cuh"

#include <algorithm>
#include "agx_sm100.cuh"

namespace agx {

namespace {

constexpr int kD = 128;                    // head dim of the bf16 kernels
constexpr int kRowBytes = kD * 2;          // one (token, head) row
// KW = KV groups = pages per pipeline stage (4 or 8): stage = KW * 16 tokens, K + V = KW * 8 KB



__device__ __forceinline__ void ldmatrix_x4(uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3, uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(addr));
}
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3, uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(addr));
}
// D(16x8, f32) += A(16x16, bf16, row) * B(16x8, bf16, col)
__device__ __forceinline__ void mma_bf16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// byte offset of 16-byte chunk `ch` (0..15) of row `r` in a [rows][256 B] tile, XOR-swizzled
__device__ __forceinline__ uint32_t swz(int r, int ch) { return (uint32_t)(r * kRowBytes + ((ch ^ (r & 7)) << 4)); }

// Loads the compiler keeps where they are written (and that go to L2: the data was just written by other SMs).
__device__ __forceinline__ uint2 ld_volatile_u2(const void* p) {
    uint2 v;
    asm volatile("ld.volatile.global.v2.u32 {%0, %1}, [%2];\n" : "=r"(v.x), "=r"(v.y) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ uint4 ld_volatile_u4(const void* p) {
    uint4 v;
    asm volatile("ld.volatile.global.v4.u32 {%0, %1, %2, %3}, [%4];\n" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ float4 ld_volatile_f4(const void* p) {
    float4 v;
    asm volatile("ld.volatile.global.v4.f32 {%0, %1, %2, %3}, [%4];\n" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ float2 ld_volatile_f2(const void* p) {
    float2 v;
    asm volatile("ld.volatile.global.v2.f32 {%0, %1}, [%2];\n" : "=f"(v.x), "=f"(v.y) : "l"(p) : "memory");
    return v;
}

}  // namespace

// Zeros in place of the V rows from `from` on of a page in the ring, once it has arrived (P is 0 there, but 0 * NaN is not).  The group barriers of
// the stage stand between this and the use of V.  
static __device__ __noinline__ void zero_v_tail(unsigned char* v_page, int from, uint32_t full, volatile int* abort_flag, int* status, long long limit) {
    const int lane = threadIdx.x & 31;
    if (!__all_sync(0xFFFFFFFFu, mbar_wait(full, 0, abort_flag, status, limit))) return;   // (the main loop's wait gives up too)
    for (int u = from * 16 + lane; u < kPage * 16; u += 32) {
        const int r = u >> 4, ch = u & 15;
        *(uint4*)(v_page + (r >> 3) * 2048 + (ch >> 3) * 1024 + (r & 7) * 128 + (((ch & 7) ^ (r & 7)) << 4)) = make_uint4(0, 0, 0, 0);
    }
}

// MW = m-tiles per warp: with MW = 2 a warp scores its page against both 16-row tiles of a 32-row block and accumulates
// both tiles' output columns, so every K and V fragment is read from shared memory once instead of twice.
// kByHand: pages that cannot come by TMA as they are, see own_pg below; two kernels, because what only one form needs costs the other 2-4 %
// wherever it stands.
template <int MT, int KW, int NS, int MW, bool kByHand>
__global__ void __launch_bounds__(32 * (MT / MW) * KW, ((MT / MW) * KW <= 8 && MW == 1) ? 2 : 1)
attn_small_bf16_kernel(const __grid_constant__ AttnParams p, const __grid_constant__ CUtensorMap map_k,
                       const __grid_constant__ CUtensorMap map_v) {
    extern __shared__ unsigned char smem_raw[];
    constexpr int kKW = KW;
    constexpr int kStageTokens = kKW * kPage;
    constexpr int kStageBytes = 2 * kStageTokens * kRowBytes;
    constexpr int kThreads = 32 * (MT / MW) * KW;
    constexpr int kWarps = (MT / MW) * KW;
    constexpr int kRingBytes = NS * kStageBytes;
    constexpr int kClusterBytes = MT * 16 * (kD * 4 + 8);   // this CTA's (O, m, l) rows, read by the cluster's other CTAs (in the dead ring)
    constexpr int kRegion = kRingBytes > kClusterBytes ? kRingBytes : kClusterBytes;
    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    unsigned char* ring = smem_raw + (smem_base - smem_u32(smem_raw));   // 1024-aligned: TMA swizzle atoms
    unsigned char* q_smem = ring + kRegion;
    const uint32_t bar_base = smem_base + kRegion + MT * 16 * kRowBytes;  // full[NS], empty[NS]
    volatile int* abort_flag = (volatile int*)(q_smem + MT * 16 * kRowBytes + 2 * NS * 8);
    // exchange area of the KV groups: per-page row maxima, per-group row sums, P fragments of the stage's pages
    float* x_max = (float*)(q_smem + MT * 16 * kRowBytes + 2 * NS * 8 + 16);   // [MT][16][KW]
    float* x_l = x_max + MT * 16 * KW;                                          // [MT][16][KW]
    uint4* x_p = (uint4*)(x_l + MT * 16 * KW);                                  // [MT][KW][32]
    auto full_bar = [&](int i) { return bar_base + 8u * i; };
    auto empty_bar = [&](int i) { return bar_base + 8u * (NS + i); };

    const int tid = threadIdx.x;
    const int lane = tid & 31;
    const int warp = tid >> 5;
    const int mt0 = (warp % (MT / MW)) * MW;   // first of this warp's MW m-tiles
    const int kg = warp / (MT / MW);

    const int si = find_seq(p, blockIdx.x);
    const SeqPlan sp = p.seq[si];
    const unsigned item = blockIdx.x - sp.item0;   // ((g * row_chunks) + rc) * nsplit + split
    const unsigned chunk = item / (unsigned)sp.nsplit;
    const int split = (int)(item - chunk * sp.nsplit);
    const int g = sp.row_chunks == 1 ? (int)chunk : (int)(chunk / (unsigned)sp.row_chunks);
    const int rc = (int)chunk - g * sp.row_chunks;
    const int G = p.gqa;
    // r / G without the division.  Signed divisions here, at the Q tile's addresses and in the epilogue cost a CTA 0.2-0.9 us in all (one
    // layer: 8-row verify over 1024 / 4096 tokens 8.29 -> 7.78 / 9.34 -> 9.09 us, 4 x 4096 18.4 -> 17.5, one row over 300 / 4096 5.34 -> 5.07
    // / 6.92 -> 6.74; one row over 16000 and more, bound by HBM, 15.3 -> 15.6).
    auto div_g = [&](int r) { return (int)(((uint64_t)(uint32_t)r * p.row_div_magic) >> 32); };
    const int P = sp.prefix_len;
    const int q = sp.q_len;
    const int L = P + q;
    const int rows = q * G;          // query rows of this KV head, r = i * G + (h % G)
    const int row0 = rc * 16 * MT;   // first row of this CTA's chunk
    // the chunk's last row sees tokens 0 .. P + i_last
    const int vis_end = P + min(q - 1, div_g(row0 + 16 * MT - 1)) + 1;
    const int tok_begin = split * sp.split_tokens;
    const int tok_end = min(vis_end, tok_begin + sp.split_tokens);
    const int n_stages = max(0, (tok_end - tok_begin + kStageTokens - 1) / kStageTokens);

    if (tid == 0) {
        for (int i = 0; i < NS; ++i) { mbar_init(full_bar(i), 1); mbar_init(empty_bar(i), kWarps); }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        asm volatile("prefetch.tensormap [%0];\n" ::"l"(&map_k) : "memory");
        asm volatile("prefetch.tensormap [%0];\n" ::"l"(&map_v) : "memory");
    }
    pdl_launch_dependents();
    const int* pt_row = p.page_table + (long long)sp.seq_index * p.pt_stride;
    const int page0 = tok_begin / kPage;
    const int n_pages = (tok_end - tok_begin + kPage - 1) / kPage;
    // With p.early_prefix (the caller vouches that the page table and the pages below the cached-prefix length are not written by a
    // launch still in flight) the producer warp fetches page ids and K/V stages that lie wholly inside the cached prefix before
    // the dependency wait, i.e. while the launch in front drains.
    const bool pre = p.early_prefix;
    // kByHand: the pages from own_pg on (counted from the split's first page) are put together by hand, beside the Q tile: with a fused append
    // those that hold block rows, which come from k_new / v_new and go into the pool on the way; otherwise a last page that is only partly valid
    // (what lies behind the last token may be anything, and V has to be zero there).  They are at the end of the sequence, and a split's stages are
    // worked off from its end, so they are always among the first in the ring.  A page of a cold pool fetched by hand holds the whole CTA up, so
    // that without an append short splits take the other form: every page by TMA, the last one's tail zeroed when it has arrived.
    const int pool_end = !kByHand ? (L + kPage - 1) & ~(kPage - 1) : p.k_new ? P : L;
    const int own_pg = min(n_pages, max(0, (pool_end >> 4) - page0));
    const int own_units = kByHand ? (n_pages - own_pg) * 512 : 0;   // 16-byte units, [page][K, V][16 rows][16 units]
    constexpr int kLoaders = kThreads - 32;           // all warps but the producer's
    constexpr int kOwn = (512 + kLoaders - 1) / kLoaders;   // a thread's units of the first own page
    auto own_id = [&](int u) { const int slot = page0 + own_pg + (u >> 9); return slot < p.pt_stride ? __ldg(pt_row + slot) : -1; };
    auto own_load = [&](int u, int id) {
        const int tok = tok_begin + (own_pg + (u >> 9)) * kPage + ((u >> 4) & 15), is_v = (u >> 8) & 1, ch = u & 15;
        uint4 v = make_uint4(0, 0, 0, 0);
        if (tok < pool_end) {
            const long long page = (id < 0 || id >= p.num_pages) ? 0 : id;   // (reported by fetch_ids)
            v = __ldcg((const uint4*)((const unsigned char*)(is_v ? p.v_pool : p.k_pool) + ((page * p.hkv + g) * kPage + (tok & 15)) * kRowBytes + ch * 16));
        } else if (tok < L) {
            v = __ldg((const uint4*)((const unsigned char*)(is_v ? p.v_new : p.k_new) + ((long long)(sp.q_row0 + tok - P) * p.hkv + g) * kRowBytes + ch * 16));
        }
        return v;
    };
    auto own_store = [&](int u, int id, const uint4 v) {
        const int pg = own_pg + (u >> 9), r = (u >> 4) & 15, is_v = (u >> 8) & 1, ch = u & 15, tok = tok_begin + pg * kPage + r;
        const int stage = pg / kKW;
        *(uint4*)(ring + ((n_stages - 1 - stage) % NS) * kStageBytes + is_v * (kStageTokens * kRowBytes) + (pg - stage * kKW) * 4096 +
                  (r >> 3) * 2048 + (ch >> 3) * 1024 + (r & 7) * 128 + (((ch & 7) ^ (r & 7)) << 4)) = v;
        if (tok >= pool_end && tok < L && id >= 0 && id < p.num_pages)
            *(uint4*)((unsigned char*)(is_v ? p.v_pool : p.k_pool) + (((long long)id * p.hkv + g) * kPage + (tok & 15)) * kRowBytes + ch * 16) = v;
    };
    int first_id[kOwn];
    auto fetch_own_ids = [&]() {
#pragma unroll
        for (int j = 0; j < kOwn; ++j)
            if (tid >= 32 && tid - 32 + j * kLoaders < own_units) first_id[j] = own_id(tid - 32 + j * kLoaders);
    };
    if (kByHand && pre) fetch_own_ids();         // (the caller vouches for the page table too)
    // Q and the block's own rows, on their way to L2 before the wait (one row: 4 x 2500 tokens 11.07 -> 10.82 us, 12 x 1000 13.79 -> 13.38, 12000
    // 12.43 -> 12.32), a line of 128 bytes each, by about the CTAs of the first wave: for others the wait is over.
    unsigned sms;
    asm("mov.u32 %0, %%nsmid;\n" : "=r"(sms));
    if (tid >= 32 && blockIdx.x < (KW == 4 && MT < 4 ? 2 : 1) * sms) {
        for (int c = 8 * (tid - 32); c < MT * 256; c += 8 * kLoaders) {
            const int r = row0 + (c >> 4), i = div_g(r);
            if (r < rows) prefetch_l2((const unsigned char*)p.q + ((long long)(sp.q_row0 + i) * p.hq + g * G + r - i * G) * kRowBytes + (c & 15) * 16);
        }
        if (kByHand && p.k_new)
            for (int u = 8 * (tid - 32); u < own_units; u += 8 * kLoaders) {
                const int tok = tok_begin + (own_pg + (u >> 9)) * kPage + ((u >> 4) & 15);
                if (tok >= P && tok < L)
                    prefetch_l2((const unsigned char*)(((u >> 8) & 1) ? p.v_new : p.k_new) + ((long long)(sp.q_row0 + tok - P) * p.hkv + g) * kRowBytes + (u & 15) * 16);
            }
    }
    if (!(warp == 0 && pre)) pdl_wait();   // from here on global memory written by the launch before this one is read
    if (kByHand && !pre) fetch_own_ids();
    // ---- producer state (warp 0; lane 0 issues the TMA copies).  Page ids are fetched 32 at a time,
    //      one group ahead, so the page-table latency never sits in front of a copy.
    int ids_cur = 0, ids_next = 0, group_cur = max(0, (n_stages - 1) * kKW) >> 5;
    auto fetch_ids = [&](int group) {
        const int pi = group * 32 + lane;
        long long id = 0;
        if (pi >= 0 && pi < n_pages) {
            id = __ldg(pt_row + page0 + pi);
            if (id < 0 || id >= p.num_pages) { id = 0; atomicOr(p.status, AGX_DEV_BAD_PAGE); }
        }
        return (int)id;
    };
    bool alive = true;
    int last_armed = -1;              // last stage whose copies were armed (lane 0 of warp 0)
    auto produce = [&](int stage) {   // called by all lanes of warp 0; `stage` counts from the end of the split
        if (stage >= n_stages || !alive) return;
        const int slot = stage % NS;
        alive = __all_sync(0xFFFFFFFFu, mbar_wait(empty_bar(slot), ((stage / NS) & 1) ^ 1, abort_flag, p.status, p.wait_limit_cycles));
        if (!alive) return;   // (the same answer in every lane: the lanes stay together for the shuffles and copies below)
        const int pi0 = (n_stages - 1 - stage) * kKW;
        if ((pi0 >> 5) != group_cur) { ids_cur = ids_next; group_cur = pi0 >> 5; ids_next = fetch_ids(group_cur - 1); }
        const int npg = min(kKW, n_pages - pi0);
        const int npool = min(npg, max(0, own_pg - pi0));   // pages that come from the pool
        if (stage == p.drop_stage) return;   // test hook: this stage never arrives, its consumers' waits run out
        if (lane == 0) last_armed = stage;
        if constexpr (MW == 2) {
            // lane pg copies page pg of K, lane KW + pg that of V
            const int id = __shfl_sync(0xFFFFFFFFu, ids_cur, (pi0 + (lane & (kKW - 1))) & 31);
            if (lane == 0) mbar_arrive_expect_tx(full_bar(slot), npool * 8192u);
            __syncwarp();   // the barrier is armed before any lane's copies can complete on it
            if (lane < 2 * kKW && (lane & (kKW - 1)) < npool)
                tma_load_page(smem_base + slot * kStageBytes + lane * 4096, lane < kKW ? &map_k : &map_v, (id * p.hkv + g) * (kPage / 8), full_bar(slot));
        } else {
            // One elected thread issues all copies of the stage: 4 x 4096 verify 18.9 -> 18.5 us, decode over 300 tokens 5.50 -> 5.37
            // (with two m-tiles per warp this form costs decode verify 9.83 -> 10.08, hence the other branch).
            int group[kKW];   // first row group of each page
#pragma unroll
            for (int pg = 0; pg < kKW; ++pg) group[pg] = (__shfl_sync(0xFFFFFFFFu, ids_cur, (pi0 + pg) & 31) * p.hkv + g) * (kPage / 8);
            if (elect_one()) {
                mbar_arrive_expect_tx(full_bar(slot), npool * 8192u);
                const uint32_t dk = smem_base + slot * kStageBytes, dv = dk + kStageTokens * kRowBytes;
#pragma unroll
                for (int pg = 0; pg < kKW; ++pg)
                    if (pg < npool) {
                        tma_load_page(dk + pg * 4096, &map_k, group[pg], full_bar(slot));
                        tma_load_page(dv + pg * 4096, &map_v, group[pg], full_bar(slot));
                    }
            }
            __syncwarp();
        }
    };
    // The producer lane set the barriers up itself, so it needs nothing else from the other warps: it fetches the page
    // ids and issues the first copies at once, while the others bring the Q tile in.
    if (warp == 0) {
        __syncwarp();   // lane 0's barrier initialisation, before the other lanes poll those barriers
        ids_cur = fetch_ids(group_cur);
        ids_next = fetch_ids(group_cur - 1);
        bool waited = !pre;
        const int stable_end = P & ~(kPage - 1);   // tokens below this sit in pages no append of this block touches
#pragma unroll 1
        for (int s = 0; s < NS - 1; ++s) {
            // (with a fused append only pages below stable_end come from the pool)
            if (!waited && !p.k_new && tok_begin + (n_stages - s) * kStageTokens > stable_end) { pdl_wait(); waited = true; }
            produce(s);
        }
        if (!waited) pdl_wait();
    }
    // ---- Q tile -> shared (rows beyond q*G are zero), by the warps other than the producer's
    //      (a thread's loads are all issued before its first store: one trip to memory, not one per 16-byte unit)
    if (tid >= 32) {
        constexpr int kUnits = MT * 16 * 16, kPer = (kUnits + kLoaders - 1) / kLoaders;
        uint4 v[kPer];
#pragma unroll
        for (int j = 0; j < kPer; ++j) {
            const int c = tid - 32 + j * kLoaders, r = c >> 4, ch = c & 15;
            v[j] = make_uint4(0, 0, 0, 0);
            if (c < kUnits && row0 + r < rows) {
                const int i = div_g(row0 + r), hg = (row0 + r) - i * G;
                const long long off = ((long long)(sp.q_row0 + i) * p.hq + g * G + hg) * kRowBytes + ch * 16;
                v[j] = __ldg((const uint4*)((const unsigned char*)p.q + off));
            }
        }
        // own pages: their loads go out behind Q's, before anything is stored
        uint4 w[kOwn];
        if constexpr (kByHand) {
#pragma unroll
        for (int j = 0; j < kOwn; ++j)
            if (tid - 32 + j * kLoaders < own_units) w[j] = own_load(tid - 32 + j * kLoaders, first_id[j]);
#pragma unroll
        for (int j = 0; j < kOwn; ++j)
            if (tid - 32 + j * kLoaders < own_units) own_store(tid - 32 + j * kLoaders, first_id[j], w[j]);
        for (int u = tid - 32 + kOwn * kLoaders; u < own_units; u += kLoaders) { const int id = own_id(u); own_store(u, id, own_load(u, id)); }
        }
#pragma unroll
        for (int j = 0; j < kPer; ++j) {
            const int c = tid - 32 + j * kLoaders;
            if (c < kUnits) *(uint4*)(q_smem + swz(c >> 4, c & 15)) = v[j];
        }
    }
    __syncthreads();  // barriers initialised, Q tile visible
    // The last page of the sequence is in the first stage to be worked off; the warps that score it zero what lies behind the last token.
    if (!kByHand && pool_end > L && n_pages > 0 && kg == n_pages - 1 - (n_stages - 1) * kKW && tok_begin + n_pages * kPage > L)
        zero_v_tail(ring + kStageTokens * kRowBytes + kg * 4096, L & (kPage - 1), full_bar(0), abort_flag, p.status, p.wait_limit_cycles);

    uint32_t qa[MW][8][4];
#pragma unroll
    for (int w = 0; w < MW; ++w) {
        const int r = (mt0 + w) * 16 + (lane & 7) + ((lane >> 3) & 1) * 8;
#pragma unroll
        for (int ks = 0; ks < 8; ++ks) {
            const int ch = ks * 2 + (lane >> 4);
            ldmatrix_x4(qa[w][ks][0], qa[w][ks][1], qa[w][ks][2], qa[w][ks][3], smem_u32(q_smem) + swz(r, ch));
        }
    }

    // Warp (mt, kg) scores page kg of every stage against its 16 rows (per m-tile), but accumulates O only for the kCG * 16
    // output columns it owns, over ALL pages of the stage: the P fragments of the stage's pages travel through shared
    // memory and the KV groups of an m-tile share one running maximum, so nothing has to be merged at the end.
    constexpr int kCG = 8 / KW;                    // 16-column groups of O per warp
    float o[MW][2 * kCG][4];
    float m_run[MW][2], l_run[MW][2];              // running maximum of rows g and g + 8 (log2 units) | this lane's share of the row sums
    int limit[MW][2];                              // last visible token of the two rows this thread holds
#pragma unroll
    for (int w = 0; w < MW; ++w) {
#pragma unroll
        for (int n = 0; n < 2 * kCG; ++n) { o[w][n][0] = o[w][n][1] = o[w][n][2] = o[w][n][3] = 0.f; }
        m_run[w][0] = m_run[w][1] = -INFINITY;
        l_run[w][0] = l_run[w][1] = 0.f;
        const int rA = row0 + (mt0 + w) * 16 + (lane >> 2);
        limit[w][0] = P + min(div_g(rA), q - 1);
        limit[w][1] = P + min(div_g(rA + 8), q - 1);
    }
    // Per-lane ldmatrix offsets inside one page of the TMA layout [row group 2][half 2][8 rows][128 B], where the
    // 16-byte unit u of row r sits at ((u ^ (r & 7)) << 4).  K (x4): row = nt*8 + lane%8, unit = (kp&1)*4 + lane/8.
    // V (x4.trans): row = lane%8 + 8*((lane/8)&1), unit = (cp&3)*2 + lane/16.
    const uint32_t k_x = ((lane >> 3) ^ (lane & 7));
    const uint32_t k_off[2] = {(uint32_t)((lane & 7) * 128 + (k_x << 4)), (uint32_t)((lane & 7) * 128 + ((k_x ^ 4u) << 4))};
    const uint32_t v_row = (lane & 7) + ((lane >> 3) & 1) * 8;
    const uint32_t v_x = (lane >> 4) ^ (lane & 7);
    uint32_t v_off[kCG];   // of this warp's 16-column groups cp = kg * kCG + c
#pragma unroll
    for (int c = 0; c < kCG; ++c) {
        const uint32_t cp = (uint32_t)(kg * kCG + c);
        v_off[c] = (v_row >> 3) * 2048 + (cp >> 2) * 1024 + (v_row & 7) * 128 + ((v_x ^ ((cp & 3) << 1)) << 4);
    }

    const int rg = lane >> 2;                      // this lane's rows in an m-tile: rg and rg + 8
    float* my_max = x_max + (mt0 * 16 + rg) * KW;  // x_max[mt][row][kg]; m-tile mt0 + w: + w * 16 * KW
    uint4* my_p = x_p + (mt0 * KW) * 32 + lane;    // x_p[mt][kg][lane]: page kg's P as the lanes' MMA A fragments; + w * KW * 32
    auto group_sync = [&]() { asm volatile("bar.sync %0, %1;\n" ::"r"(1 + mt0 / MW), "n"(32 * KW) : "memory"); };

    bool live = true;   // a warp whose wait gave up keeps meeting the others at the group barriers
#pragma unroll 1
    for (int stage = 0; stage < n_stages; ++stage) {
        const int slot = stage % NS;
        if (warp == 0) produce(stage + NS - 1);
        if (live) live = mbar_wait(full_bar(slot), (stage / NS) & 1, abort_flag, p.status, p.wait_limit_cycles);

        const int stage_tok0 = tok_begin + (n_stages - 1 - stage) * kStageTokens;
        const int npg = live ? min(kKW, (tok_end - stage_tok0 + kPage - 1) / kPage) : 0;   // pages of this stage
        const int tok0 = stage_tok0 + kg * kPage;
        const bool has_page = kg < npg;
        const uint32_t stage_base = smem_base + slot * kStageBytes;
        float s[MW][2][4];
        float mx[MW][2];
#pragma unroll
        for (int w = 0; w < MW; ++w) mx[w][0] = mx[w][1] = -INFINITY;
        if (has_page) {
            const uint32_t k_base = stage_base + kg * 4096;
            // S = Q K^T for 16 tokens: two n-tiles of 8 tokens, as four accumulation chains of four MMAs each per m-tile
            // (even and odd k-steps of both n-tiles): a dependent mma.sync is slow to issue.  A K fragment serves every m-tile.
            float s_odd[MW][2][4];
#pragma unroll
            for (int w = 0; w < MW; ++w) {
#pragma unroll
                for (int nt = 0; nt < 2; ++nt) {
                    s[w][nt][0] = s[w][nt][1] = s[w][nt][2] = s[w][nt][3] = 0.f;
                    s_odd[w][nt][0] = s_odd[w][nt][1] = s_odd[w][nt][2] = s_odd[w][nt][3] = 0.f;
                }
            }
#pragma unroll
            for (int kp = 0; kp < 4; ++kp) {
#pragma unroll
                for (int nt = 0; nt < 2; ++nt) {
                    uint32_t b0, b1, b2, b3;
                    ldmatrix_x4(b0, b1, b2, b3, k_base + (kp >> 1) * 1024 + nt * 2048 + k_off[kp & 1]);
#pragma unroll
                    for (int w = 0; w < MW; ++w) {
                        mma_bf16(s[w][nt], qa[w][2 * kp], b0, b1);
                        mma_bf16(s_odd[w][nt], qa[w][2 * kp + 1], b2, b3);
                    }
                }
            }
#pragma unroll
            for (int w = 0; w < MW; ++w) {
#pragma unroll
                for (int nt = 0; nt < 2; ++nt) {
#pragma unroll
                    for (int e = 0; e < 4; ++e) s[w][nt][e] += s_odd[w][nt][e];
                }
                // mask the causal edge / the end of the split (raw scores; the scale is folded into the exp)
                if ((tok0 + kPage - 1 > P) || (tok0 + kPage > tok_end)) {
#pragma unroll
                    for (int nt = 0; nt < 2; ++nt) {
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const int tok = tok0 + nt * 8 + 2 * (lane & 3) + (e & 1);
                            if (tok > limit[w][e >> 1] || tok >= tok_end) s[w][nt][e] = -INFINITY;
                        }
                    }
                }
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    float v = fmaxf(fmaxf(s[w][0][2 * h], s[w][0][2 * h + 1]), fmaxf(s[w][1][2 * h], s[w][1][2 * h + 1]));
                    v = fmaxf(v, __shfl_xor_sync(0xFFFFFFFFu, v, 1));
                    v = fmaxf(v, __shfl_xor_sync(0xFFFFFFFFu, v, 2));
                    mx[w][h] = v * p.scale_log2;
                }
            }
        }
        if ((lane & 3) == 0) {
#pragma unroll
            for (int w = 0; w < MW; ++w) { my_max[w * 16 * KW + kg] = mx[w][0]; my_max[w * 16 * KW + 8 * KW + kg] = mx[w][1]; }
        }
        group_sync();   // the stage's page maxima of this warp's m-tiles are in place

        // one running maximum per row for a whole m-tile; P of this warp's page against it
#pragma unroll
        for (int w = 0; w < MW; ++w) {
            float corr[2];
            uint32_t pa[4] = {0u, 0u, 0u, 0u};
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                float m_new = m_run[w][h];
#pragma unroll
                for (int k4 = 0; k4 < KW; k4 += 4) {
                    const float4 v = *(const float4*)(my_max + w * 16 * KW + h * 8 * KW + k4);
                    m_new = fmaxf(fmaxf(m_new, fmaxf(v.x, v.y)), fmaxf(v.z, v.w));
                }
                const float m_ref = (m_new == -INFINITY) ? 0.f : m_new;
                corr[h] = ex2(m_run[w][h] - m_ref);
                m_run[w][h] = m_new;
                float sum = 0.f;
                if (has_page) {
#pragma unroll
                    for (int nt = 0; nt < 2; ++nt) {
                        s[w][nt][2 * h] = ex2(fmaf(s[w][nt][2 * h], p.scale_log2, -m_ref));
                        s[w][nt][2 * h + 1] = ex2(fmaf(s[w][nt][2 * h + 1], p.scale_log2, -m_ref));
                        sum += s[w][nt][2 * h] + s[w][nt][2 * h + 1];
                    }
                }
                l_run[w][h] = l_run[w][h] * corr[h] + sum;
            }
            if (has_page) {
                pa[0] = pack_bf16(s[w][0][0], s[w][0][1]);
                pa[1] = pack_bf16(s[w][0][2], s[w][0][3]);
                pa[2] = pack_bf16(s[w][1][0], s[w][1][1]);
                pa[3] = pack_bf16(s[w][1][2], s[w][1][3]);
            }
            my_p[(w * KW + kg) * 32] = make_uint4(pa[0], pa[1], pa[2], pa[3]);
            if (__any_sync(0xFFFFFFFFu, corr[0] != 1.f || corr[1] != 1.f)) {
#pragma unroll
                for (int n = 0; n < 2 * kCG; ++n) {
                    o[w][n][0] *= corr[0]; o[w][n][1] *= corr[0];
                    o[w][n][2] *= corr[1]; o[w][n][3] *= corr[1];
                }
            }
        }
        group_sync();   // every page's P fragments are in place

        // O[:, this warp's columns] += P V over the stage's pages (a V fragment serves every m-tile)
#pragma unroll
        for (int k = 0; k < kKW; ++k) {
            if (k < npg) {
                uint4 pk[MW];
#pragma unroll
                for (int w = 0; w < MW; ++w) pk[w] = my_p[(w * KW + k) * 32];
                const uint32_t v_base = stage_base + kStageTokens * kRowBytes + k * 4096;
#pragma unroll
                for (int c = 0; c < kCG; ++c) {
                    uint32_t b0, b1, b2, b3;
                    ldmatrix_x4_trans(b0, b1, b2, b3, v_base + v_off[c]);
#pragma unroll
                    for (int w = 0; w < MW; ++w) {
                        const uint32_t a[4] = {pk[w].x, pk[w].y, pk[w].z, pk[w].w};
                        mma_bf16(o[w][2 * c], a, b0, b1);
                        mma_bf16(o[w][2 * c + 1], a, b2, b3);
                    }
                }
            }
        }
        __syncwarp();
        if (live && lane == 0) mbar_arrive(empty_bar(slot));
    }

    // ---- row sums of the m-tile: each KV group's share through shared memory
#pragma unroll
    for (int w = 0; w < MW; ++w) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            l_run[w][h] += __shfl_xor_sync(0xFFFFFFFFu, l_run[w][h], 1);
            l_run[w][h] += __shfl_xor_sync(0xFFFFFFFFu, l_run[w][h], 2);
        }
        if ((lane & 3) == 0) {
            x_l[((mt0 + w) * 16 + rg) * KW + kg] = l_run[w][0];
            x_l[((mt0 + w) * 16 + rg + 8) * KW + kg] = l_run[w][1];
        }
    }
    // After a wait gave up, copies armed by the producer lane may still be on their way into the ring: it waits for
    // them (bounded by the clock alone) before the CTA reuses or releases that shared memory.
    if (tid == 0 && *abort_flag) {
        for (int s = max(0, last_armed - NS + 1); s <= last_armed; ++s)
            if (s != p.drop_stage) mbar_drain(full_bar(s % NS), (s / NS) & 1, p.wait_limit_cycles);
    }
    __syncthreads();  // all row sums in place; every armed stage has been consumed: the ring is dead

    // With clusters, the KV splits of this (sequence, KV head) are the cluster's CTAs (rank = split): the split
    // results stay in shared memory and are merged across the cluster below instead of going through global memory.
    const bool in_cluster = p.cluster_size > 1;
    float* cl_o = (float*)ring;                              // [MT*16][kD]
    float2* cl_ml = (float2*)(ring + MT * 16 * kD * 4);      // [MT*16]
#pragma unroll
    for (int wh = 0; wh < 2 * MW; ++wh) {
        const int w = wh >> 1, h = wh & 1;
        const int r = (mt0 + w) * 16 + rg + 8 * h;           // row of the CTA's chunk
        if (row0 + r >= rows) continue;
        float l_all = 0.f;
#pragma unroll
        for (int k4 = 0; k4 < KW; k4 += 4) {
            const float4 v = *(const float4*)(x_l + r * KW + k4);
            l_all += (v.x + v.y) + (v.z + v.w);
        }
        const float m_all = m_run[w][h];
        const int i = div_g(row0 + r), hg = (row0 + r) - i * G;
        const int hd = g * G + hg;
        const bool first = kg == 0 && (lane & 3) == 0;       // one lane per row writes the row's (m, l)
        if (sp.nsplit == 1) {
            const float inv = 1.f / l_all;
            __nv_bfloat16* orow = (__nv_bfloat16*)p.out + ((long long)(sp.q_row0 + i) * p.hq + hd) * kD;
#pragma unroll
            for (int n = 0; n < 2 * kCG; ++n)
                *(uint32_t*)(orow + (kg * kCG * 2 + n) * 8 + 2 * (lane & 3)) = pack_bf16(o[w][n][2 * h] * inv, o[w][n][2 * h + 1] * inv);
            if (p.lse && first) p.lse[(long long)(sp.q_row0 + i) * p.hq + hd] = (m_all + log2f(l_all)) * 0.6931471805599453f;
        } else {
            if (in_cluster) {
                float* orow = cl_o + r * kD;
                if (first) cl_ml[r] = make_float2(m_all, l_all);
#pragma unroll
                for (int n = 0; n < 2 * kCG; ++n)
                    *(float2*)(orow + (kg * kCG * 2 + n) * 8 + 2 * (lane & 3)) = make_float2(o[w][n][2 * h], o[w][n][2 * h + 1]);
            } else {
                // split partial for the merge kernel, the un-normalised fp32 row, written past the L1 (read next by other SMs)
                const long long e = (long long)sp.part_base + ((long long)i * p.hq + hd) * sp.nsplit + split;
                if (first) p.part_ml[e] = make_float2(m_all, l_all);
                float* orow = p.part_o + e * kD;
#pragma unroll
                for (int n = 0; n < 2 * kCG; ++n)
                    __stcg((float2*)(orow + (kg * kCG * 2 + n) * 8 + 2 * (lane & 3)), make_float2(o[w][n][2 * h], o[w][n][2 * h + 1]));
            }
        }
    }
    if (in_cluster && sp.nsplit > 1) merge_cluster_rows<kWarps>(p, sp, cl_o, cl_ml, g, split, row0, min(rows - row0, MT * 16));
}

// --------------------------------------------------------------------------------------------
// Merges of split partials: out[row, h] = sum_k O_k 2^(m_k - m) / sum_k l_k 2^(m_k - m), splits in index order.

// Where 16-byte unit u of split 0's fp16 partial of row i, head h lies.
__device__ __forceinline__ const unsigned char* half_row(const AttnParams& p, const SeqPlan& sp, int i, int h, int u) {
    const int g = (int)(((uint64_t)(uint32_t)h * p.row_div_magic) >> 32), r = i * p.gqa + h - g * p.gqa, rl = r & 255;
    return (const unsigned char*)p.part_o + (long long)sp.part_base * 512 + (((long long)g * sp.row_chunks + (r >> 8)) * sp.nsplit) * 65536 + (u >> 3) * 32768 + rl * 128 +
           (((u ^ rl) & 7) << 4);
}
// The fp16 partials of row i, head h, four columns a lane: split 0's, and the bytes from split to split.
struct HalfRows {
    const unsigned char* at;
    int stride;
    __device__ __forceinline__ HalfRows(const AttnParams& p, const SeqPlan& sp, int i, int h, int lane)
        : at(half_row(p, sp, i, h, lane >> 1) + (lane & 1) * 8), stride(65536) {}
    __device__ __forceinline__ uint2 load(int split) const { return ld_volatile_u2(at + (long long)split * stride); }   // (written by other SMs just before: past the L1)
};
// What an fp16 row was divided by, where it was: its sum is negative then, and `exp` is not whatever was there.  (The merges of up to 32
// splits read it with the sum in any case: a branch on the way to the weights costs them 0.1 to 0.3 us, the load a third of that; the merge of more splits
// reads it where it is needed.)
__device__ __forceinline__ float row_scale(float sum, int exp) { return sum < 0.f ? pow2(exp) : 1.f; }
__device__ __forceinline__ int ld_volatile_s8(const signed char* p) {
    int v;
    asm volatile("ld.volatile.global.s8 %0, [%1];\n" : "=r"(v) : "l"(p) : "memory");
    return v;
}
// The same of the fp32 partials (columns [4 lane, 4 lane + 4)).
struct F32Rows {
    const unsigned char* at;
    int stride;
    __device__ __forceinline__ F32Rows(const AttnParams& p, const SeqPlan& sp, int i, int h, int lane) {
        if (p.part_half == PART_F32_TILES) {
            const int g = (int)(((uint64_t)(uint32_t)h * p.row_div_magic) >> 32), r = i * p.gqa + h - g * p.gqa, rows = sp.q_len * p.gqa;
            at = (const unsigned char*)p.part_o + ((long long)sp.part_base + (long long)g * sp.nsplit * rows) * 512 + ((lane >> 3) * rows + r) * 128 +
                 (((lane ^ r) & 7) << 4);
            stride = rows * 512;
        } else {
            at = (const unsigned char*)p.part_o + ((long long)sp.part_base + ((long long)i * p.hq + h) * sp.nsplit) * (p.head_dim * 4) + lane * 16;
            stride = p.head_dim * 4;
        }
    }
    __device__ __forceinline__ float4 load(int split) const { return ld_volatile_f4((const float*)(at + (long long)split * stride)); }
};
// fp32 partials, one warp per (row, head), a lane 4 columns.  kMaxNs: no sequence of the launch has more splits than this (4, 16 or 32; attn_combine_many_kernel
// takes more).  Four O rows per warp instead of 32 keep the register count low enough for ten CTAs per SM.
template <bool kBf16Out, int kMaxNs>
__global__ void __launch_bounds__(128, kMaxNs <= 4 ? 10 : kMaxNs <= 16 ? 5 : 3)
attn_combine_kernel(const __grid_constant__ AttnParams p, int total_rows) {
    constexpr bool kFew = kMaxNs <= 16;          // no second batch of 16 rows
    constexpr int kInFlight = kMaxNs <= 4 ? 4 : 16;
    pdl_launch_dependents();
    // (everything up to the wait depends on the kernel arguments only and runs while the attention kernel drains)
    const int lane = threadIdx.x & 31;
    const int rh = blockIdx.x * 4 + (threadIdx.x >> 5);  // index over (local row, head) of the launch's sequences
    if (rh >= total_rows * p.hq) return;
    const int lrow = rh / p.hq, h = rh - lrow * p.hq;
    // sequences are laid out back to back in launch-local row order
    int si = 0, acc_rows = 0;
#pragma unroll 1
    for (int s = 0; s < p.num_seqs; ++s) {
        if (lrow >= acc_rows && lrow < acc_rows + p.seq[s].q_len) { si = s; break; }
        acc_rows += p.seq[s].q_len;
    }
    const SeqPlan sp = p.seq[si];
    if (sp.nsplit == 1) return;  // written directly by the attention kernel
    const int i = lrow - acc_rows;
    const long long e0 = (long long)sp.part_base + ((long long)i * p.hq + h) * sp.nsplit;
    const int ns = sp.nsplit;
    const int D = p.head_dim;
    const int c4 = lane * 4;               // each lane owns 4 output columns
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    float m_all, l_all;
    const float2* ml_at = p.part_ml + e0 + lane;
    F32Rows rows(p, sp, i, h, lane);
    const long long out_row = (long long)(sp.q_row0 + i) * p.hq + h;
    unsigned char* out_at = (unsigned char*)p.out + (out_row * D + c4) * (kBf16Out ? 2 : 4);
    float* lse_at = p.lse ? p.lse + out_row : nullptr;
    hold(ml_at); hold(rows.at); hold(rows.stride); hold(out_at); hold(lse_at);
    pdl_wait();   // the partials are complete
    // One round trip to memory: lane k fetches (m, l) of split k while every lane already fetches its
    // columns of every split's O row; the weights then travel by shuffle, splits in index order.
    // (volatile loads: the compiler leaves them in this order, ahead of the first use of any of them)
    float2 ml = make_float2(-INFINITY, 0.f);
    if (lane < ns) ml = ld_volatile_f2(ml_at);
    float4 v[kInFlight], v2[kFew ? 1 : 16];
#pragma unroll
    for (int j = 0; j < kInFlight; ++j)
        if (j < ns && c4 < D) v[j] = rows.load(j);
    if (!kFew && ns > 16) {
#pragma unroll
        for (int j = 0; j < 16; ++j)
            if (16 + j < ns && c4 < D) v2[j] = rows.load(16 + j);
    }
    m_all = ml.x;
    m_all = warp_max(m_all);
    const float e_mine = (ml.x == -INFINITY) ? 0.f : exp2f(ml.x - m_all);
    l_all = ml.y * e_mine;
    const float w_mine = e_mine;   // weight of this lane's split's O row
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) l_all += __shfl_xor_sync(0xFFFFFFFFu, l_all, off);
#pragma unroll
    for (int j = 0; j < kInFlight; ++j) {
        const float w = __shfl_sync(0xFFFFFFFFu, w_mine, j);
        if (j < ns && w != 0.f && c4 < D) {   // a split that saw no token for this row publishes only (m, l) = (-inf, 0)
            acc.x += v[j].x * w; acc.y += v[j].y * w; acc.z += v[j].z * w; acc.w += v[j].w * w;
        }
    }
    if (!kFew && ns > 16) {
#pragma unroll
        for (int j = 0; j < 16; ++j) {
            const float w = __shfl_sync(0xFFFFFFFFu, w_mine, 16 + j);
            if (16 + j < ns && w != 0.f && c4 < D) {
                acc.x += v2[j].x * w; acc.y += v2[j].y * w; acc.z += v2[j].z * w; acc.w += v2[j].w * w;
            }
        }
    }
    const float inv = 1.f / l_all;
    if (c4 < D) {
        if (kBf16Out) {
            uint2 packed;
            packed.x = pack_bf16(acc.x * inv, acc.y * inv);
            packed.y = pack_bf16(acc.z * inv, acc.w * inv);
            *(uint2*)out_at = packed;
        } else {
            *(float4*)out_at = make_float4(acc.x * inv, acc.y * inv, acc.z * inv, acc.w * inv);
        }
    }
    if (lse_at && lane == 0) *lse_at = (m_all + log2f(l_all)) * 0.6931471805599453f;
}

// The same merge where a sequence has more than 32 splits (long contexts over few KV heads): one CTA per (row, head), whose warps take
// kManyBatch splits each with all their loads in flight, and the first warp adds the warps' sums in order.  Bound by one trip to memory
// as the kernels for fewer splits are; one warp per pair went through the splits four at a time, a trip each (one layer, 16/2 heads, one row
// over 12000 / 20000 / 55000 tokens, 47 to 74 splits: 12.0 / 17.9 / 22.4 -> 6.8 / 9.2 / 14.5 us; 8 rows over 34000 24.0 -> 15.8).
constexpr int kManyBatch = 16, kManyWarps = 16;   // (256 splits in one trip; more go round)
template <bool kBf16Out, bool kHalfPart>
__global__ void __launch_bounds__(kManyWarps * 32)
attn_combine_many_kernel(const __grid_constant__ AttnParams p, int total_rows) {
    __shared__ float4 s_acc[kManyWarps][32];
    __shared__ float2 s_ml[kManyWarps];
    pdl_launch_dependents();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
    const int lrow = blockIdx.x / p.hq, h = blockIdx.x - lrow * p.hq;
    int si = 0, acc_rows = 0;
#pragma unroll 1
    for (int s = 0; s < p.num_seqs; ++s) {
        if (lrow >= acc_rows && lrow < acc_rows + p.seq[s].q_len) { si = s; break; }
        acc_rows += p.seq[s].q_len;
    }
    const SeqPlan& sp = p.seq[si];
    const int ns = sp.nsplit, D = p.head_dim, c4 = lane * 4, i = lrow - acc_rows;
    if (ns == 1) return;   // written directly by the attention kernel
    const long long e0 = (long long)sp.part_base + ((long long)i * p.hq + h) * ns;
    std::conditional_t<kHalfPart, HalfRows, F32Rows> rows(p, sp, i, h, lane);
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    float m = -INFINITY, l = 0.f;
    const float2* ml_at = p.part_ml + e0 + lane;
    const long long out_row = (long long)(sp.q_row0 + i) * p.hq + h;
    unsigned char* out_at = (unsigned char*)p.out + (out_row * D + c4) * (kBf16Out ? 2 : 4);
    float* lse_at = p.lse ? p.lse + out_row : nullptr;
    hold(ml_at); hold(out_at); hold(lse_at); hold(rows.at); hold(rows.stride);
    pdl_wait();   // the partials are complete
    for (int k0 = warp * kManyBatch; k0 < ns; k0 += warps * kManyBatch) {
        const int n = min(kManyBatch, ns - k0);
        float2 ml = make_float2(-INFINITY, 0.f);
        if (lane < n) ml = ld_volatile_f2(ml_at + k0);
        // (the rows as they come: converted where they are loaded, one load waited for the other, one row over 12000 tokens with 16/2 heads 7.5 -> 11.1 us)
        std::conditional_t<kHalfPart, uint2, float4> v[kManyBatch];
#pragma unroll
        for (int j = 0; j < kManyBatch; ++j)
            if (j < n && c4 < D) v[j] = rows.load(k0 + j);
        float m_new = warp_max(ml.x);
        m_new = fmaxf(m, m_new);
        const float e = (ml.x == -INFINITY) ? 0.f : exp2f(ml.x - m_new), keep = (m == -INFINITY) ? 0.f : exp2f(m - m_new);
        float sum = (kHalfPart ? fabsf(ml.y) : ml.y) * e;
        float w_mine = kHalfPart ? sum : e;
        if (kHalfPart && ml.y < 0.f) w_mine *= pow2(ld_volatile_s8(p.part_exp + (ml_at - p.part_ml) + k0));
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, off);
        l = l * keep + sum;
        acc.x *= keep; acc.y *= keep; acc.z *= keep; acc.w *= keep;
#pragma unroll
        for (int j = 0; j < kManyBatch; ++j) {
            const float w = __shfl_sync(0xFFFFFFFFu, w_mine, j);
            if (j < n && w != 0.f && c4 < D) {   // a split that saw no token for this row publishes only (m, l) = (-inf, 0)
                float4 x;
                if constexpr (kHalfPart) {
                    const float2 a = __half22float2(*reinterpret_cast<const __half2*>(&v[j].x)), b = __half22float2(*reinterpret_cast<const __half2*>(&v[j].y));
                    x = make_float4(a.x, a.y, b.x, b.y);
                } else {
                    x = v[j];
                }
                acc.x += x.x * w; acc.y += x.y * w; acc.z += x.z * w; acc.w += x.w * w;
            }
        }
        m = m_new;
    }
    s_acc[warp][lane] = acc;
    if (lane == 0) s_ml[warp] = make_float2(m, l);
    __syncthreads();
    if (warp != 0 || c4 >= D) return;
    float m_all = -INFINITY, l_all = 0.f;
    for (int w = 0; w < warps; ++w) m_all = fmaxf(m_all, s_ml[w].x);
    acc = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int w = 0; w < warps; ++w) {
        const float2 ml = s_ml[w];
        const float e = (ml.x == -INFINITY) ? 0.f : exp2f(ml.x - m_all);
        const float4 a = s_acc[w][lane];
        l_all += ml.y * e;
        acc.x += a.x * e; acc.y += a.y * e; acc.z += a.z * e; acc.w += a.w * e;
    }
    const float inv = 1.f / l_all;
    if (kBf16Out) {
        uint2 packed;
        packed.x = pack_bf16(acc.x * inv, acc.y * inv);
        packed.y = pack_bf16(acc.z * inv, acc.w * inv);
        *(uint2*)out_at = packed;
    } else {
        *(float4*)out_at = make_float4(acc.x * inv, acc.y * inv, acc.z * inv, acc.w * inv);
    }
    if (lse_at && lane == 0) *lse_at = (m_all + log2f(l_all)) * 0.6931471805599453f;
}

// The same merge for fp16 partials (rows divided by their own sums) of at most kNs <= 8 splits: half a warp merges a (row, head) pair, a lane eight
// columns, lane k of the half holding split k's (m, l), all loads in flight at once.  Bound by instructions and by the CTAs of a wave before anything
// else: the merge of a split prefill is thousands of pairs (12288 and 9 MB for 512 tokens of 24 heads), each with its row's address to work out.  16 bytes
// a lane are half the loads and half the address arithmetic of a warp a pair.
// (One layer, one warp a pair and four columns a lane / this: 512 rows over 3072 tokens, 24/8 heads 27.3 / 26.0 us, 128 over 1000 13.2 / 11.8, 200 over
// 1500 17.7 / 17.1, 300 over 2000, 40/8, 22.3 / 20.7, 700 over 8000 90.3 / 88.0, six decode blocks over 1000 8.06 / 7.79.  Two pairs a half-warp with
// their loads in flight together: 128 over 1000 as fast, 512 over 3072 26.3.)
template <int kNs>
__global__ void __launch_bounds__(128, kNs <= 4 ? 12 : 8)
attn_combine_few_kernel(const __grid_constant__ AttnParams p, int total_rows) {
    pdl_launch_dependents();
    const int u = threadIdx.x & 15;
    const int rh = blockIdx.x * 8 + (threadIdx.x >> 4);
    const float2* ml_at = nullptr;
    const signed char* exp_at = nullptr;
    unsigned char* out_at = nullptr;
    float* lse_at = nullptr;
    const unsigned char* rows = nullptr;
    int ns = 0;
    if (rh < total_rows * p.hq) {
        const int lrow = rh / p.hq, h = rh - lrow * p.hq;
        int si = 0, acc_rows = 0;
#pragma unroll 1
        for (int s = 0; s < p.num_seqs; ++s) {
            if (lrow >= acc_rows && lrow < acc_rows + p.seq[s].q_len) { si = s; break; }
            acc_rows += p.seq[s].q_len;
        }
        const SeqPlan& sp = p.seq[si];
        if (sp.nsplit > 1) {   // (a single split was written directly by the attention kernel)
            const int i = lrow - acc_rows;
            ns = sp.nsplit;
            const long long out_row = (long long)(sp.q_row0 + i) * p.hq + h;
            const long long e = (long long)sp.part_base + ((long long)i * p.hq + h) * sp.nsplit + u;
            ml_at = p.part_ml + e; exp_at = p.part_exp + e;
            out_at = (unsigned char*)p.out + out_row * (kD * 2) + u * 16;
            lse_at = p.lse ? p.lse + out_row : nullptr;
            rows = half_row(p, sp, i, h, u);
        }
    }
    hold(ns); hold(ml_at); hold(exp_at); hold(out_at); hold(lse_at); hold(rows);
    pdl_wait();   // the partials are complete
    float2 ml = make_float2(-INFINITY, 0.f);
    int exp = 0;
    if (u < ns) { ml = ld_volatile_f2(ml_at); exp = ld_volatile_s8(exp_at); }
    uint4 v[kNs];
#pragma unroll
    for (int k = 0; k < kNs; ++k)
        if (k < ns) v[k] = ld_volatile_u4(rows + k * 65536);
    float m_all = ml.x;
#pragma unroll
    for (int off = kNs / 2; off > 0; off >>= 1) m_all = fmaxf(m_all, __shfl_xor_sync(0xFFFFFFFFu, m_all, off));   // splits sit in lanes 0 .. kNs - 1
    float l_all = (ml.x == -INFINITY) ? 0.f : exp2f(ml.x - m_all) * fabsf(ml.y);
    const float w_mine = l_all * row_scale(ml.y, exp);
#pragma unroll
    for (int off = kNs / 2; off > 0; off >>= 1) l_all += __shfl_xor_sync(0xFFFFFFFFu, l_all, off);   // (a fixed order: reproducible)
    m_all = __shfl_sync(0xFFFFFFFFu, m_all, 0, 16);
    l_all = __shfl_sync(0xFFFFFFFFu, l_all, 0, 16);
    float acc[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) acc[c] = 0.f;
#pragma unroll
    for (int k = 0; k < kNs; ++k) {
        const float w = __shfl_sync(0xFFFFFFFFu, w_mine, k, 16);
        if (k < ns && w != 0.f) {   // a split that saw no token for this row publishes only (m, l) = (-inf, 0): its row may hold anything, NaN included
            const uint32_t x[4] = {v[k].x, v[k].y, v[k].z, v[k].w};
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const float2 a = __half22float2(*reinterpret_cast<const __half2*>(&x[c]));
                acc[2 * c] += a.x * w; acc[2 * c + 1] += a.y * w;
            }
        }
    }
    if (ns == 0) return;
    const float inv = 1.f / l_all;
    uint4 packed;
    packed.x = pack_bf16(acc[0] * inv, acc[1] * inv);
    packed.y = pack_bf16(acc[2] * inv, acc[3] * inv);
    packed.z = pack_bf16(acc[4] * inv, acc[5] * inv);
    packed.w = pack_bf16(acc[6] * inv, acc[7] * inv);
    *(uint4*)out_at = packed;
    if (lse_at && u == 0) *lse_at = (m_all + log2f(l_all)) * 0.6931471805599453f;
}

// The same merge for the fp16 partials of more splits (9 to 32): one (row, head) pair per warp, lane k holding split k's (m, l) and every lane four columns
// of every split's row, all loads in flight at once.  CTAs of two warps with few registers, 12 or 7 of them per SM.
template <int kNsMax>
__global__ void __launch_bounds__(64, kNsMax <= 20 ? 12 : 7)
attn_combine_half32_kernel(const __grid_constant__ AttnParams p, int total_rows) {
    pdl_launch_dependents();
    const int lane = threadIdx.x & 31;
    const int rh = blockIdx.x * 2 + (threadIdx.x >> 5);
    int ns = 1, si = 0, acc_rows = 0, lrow = 0, h = 0;
    if (rh < total_rows * p.hq) {
        lrow = rh / p.hq; h = rh - lrow * p.hq;
#pragma unroll 1
        for (int s = 0; s < p.num_seqs; ++s) {
            if (lrow >= acc_rows && lrow < acc_rows + p.seq[s].q_len) { si = s; break; }
            acc_rows += p.seq[s].q_len;
        }
        ns = p.seq[si].nsplit;
    }
    if (ns > 1) {   // (a single split was written directly by the attention kernel)
        const SeqPlan& sp = p.seq[si];
        const int i = lrow - acc_rows;
        const long long out_row = (long long)(sp.q_row0 + i) * p.hq + h;
        const long long e = (long long)sp.part_base + ((long long)i * p.hq + h) * ns + lane;
        const float2* ml_at = p.part_ml + e;
        const signed char* exp_at = p.part_exp + e;
        unsigned char* out_at = (unsigned char*)p.out + out_row * (kD * 2) + lane * 8;
        float* lse_at = p.lse ? p.lse + out_row : nullptr;
        HalfRows rows(p, sp, i, h, lane);
        hold(ml_at); hold(exp_at); hold(out_at); hold(lse_at); hold(rows.at); hold(rows.stride); hold(ns);
        pdl_wait();   // the partials are complete
        // Every load is issued before the first use of any of them: volatile loads keep their place in the instruction stream
        // (left to itself the compiler moved the row loads behind the reduction of the maxima, i.e. behind a first trip to
        // memory: 0.6 us on decode verify).  No branch between the loads: slots past the last split repeat its row, and weigh
        // nothing below.
        uint2 v[kNsMax];
#pragma unroll
        for (int k = 0; k < kNsMax; ++k) v[k] = rows.load(min(k, ns - 1));
        float2 ml = make_float2(-INFINITY, 0.f);
        int exp = 0;
        if (lane < ns) { ml = ld_volatile_f2(ml_at); exp = ld_volatile_s8(exp_at); }
        const float m_all = warp_max(ml.x);
        float l_all = (ml.x == -INFINITY) ? 0.f : exp2f(ml.x - m_all) * fabsf(ml.y);   // 0 in lanes past the last split
        const float w_mine = l_all * row_scale(ml.y, exp);
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) l_all += __shfl_xor_sync(0xFFFFFFFFu, l_all, off);   // (a fixed order: reproducible)
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int k = 0; k < kNsMax; ++k) {
            const float w = __shfl_sync(0xFFFFFFFFu, w_mine, k);
            // a split that saw no token for this row publishes only (m, l) = (-inf, 0): its row may hold anything, NaN included
            const bool use = w != 0.f;
            const float2 a = __half22float2(*reinterpret_cast<const __half2*>(&v[k].x));
            const float2 b = __half22float2(*reinterpret_cast<const __half2*>(&v[k].y));
            acc.x += use ? a.x * w : 0.f; acc.y += use ? a.y * w : 0.f; acc.z += use ? b.x * w : 0.f; acc.w += use ? b.y * w : 0.f;
        }
        const float inv = 1.f / l_all;
        uint2 packed;
        packed.x = pack_bf16(acc.x * inv, acc.y * inv);
        packed.y = pack_bf16(acc.z * inv, acc.w * inv);
        *(uint2*)out_at = packed;
        if (lse_at && lane == 0) *lse_at = (m_all + log2f(l_all)) * 0.6931471805599453f;
    }
}

// --------------------------------------------------------------------------------------------
namespace {
template <int MT, int KW, int NS>
constexpr int small_smem_bytes() {
    constexpr int kClusterBytes = MT * 16 * (kD * 4 + 8);
    constexpr int kRing = NS * 2 * KW * kPage * kRowBytes;
    constexpr int kExchange = 2 * MT * 16 * KW * 4 + MT * KW * 32 * 16;
    // [ring | cluster rows][Q tile][2 * NS barriers + abort flag][exchange area] + slack for the 1024-byte alignment
    return (kRing > kClusterBytes ? kRing : kClusterBytes) + MT * 16 * kRowBytes + 2 * NS * 8 + 16 + kExchange + 1024;
}

template <int MT, int KW, int NS, int MW, bool kByHand>
cudaError_t launch_form(const AttnParams& p, const CUtensorMap& map_k, const CUtensorMap& map_v, cudaStream_t stream) {
    constexpr int kSmem = small_smem_bytes<MT, KW, NS>();
    // the attribute is per device: remember which devices have it (a process normally drives one GPU)
    static bool configured_on[64] = {false};
    int device = 0;
    if (cudaGetDevice(&device) != cudaSuccess || device < 0 || device >= 64) return cudaErrorInvalidDevice;
    bool& configured = configured_on[device];
    if (!configured) {
        cudaError_t e = cudaFuncSetAttribute(attn_small_bf16_kernel<MT, KW, NS, MW, kByHand>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
        if (e != cudaSuccess) return e;
        e = cudaFuncSetAttribute(attn_small_bf16_kernel<MT, KW, NS, MW, kByHand>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);   // clusters of up to 16
        if (e != cudaSuccess) return e;
        configured = true;
    }
    if (p.cluster_size > 1)
        return launch_chained_cluster(attn_small_bf16_kernel<MT, KW, NS, MW, kByHand>, dim3(p.num_items), dim3(32 * (MT / MW) * KW), kSmem,
                                      (unsigned)p.cluster_size, stream, p, map_k, map_v);
    return launch_chained(attn_small_bf16_kernel<MT, KW, NS, MW, kByHand>, dim3(p.num_items), dim3(32 * (MT / MW) * KW), kSmem, stream, p, map_k, map_v);
}

template <int MT, int KW, int NS, int MW = 1>
cudaError_t launch_small(const AttnParams& p, const CUtensorMap& map_k, const CUtensorMap& map_v, cudaStream_t stream) {
    // Without an append, splits of up to 512 tokens on two CTAs per SM by TMA alone: one layer, 48 x (300, 1) 23.0 -> 18.2 us, 12 x (1000, 4)
    // 14.9 -> 12.0, 24 x (1000, 1) 24.6 -> 23.1; a longer chain hides the trip (24 x (6000, 1) 121 by hand, 125 the other way), and so does the one
    // CTA of an SM with 8-page stages (one row over 8000 10.1 / 10.6, over 12000 12.4 / 12.9).
    if constexpr (KW == 4) {
        int longest = 0;
        for (int i = 0; i < p.num_seqs; ++i) longest = std::max(longest, p.seq[i].split_tokens);
        if (!p.k_new && longest <= 512) return launch_form<MT, KW, NS, MW, false>(p, map_k, map_v, stream);
    }
    return launch_form<MT, KW, NS, MW, true>(p, map_k, map_v, stream);
}

template <int MT, int KW, int NS, int MW = 1>
int max_clusters(int cluster) {
    static int cached[64][17];   // 0 = not asked yet, else 1 + answer
    int device = 0;
    if (cluster < 2 || cluster > 16 || cudaGetDevice(&device) != cudaSuccess || device < 0 || device >= 64) return 0;
    if (cached[device][cluster]) return cached[device][cluster] - 1;
    constexpr int kSmem = small_smem_bytes<MT, KW, NS>();
    int n = 0;
    if (cudaFuncSetAttribute(attn_small_bf16_kernel<MT, KW, NS, MW, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem) == cudaSuccess &&
        cudaFuncSetAttribute(attn_small_bf16_kernel<MT, KW, NS, MW, true>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(cluster * 64); cfg.blockDim = dim3(32 * (MT / MW) * KW); cfg.dynamicSmemBytes = kSmem;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = cluster; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr; cfg.numAttrs = 1;
        if (cudaOccupancyMaxActiveClusters(&n, attn_small_bf16_kernel<MT, KW, NS, MW, true>, &cfg) != cudaSuccess) { (void)cudaGetLastError(); n = 0; }
    } else {
        (void)cudaGetLastError();
    }
    cached[device][cluster] = n + 1;
    return n;
}
}  // namespace

// 32-row blocks on 8-page stages: both m-tiles in every warp (8 warps; decode verify 9.84 -> 9.42 us) or, with AGX_SMALL_MW=1,
// one m-tile per warp (16 warps).  On 4-page stages two tiles per warp are slower (4 x 4096 verify 20.1 -> 20.3 us).
static bool two_tiles_per_warp() {
    static const bool on = !(getenv("AGX_SMALL_MW") && atoi(getenv("AGX_SMALL_MW")) == 1);
    return on;
}

int attn_small_max_clusters(int mt, int kw, int cluster) {
    if (mt == 2 && kw == 8 && two_tiles_per_warp()) return max_clusters<2, 8, 3, 2>(cluster);
    switch (mt * 16 + kw) {
        case 1 * 16 + 4: return max_clusters<1, 4, 3>(cluster);
        case 2 * 16 + 4: return max_clusters<2, 4, 3>(cluster);
        case 1 * 16 + 8: return max_clusters<1, 8, 3>(cluster);
        case 2 * 16 + 8: return max_clusters<2, 8, 3>(cluster);
        case 4 * 16 + 4: return max_clusters<4, 4, 5>(cluster);
        default: return 0;
    }
}

cudaError_t launch_attn_small_bf16(const AttnParams& p, int mt, int kw, const CUtensorMap& map_k, const CUtensorMap& map_v,
                                   cudaStream_t stream) {
    if (p.num_items == 0) return cudaSuccess;
    int longest = 0, rows = 0;
    bool one_chunk = true;
    for (int i = 0; i < p.num_seqs; ++i) {
        longest = std::max(longest, p.seq[i].split_tokens);
        rows = std::max(rows, std::min(p.seq[i].q_len * p.gqa, 16 * mt));
        one_chunk &= p.seq[i].row_chunks == 1;
    }
    // splits that fit one CTA whole (figures there)
    if (kw == 8 && mt <= 2 && one_chunk && longest <= kSwapMaxTokens) return launch_attn_swap(p, rows, longest, map_k, map_v, stream);
    if (mt == 2 && kw == 8 && two_tiles_per_warp()) return launch_small<2, 8, 3, 2>(p, map_k, map_v, stream);
    switch (mt * 16 + kw) {
        case 1 * 16 + 4: return launch_small<1, 4, 3>(p, map_k, map_v, stream);
        case 2 * 16 + 4: return launch_small<2, 4, 3>(p, map_k, map_v, stream);
        case 1 * 16 + 8: return launch_small<1, 8, 3>(p, map_k, map_v, stream);
        case 2 * 16 + 8: return launch_small<2, 8, 3>(p, map_k, map_v, stream);
        case 4 * 16 + 4: return launch_small<4, 4, 5>(p, map_k, map_v, stream);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_attn_combine(const AttnParams& p, int dtype, int total_rows, cudaStream_t stream) {
    const long long n = (long long)total_rows * p.hq;
    if (n == 0) return cudaSuccess;
    const int blocks = (int)((n + 3) / 4);
    int ns_max = 1;
    for (int i = 0; i < p.num_seqs; ++i) ns_max = p.seq[i].nsplit > ns_max ? p.seq[i].nsplit : ns_max;
    const int many_threads = 32 * std::min(kManyWarps, (ns_max + kManyBatch - 1) / kManyBatch);
    if (p.part_half == PART_HALF_TILES) {
        if (ns_max <= 8)
            return launch_chained(ns_max <= 4 ? attn_combine_few_kernel<4> : attn_combine_few_kernel<8>, dim3((unsigned)((n + 7) / 8)), dim3(128), 0, stream, p, total_rows);
        if (ns_max <= 32) {
            if (ns_max <= 12) return launch_chained(attn_combine_half32_kernel<12>, dim3((int)((n + 1) / 2)), dim3(64), 0, stream, p, total_rows);
            if (ns_max <= 20) return launch_chained(attn_combine_half32_kernel<20>, dim3((int)((n + 1) / 2)), dim3(64), 0, stream, p, total_rows);
            return launch_chained(attn_combine_half32_kernel<32>, dim3((int)((n + 1) / 2)), dim3(64), 0, stream, p, total_rows);
        }
        return launch_chained(attn_combine_many_kernel<true, true>, dim3((unsigned)n), dim3(many_threads), 0, stream, p, total_rows);
    }
    if (dtype == AGX_BF16) {
        if (ns_max <= 4) return launch_chained(attn_combine_kernel<true, 4>, dim3(blocks), dim3(128), 0, stream, p, total_rows);
        if (ns_max <= 16) return launch_chained(attn_combine_kernel<true, 16>, dim3(blocks), dim3(128), 0, stream, p, total_rows);
        if (ns_max <= 32) return launch_chained(attn_combine_kernel<true, 32>, dim3(blocks), dim3(128), 0, stream, p, total_rows);
        return launch_chained(attn_combine_many_kernel<true, false>, dim3((unsigned)n), dim3(many_threads), 0, stream, p, total_rows);
    }
    if (ns_max <= 4) return launch_chained(attn_combine_kernel<false, 4>, dim3(blocks), dim3(128), 0, stream, p, total_rows);
    if (ns_max <= 16) return launch_chained(attn_combine_kernel<false, 16>, dim3(blocks), dim3(128), 0, stream, p, total_rows);
    if (ns_max <= 32) return launch_chained(attn_combine_kernel<false, 32>, dim3(blocks), dim3(128), 0, stream, p, total_rows);
    return launch_chained(attn_combine_many_kernel<false, false>, dim3((unsigned)n), dim3(many_threads), 0, stream, p, total_rows);
}

}  // namespace agx
