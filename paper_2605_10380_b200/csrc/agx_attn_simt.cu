// Attention for fp32 pools (any q, head_dim 64 or 128) and for bf16 pools with head_dim 64: fp32 arithmetic on the FMA pipes.
//
// Work item = (sequence, KV head, chunk of 8 query rows, KV split); CTA = 8 warps.  Per tile of 64 tokens all threads bring K and V into
// shared memory (one trip, every load in flight), score 8 x 64 pairs (a thread: one token, two rows), warp r does the softmax of
// row r, and warp w adds up the tokens [8 w, 8 w + 8) of the tile for all rows, so that V is read from shared memory once; the
// warps' sums meet at the end.  The KV splits of an item form a thread-block cluster and are merged through distributed
// shared memory; contexts that take more than 16 splits leave partials for the merge kernel.  With a fused append the block's
// rows come from k_new / v_new, and the item of a head's last row chunk stores them into the pages.
//
// Bounded by latency at the sizes it is meant for.  256 cached tokens, q = 4, 4/2 heads, fp32: 5.0 us in one launch; append, attention and
// merge were three launches of 27 us together, of which a kernel whose warps took one token at a time was most.  A second tile in
// a row costs a CTA 2.3-3.2 us (page ids, loads, four barriers), so that contexts of more than 16 tiles are better split further than a
// cluster reaches, with partials and the merge launch: 1500 tokens, head_dim 128 11.5 us in clusters, 8.1 with partials.
#include <math.h>

#include "agx_internal.cuh"
#include "agx_sm100.cuh"

namespace agx {

namespace {

constexpr int kR = 8;          // query rows per CTA
constexpr int kT = 64;         // tokens per tile
constexpr int kWarps = 8;
constexpr int kThreads = 32 * kWarps;

template <int D>
struct SimtSmem {
    float q[kR][D];
    float k[kT][D + 4];        // (a row's 16-byte units start four banks after the row's before it: conflict-free)
    float v[kT][D];
    float s[kR][kT];
    float o[kR][D];            // the split's rows, read by the cluster's other CTAs
    float corr[kR];
    float2 ml[kR];
    int odd;                   // != 0: V of the block holds a value that is not finite
};

// Four elements of a row at element offset `at` as floats.
template <bool kBf16>
__device__ __forceinline__ float4 load4(const void* base, long long at) {
    if (kBf16) {
        const uint2 r = __ldcg((const uint2*)((const __nv_bfloat16*)base + at));
        return make_float4(__uint_as_float(r.x << 16), __uint_as_float(r.x & 0xFFFF0000u), __uint_as_float(r.y << 16), __uint_as_float(r.y & 0xFFFF0000u));
    }
    return __ldcg((const float4*)((const float*)base + at));
}
template <bool kBf16>
__device__ __forceinline__ void store4(void* base, long long at, float4 v) {
    if (kBf16) *(uint2*)((__nv_bfloat16*)base + at) = make_uint2(pack_bf16(v.x, v.y), pack_bf16(v.z, v.w));
    else *(float4*)((float*)base + at) = v;
}

// The tile's products where V holds values that are not finite: a row stops at its last visible token.  Out of line, so that the kernel's
// instructions stay in one piece (inline it cost every launch 0.25 us).
template <int D>
__device__ __noinline__ void add_visible(const SimtSmem<D>& sm, float (&acc)[kR][D / 32], int t0, int P, int q, int row0, int G) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int t = warp * 8; t < warp * 8 + 8; ++t)
        for (int r = 0; r < kR; ++r)
            if (t0 + t <= P + min((row0 + r) / G, q - 1))
                for (int c = 0; c < D / 32; ++c) acc[r][c] += sm.s[r][t] * sm.v[t][c * 32 + lane];
}

}  // namespace

template <int D, bool kBf16>
__global__ void __launch_bounds__(kThreads, 2)
attn_simt_kernel(const __grid_constant__ AttnParams p) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    SimtSmem<D>& sm = *(SimtSmem<D>*)smem_raw;
    constexpr int kUnits = D / 4;                              // groups of four elements per row
    constexpr int kPer = kT * kUnits / kThreads;               // per thread and operand
    constexpr int kCols = D / 32;                              // output columns per lane
    pdl_launch_dependents();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const SeqPlan& sp = p.seq[find_seq(p, blockIdx.x)];
    int local = blockIdx.x - sp.item0;                         // ((g * row_chunks) + rc) * nsplit + split
    const int nsplit = sp.nsplit, split = local % nsplit;
    local /= nsplit;
    const int rc = local % sp.row_chunks, g = local / sp.row_chunks;
    const int G = p.gqa, P = sp.prefix_len, q = sp.q_len, L = P + q, rows = q * G, row0 = rc * kR;
    auto div_g = [&](int r) { return (int)(((uint64_t)(uint32_t)r * p.row_div31) >> p.row_div_shift); };   // r / G without the division
    auto row_of = [&](int r) { const int i = div_g(r); return (long long)(sp.q_row0 + i) * p.hq + g * G + r - i * G; };   // of q and out
    const int vis_end = P + min(q - 1, div_g(row0 + kR - 1)) + 1;
    const int tok_begin = split * sp.split_tokens, tok_end = min(vis_end, tok_begin + sp.split_tokens);
    const int pool_end = p.k_new ? P : L;
    const bool writer = p.k_new && rc == sp.row_chunks - 1;
    const int* pt_row = p.page_table + (long long)sp.seq_index * p.pt_stride;
    // the first tile's page ids may be read before the dependency wait if the caller vouches for the page table
    auto page_id = [&](int tok) {
        const bool need = tok < tok_end && (tok < pool_end || writer);
        return !need ? 0 : (tok >> 4) < p.pt_stride ? __ldg(pt_row + (tok >> 4)) : -1;
    };
    int id[kPer];
    if (p.early_prefix) {
#pragma unroll
        for (int j = 0; j < kPer; ++j) id[j] = page_id(tok_begin + (tid + j * kThreads) / kUnits);
    }
    // what the parameters are needed for behind the wait, worked out before it (the kernel is a chain of latencies; with this and without
    // divisions behind the wait 256 cached tokens, q = 4, 4/2 heads, fp32 with its acceptance 8.8 -> 8.1 us)
    static_assert(kR * kUnits <= kThreads, "one unit of Q per thread");
    const bool has_q = tid < kR * kUnits && row0 + tid / kUnits < rows;
    const unsigned char* q_at = (const unsigned char*)p.q + (row_of(has_q ? row0 + tid / kUnits : 0) * D + (tid % kUnits) * 4) * (kBf16 ? 2 : 4);
    const void *k_pool = p.k_pool, *v_pool = p.v_pool, *k_new = p.k_new, *v_new = p.v_new;
    int num_pages = (int)min(p.num_pages, 0x7FFFFFFFll), hkv = p.hkv;
    float scale = p.scale_log2;
    hold(q_at); hold(k_pool); hold(v_pool); hold(k_new); hold(v_new); hold(num_pages); hold(hkv); hold(scale);
    // the first result of this thread (of its cluster's share where there is one)
    const bool in_cluster = p.cluster_size > 1;
    const int out0 = in_cluster ? split + nsplit * tid : tid;
    unsigned char* out_at = nullptr;
    float* lse_at = nullptr;
    if (out0 < kR * kUnits && row0 + out0 / kUnits < rows && (in_cluster || nsplit == 1)) {
        const long long at = row_of(row0 + out0 / kUnits);
        out_at = (unsigned char*)p.out + (at * D + (out0 % kUnits) * 4) * (kBf16 ? 2 : 4);
        if (p.lse && out0 % kUnits == 0) lse_at = p.lse + at;
    }
    hold(out_at); hold(lse_at);
    pdl_wait();
    if (!p.early_prefix) {
#pragma unroll
        for (int j = 0; j < kPer; ++j) id[j] = page_id(tok_begin + (tid + j * kThreads) / kUnits);
    }
    // Q (a unit per thread), scaled so that the scores are in log2 units; rows past q * G are zeros
    float4 qx = make_float4(0.f, 0.f, 0.f, 0.f);
    if (has_q) qx = load4<kBf16>(q_at, 0);
    float acc[kR][kCols];
#pragma unroll
    for (int r = 0; r < kR; ++r)
#pragma unroll
        for (int c = 0; c < kCols; ++c) acc[r][c] = 0.f;
    float m_run = -INFINITY, l_run = 0.f;                      // of row `warp`
    const int st = tid & (kT - 1), sr = (tid / kT) * 2;        // this thread's token and first row in the scoring step
    const int lim0 = P + min(div_g(row0 + sr), q - 1), lim1 = P + min(div_g(row0 + sr + 1), q - 1);

    const int hidden = P + div_g(row0) + 1;                       // the first token that not every row sees
    if (tid == 0) sm.odd = 0;
    for (int t0 = tok_begin; t0 < tok_end; t0 += kT) {
        float4 kv[2][kPer];
#pragma unroll
        for (int j = 0; j < kPer; ++j) {
            const int u = tid + j * kThreads, tok = t0 + u / kUnits, c = (u % kUnits) * 4;
            kv[0][j] = kv[1][j] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (tok >= tok_end) continue;
            const long long page = id[j];
            const bool ok = page >= 0 && page < num_pages;
            if (!ok) atomicOr(p.status, AGX_DEV_BAD_PAGE);
            const long long slot = ((page * hkv + g) * kPage + (tok & 15)) * (long long)D + c;
            if (tok < pool_end) {
                if (ok) { kv[0][j] = load4<kBf16>(k_pool, slot); kv[1][j] = load4<kBf16>(v_pool, slot); }
            } else {
                const long long at = ((long long)(sp.q_row0 + tok - P) * hkv + g) * D + c;
                kv[0][j] = load4<kBf16>(k_new, at); kv[1][j] = load4<kBf16>(v_new, at);
                if (writer && ok) { store4<kBf16>((void*)k_pool, slot, kv[0][j]); store4<kBf16>((void*)v_pool, slot, kv[1][j]); }
            }
        }
        __syncthreads();                                       // the tile before this one has been used
        if (t0 == tok_begin && tid < kR * kUnits)
            *(float4*)&sm.q[tid / kUnits][(tid % kUnits) * 4] = make_float4(qx.x * scale, qx.y * scale, qx.z * scale, qx.w * scale);
#pragma unroll
        for (int j = 0; j < kPer; ++j) {
            const int u = tid + j * kThreads;
            *(float4*)&sm.k[u / kUnits][(u % kUnits) * 4] = kv[0][j];
            *(float4*)&sm.v[u / kUnits][(u % kUnits) * 4] = kv[1][j];
        }
        if (t0 + kT > hidden) {   // (a weight of 0 does not hide a value that is not finite from a row that must not see it)
#pragma unroll
            for (int j = 0; j < kPer; ++j) {
                const float4 v = kv[1][j];
                if (v.x * 0.f + v.y * 0.f + v.z * 0.f + v.w * 0.f != 0.f) sm.odd = 1;
            }
        }
        __syncthreads();
        if (t0 + kT < tok_end) {                               // page ids of the next tile
#pragma unroll
            for (int j = 0; j < kPer; ++j) id[j] = page_id(t0 + kT + (tid + j * kThreads) / kUnits);
        }
        {
            float s0[4] = {0.f, 0.f, 0.f, 0.f}, s1[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 8
            for (int c = 0; c < D; c += 4) {
                const float4 k = *(const float4*)&sm.k[st][c], a = *(const float4*)&sm.q[sr][c], b = *(const float4*)&sm.q[sr + 1][c];
                s0[0] += a.x * k.x; s0[1] += a.y * k.y; s0[2] += a.z * k.z; s0[3] += a.w * k.w;
                s1[0] += b.x * k.x; s1[1] += b.y * k.y; s1[2] += b.z * k.z; s1[3] += b.w * k.w;
            }
            const int tok = t0 + st;
            sm.s[sr][st] = (tok <= lim0 && tok < tok_end) ? (s0[0] + s0[1]) + (s0[2] + s0[3]) : -INFINITY;
            sm.s[sr + 1][st] = (tok <= lim1 && tok < tok_end) ? (s1[0] + s1[1]) + (s1[2] + s1[3]) : -INFINITY;
        }
        __syncthreads();
        {   // warp r: softmax of row r
            const float2 x = *(const float2*)&sm.s[warp][2 * lane];
            const float mx = warp_max(fmaxf(x.x, x.y));
            const float m_new = fmaxf(m_run, mx), m_ref = m_new == -INFINITY ? 0.f : m_new;
            const float corr = exp2f(m_run - m_ref);
            const float2 w = make_float2(exp2f(x.x - m_ref), exp2f(x.y - m_ref));
            float sum = w.x + w.y;
#pragma unroll
            for (int d = 16; d > 0; d >>= 1) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, d);
            l_run = l_run * corr + sum;
            m_run = m_new;
            *(float2*)&sm.s[warp][2 * lane] = w;
            if (lane == 0) sm.corr[warp] = corr;
        }
        __syncthreads();
        float4 w0[kR], w1[kR];
#pragma unroll
        for (int r = 0; r < kR; ++r) {
            const float corr = sm.corr[r];
            w0[r] = *(const float4*)&sm.s[r][warp * 8];
            w1[r] = *(const float4*)&sm.s[r][warp * 8 + 4];
#pragma unroll
            for (int c = 0; c < kCols; ++c) acc[r][c] *= corr;
        }
        if (__builtin_expect(sm.odd, 0)) {
            float a[kR][kCols];
#pragma unroll
            for (int r = 0; r < kR; ++r)
#pragma unroll
                for (int c = 0; c < kCols; ++c) a[r][c] = acc[r][c];
            add_visible(sm, a, t0, P, q, row0, G);
#pragma unroll
            for (int r = 0; r < kR; ++r)
#pragma unroll
                for (int c = 0; c < kCols; ++c) acc[r][c] = a[r][c];
            continue;
        }
#pragma unroll
        for (int t = 0; t < 8; ++t) {
            float v[kCols];
#pragma unroll
            for (int c = 0; c < kCols; ++c) v[c] = sm.v[warp * 8 + t][c * 32 + lane];
#pragma unroll
            for (int r = 0; r < kR; ++r) {
                const float4& w = t < 4 ? w0[r] : w1[r];
                const float x = (t & 3) == 0 ? w.x : (t & 3) == 1 ? w.y : (t & 3) == 2 ? w.z : w.w;
#pragma unroll
                for (int c = 0; c < kCols; ++c) acc[r][c] += x * v[c];
            }
        }
    }
    // ---- the warps' sums, in warp order: [warp][row][D] in the K / V area
    __syncthreads();
    float* part = &sm.k[0][0];
    static_assert(sizeof(sm.k) + sizeof(sm.v) >= sizeof(float) * kWarps * kR * D, "the partial sums of the warps fit the K / V tiles");
#pragma unroll
    for (int r = 0; r < kR; ++r)
#pragma unroll
        for (int c = 0; c < kCols; ++c) part[(warp * kR + r) * D + c * 32 + lane] = acc[r][c];
    if (lane == 0) sm.ml[warp] = make_float2(m_run, l_run);
    __syncthreads();
    for (int i = tid; i < kR * kUnits; i += kThreads) {   // (once: kR * kUnits <= kThreads)
        const int rl = i / kUnits, c = (i % kUnits) * 4, r = row0 + rl;
        float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int w = 0; w < kWarps; ++w) {
            const float4 x = *(const float4*)&part[(w * kR + rl) * D + c];
            o.x += x.x; o.y += x.y; o.z += x.z; o.w += x.w;
        }
        const float2 ml = sm.ml[rl];
        if (in_cluster) {
            *(float4*)&sm.o[rl][c] = o;
        } else if (r < rows) {
            if (nsplit == 1) {
                store4<kBf16>(out_at, 0, make_float4(o.x / ml.y, o.y / ml.y, o.z / ml.y, o.w / ml.y));
                if (lse_at) *lse_at = (ml.x + log2f(ml.y)) * 0.6931471805599453f;
            } else {
                const long long e = (long long)sp.part_base + (row_of(r) - (long long)sp.q_row0 * p.hq) * nsplit + split;
                *(float4*)(p.part_o + e * D + c) = o;
                if (c == 0) p.part_ml[e] = ml;
            }
        }
    }
    if (in_cluster) {
        cluster_sync();
        // groups of four columns are dealt round-robin to the cluster's CTAs
        for (int i = out0; i < kR * kUnits; i += nsplit * kThreads) {   // (once)
            const int rl = i / kUnits, c = (i % kUnits) * 4;
            if (!out_at) continue;
            const uint32_t ml_addr = smem_u32(&sm.ml[rl]), o_addr = smem_u32(&sm.o[rl][c]);
            float2 ml[16];
            float4 x[16];
#pragma unroll
            for (int k = 0; k < 16; ++k)
                if (k < nsplit) { ml[k] = ld_cluster_f2(cluster_map(ml_addr, k)); x[k] = ld_cluster_f4(cluster_map(o_addr, k)); }
            float m = -INFINITY, l = 0.f;
#pragma unroll
            for (int k = 0; k < 16; ++k) if (k < nsplit) m = fmaxf(m, ml[k].x);
            float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int k = 0; k < 16; ++k)
                if (k < nsplit && ml[k].x != -INFINITY) {
                    const float w = exp2f(ml[k].x - m);
                    l += ml[k].y * w;
                    o.x += x[k].x * w; o.y += x[k].y * w; o.z += x[k].z * w; o.w += x[k].w * w;
                }
            store4<kBf16>(out_at, 0, make_float4(o.x / l, o.y / l, o.z / l, o.w / l));
            if (lse_at) *lse_at = (m + log2f(l)) * 0.6931471805599453f;
        }
        cluster_sync();   // no CTA leaves while its rows may still be read
    }
}

namespace {
template <int D, bool kBf16>
cudaError_t configure() {
    static bool done[64] = {false};   // the attributes are per device
    int device = 0;
    if (cudaGetDevice(&device) != cudaSuccess || device < 0 || device >= 64) return cudaErrorInvalidDevice;
    if (done[device]) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(attn_simt_kernel<D, kBf16>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SimtSmem<D>));
    if (e == cudaSuccess) e = cudaFuncSetAttribute(attn_simt_kernel<D, kBf16>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);   // clusters of up to 16
    done[device] = e == cudaSuccess;
    return e;
}
template <int D, bool kBf16>
cudaError_t launch(const AttnParams& p, cudaStream_t stream) {
    cudaError_t e = configure<D, kBf16>();
    if (e != cudaSuccess) return e;
    if (p.cluster_size > 1)
        return launch_chained_cluster(attn_simt_kernel<D, kBf16>, dim3(p.num_items), dim3(kThreads), sizeof(SimtSmem<D>), (unsigned)p.cluster_size, stream, p);
    return launch_chained(attn_simt_kernel<D, kBf16>, dim3(p.num_items), dim3(kThreads), sizeof(SimtSmem<D>), stream, p);
}
}  // namespace

cudaError_t launch_attn_simt(const AttnParams& p, int dtype, cudaStream_t stream) {
    if (p.num_items == 0) return cudaSuccess;
    if (dtype == AGX_F32 && p.head_dim == 64) return launch<64, false>(p, stream);
    if (dtype == AGX_F32 && p.head_dim == 128) return launch<128, false>(p, stream);
    if (dtype == AGX_BF16 && p.head_dim == 64) return launch<64, true>(p, stream);
    return cudaErrorInvalidValue;
}

}  // namespace agx
