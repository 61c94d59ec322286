// PTX wrappers shared by the sm_100a kernels: mbarrier (with bounded waits), TMA tile loads, fast exp2.
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include <stdint.h>

#include "agx.h"
#include "agx_internal.cuh"

namespace agx {

namespace {

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {   // (no arrival)
    asm volatile("mbarrier.expect_tx.relaxed.cta.shared::cta.b64 [%0], %1;\n" ::"r"(bar), "r"(bytes) : "memory");
}
// kSuspendNs > 0: how long the thread may be suspended before it has to look again (0: the hardware's own limit).  For waits of a microsecond a long
// suspension is over sooner than a loop of short ones: decode over 4096 tokens, 32 layers of the swapped-operand kernel, 209.3 -> 205.5 us; the
// tensor-core kernel, whose waits are many and short, loses 0.5 % by it.
template <unsigned kSuspendNs = 0>
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    if constexpr (kSuspendNs > 0) {
        asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\nselp.u32 %0, 1, 0, p;\n}\n"
                     : "=r"(ok) : "r"(bar), "r"(parity), "r"(kSuspendNs) : "memory");
        return ok != 0;
    }
    asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
                 : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
// Bounded wait.  Returns false (and raises the CTA's abort flag) when the limit is hit or another
// role already gave up.
template <unsigned kSuspendNs = 0>
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag, int* status,
                                          long long limit_cycles) {
    constexpr int kLookEvery = kSuspendNs > 0 ? 4 : 64;   // waits between two looks at the clock
    if (mbar_try_wait<kSuspendNs>(bar, parity)) return true;
    const long long t0 = clock64();
    int spins = 0;
    for (;;) {
        if (mbar_try_wait<kSuspendNs>(bar, parity)) return true;
        if ((++spins & (kLookEvery - 1)) == 0) {
            if (*abort_flag) return false;
            if (clock64() - t0 > limit_cycles) {
                *abort_flag = 1;
                if (status) atomicOr(status, AGX_DEV_WAIT_TIMEOUT);
                return false;
            }
        }
    }
}

// Wait of the copy-issuing lane for copies it has armed itself, when the CTA winds down: bounded by the clock only.
// The abort flag is ignored on purpose, since the shared memory the copies land in must stay allocated until they have.
__device__ __forceinline__ bool mbar_drain(uint32_t bar, uint32_t parity, long long limit_cycles) {
    const long long t0 = clock64();
    while (!mbar_try_wait(bar, parity))
        if (clock64() - t0 > limit_cycles) return false;
    return true;
}

// One page of one KV head (16 tokens x 256 B, 4 KB in HBM and in shared memory) through the pool's tensor map; `group` = row / 8 of
// the page's first row.  Layout in shared memory: [row group of 8][half of 64 dims][8 rows][128 B], 128-byte swizzled.
__device__ __forceinline__ void tma_load_page(uint32_t dst, const CUtensorMap* map, int group, uint32_t bar) {
    asm volatile("cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %2, %2, %3}], [%4];\n"
                 ::"r"(dst), "l"(map), "r"(0), "r"(group), "r"(bar) : "memory");
}

// Eight or 128 rows of one KV head of the block's own K or V ([total_q][hkv][128]) from `row` on (see RowsMaps), in the layout of
// row groups.  Past the end the 8-row copy brings zeros; the 128 rows must all exist.
__device__ __forceinline__ void tma_load_rows8(uint32_t dst, const CUtensorMap* map, int row, int head, uint32_t bar) {
    asm volatile("cp.async.bulk.tensor.5d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %2, %2, %4}], [%5];\n"
                 ::"r"(dst), "l"(map), "r"(0), "r"(row), "r"(head), "r"(bar) : "memory");
}
__device__ __forceinline__ void tma_load_rows128(uint32_t dst, const CUtensorMap* map, int row, int head, uint32_t bar) {
    tma_load_rows8(dst, map, row, head, bar);   // (the map's box is 16 row groups)
}

// Eight rows of one KV head, as they lie in a K or V tile, to half a page of the pool (RowsMaps::k_pool8 / v_pool8); `group` as above.
__device__ __forceinline__ void tma_store_group(const CUtensorMap* map, int group, uint32_t src) {
    asm volatile("cp.async.bulk.tensor.4d.global.shared::cta.bulk_group [%0, {%1, %1, %1, %2}], [%3];\n" ::"l"(map), "r"(0), "r"(group), "r"(src) : "memory");
}

// One half (64 dims) of Q rows of KV head g through RowsMaps::q_box (all heads of q_tokens tokens from `token` on) or q_row (head `hh` of the
// group, one token), one 128-byte line per row.  The 128-byte swizzle goes by the address in shared memory, so that a copy may start at any row
// of a tile.  Past the end zeros arrive.
__device__ __forceinline__ void tma_load_q(uint32_t dst, const CUtensorMap* map, int hh, int token, int half, int g, uint32_t bar) {
    asm volatile("cp.async.bulk.tensor.5d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5, %6}], [%7];\n"
                 ::"r"(dst), "l"(map), "r"(0), "r"(hh), "r"(token), "r"(half), "r"(g), "r"(bar) : "memory");
}

// One lane of a converged warp.  Unlike `lane == 0` this tells the compiler that a single thread takes the branch, so the
// instructions that want their operands in uniform registers (tcgen05.mma, TMA copies) are issued without a loop over lanes.
__device__ __forceinline__ bool elect_one() {
    uint32_t p;
    asm volatile("{\n.reg .pred p;\nelect.sync _|p, 0xFFFFFFFF;\nselp.u32 %0, 1, 0, p;\n}\n" : "=r"(p));
    return p != 0;
}

// Holds a value in a register from here on.  Kernel parameters are read through the constant cache where they are used, and the cache is cold at the
// start of a launch: what is needed behind the dependency wait is worked out and held before it.  (A decode layer over 4096 tokens, launched as
// a stream of kernels: 7.7 -> 7.25 us with it in the merge kernel, whose addresses come from six parameters, 6.8 with the attention kernel's; in
// a graph, where the cache is warm, 6.15.  The warp-MMA and the tensor-core kernel gain nothing: the addresses are not on their critical path.)
__device__ __forceinline__ void hold(int& x) { asm volatile("" : "+r"(x)); }
__device__ __forceinline__ void hold(unsigned& x) { asm volatile("" : "+r"(x)); }
__device__ __forceinline__ void hold(float& x) { asm volatile("" : "+f"(x)); }
__device__ __forceinline__ void hold(long long& x) { asm volatile("" : "+l"(x)); }
template <typename T>
__device__ __forceinline__ void hold(T*& x) { asm volatile("" : "+l"(x)); }
template <typename T>
__device__ __forceinline__ void hold(T* __restrict__& x) { asm volatile("" : "+l"(x)); }

// Programmatic dependent launch: a kernel lets the next launch in the stream start early (its CTAs then run
// their set-up and block in pdl_wait), and itself waits, before it touches global memory, until the launch
// before it has completed and its writes are visible.  Both are no-ops for launches without the attribute.
__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }

// On its way to L2 before the dependency wait: a hint that moves no data to the SM, so that it may run ahead of the launch that writes the line.
__device__ __forceinline__ void prefetch_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];\n" ::"l"(p) : "memory"); }

// The sequence plan of a work item.
__device__ __forceinline__ int find_seq(const AttnParams& p, int item) {
    int s = 0;
#pragma unroll 1
    for (int i = 1; i < p.num_seqs; ++i)
        if (p.seq[i].item0 <= item) s = i;
    return s;
}

// ---- tcgen05: descriptors, MMA, TMEM
// shared-memory matrix descriptor, SWIZZLE_128B, descriptor version 1
__device__ __forceinline__ uint64_t make_desc(uint32_t saddr, uint32_t lbo_bytes, uint32_t sbo_bytes) {
    return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)(lbo_bytes >> 4) << 16) | ((uint64_t)(sbo_bytes >> 4) << 32) |
           (1ull << 46) | (2ull << 61);
}

__device__ __forceinline__ void umma_ss(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t acc) {
    asm volatile("{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\ntcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n"
                 ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(acc) : "memory");
}
__device__ __forceinline__ void umma_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc, uint32_t acc) {
    asm volatile("{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\ntcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}\n"
                 ::"r"(d_tmem), "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(acc) : "memory");
}
__device__ __forceinline__ void umma_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;\n" ::: "memory"); }

__device__ __forceinline__ void tmem_ld_x32(uint32_t taddr, uint32_t* r) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
                 : "r"(taddr));
}
// N = 2, 4, 8, 16 or 32 columns from taddr on
template <int N>
__device__ __forceinline__ void tmem_ld(uint32_t taddr, uint32_t* r) {
    if constexpr (N == 2) {
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0, %1}, [%2];\n" : "=r"(r[0]), "=r"(r[1]) : "r"(taddr));
    } else if constexpr (N == 4) {
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];\n" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(taddr));
    } else if constexpr (N == 8) {
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];\n"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]) : "r"(taddr));
    } else if constexpr (N == 16) {
        tmem_ld<8>(taddr, r);
        tmem_ld<8>(taddr + 8, r + 8);
    } else {
        tmem_ld_x32(taddr, r);
    }
}
__device__ __forceinline__ uint32_t pack_f16(float lo, float hi) {
    uint32_t r;
    asm("cvt.rn.f16x2.f32 %0, %1, %2;\n" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}

// ---- thread-block clusters: barrier over all threads of all CTAs, and loads from a peer CTA's shared memory
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}
__device__ __forceinline__ uint32_t cluster_map(uint32_t smem_addr, uint32_t cta_rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(r) : "r"(smem_addr), "r"(cta_rank));
    return r;
}
__device__ __forceinline__ float4 ld_cluster_f4(uint32_t addr) {
    float4 v;
    asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];\n" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ float2 ld_cluster_f2(uint32_t addr) {
    float2 v;
    asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];\n" : "=f"(v.x), "=f"(v.y) : "r"(addr) : "memory");
    return v;
}

// Maximum over the warp, in every lane, by one instruction (a NaN loses, as with fmaxf).  Five steps of shuffles and maxima in its place are a chain of
// some 130 clocks.
__device__ __forceinline__ float warp_max(float x) {
    float m;
    asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;\n" : "=f"(m) : "f"(x));
    return m;
}

// Partials in fp16.  A row divided by its own sum is of V's magnitude, which may be anything that bf16 holds.  One whose largest magnitude `top` is above fp16's
// range or below 2^-11 is stored divided by 2^fp16_exponent(top), to at most 2^15, with the sum's sign as the mark of it, and the merge multiplies it back;
// others are stored as they are.  So a value is rounded to 11 bits or to 2^-14 of the row's largest, whichever is more (2^-25, half of fp16's smallest step, is
// 2^-14 of 2^-11).  The kernels store every row as it is and look at it on the way; what does not fit is stored once more.
constexpr float kFp16Least = 0x1p-11f, kFp16Most = 65504.f;
__device__ __forceinline__ int fp16_exponent(float top) {   // (top finite; not below -110, so that 2^-e times any value is finite: fp16 holds 2^-126 times 2^110)
    return (top >= kFp16Least && top <= kFp16Most) || top == 0.f ? 0 : max((__float_as_int(top) >> 23) - 127 - 14, -110);
}
__device__ __forceinline__ float pow2(int e) { return __int_as_float((e + 127) << 23); }   // |e| <= 126
__device__ __forceinline__ float finite_abs(float x) { return fabsf(x) < INFINITY ? fabsf(x) : 0.f; }   // (infinities and NaN stay what they are and do not count)
__device__ __forceinline__ float max3_abs(float a, float b, float c) {
    float d;
    asm("max.abs.f32 %0, %1, %2, %3;\n" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;\n" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&v);
}

// Merge of the KV splits of one (sequence, KV head) = the CTAs of a cluster (rank = split), each holding n_rows un-normalised fp32 rows of O
// ([row][128]) and their (m, l) in shared memory.  Rows are dealt round-robin to the CTAs; one warp merges one row, lane k < splits
// holding split k's (m, l), every lane four columns of each split's O row (all loads in flight at once).
template <int kWarps>
__device__ __forceinline__ void merge_cluster_rows(const AttnParams& p, const SeqPlan& sp, const float* cl_o, const float2* cl_ml, int g, int split,
                                                   int row0, int n_rows) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, G = p.gqa;
    cluster_sync();   // every split's rows are in place
    const int cs = sp.nsplit;
    for (int r = split + warp * cs; r < n_rows; r += kWarps * cs) {
        float2 ml = make_float2(-INFINITY, 0.f);
        if (lane < cs) ml = ld_cluster_f2(cluster_map(smem_u32(cl_ml + r), lane));
        const float m_all = warp_max(ml.x);
        const float w = (ml.x == -INFINITY) ? 0.f : exp2f(ml.x - m_all);
        float l_all = ml.y * w;
#pragma unroll
        for (int d = 16; d >= 1; d >>= 1) l_all += __shfl_xor_sync(0xFFFFFFFFu, l_all, d);
        const uint32_t row_addr = smem_u32(cl_o + r * 128 + lane * 4);
        float4 v[16];
#pragma unroll
        for (int k = 0; k < 16; ++k)
            if (k < cs) v[k] = ld_cluster_f4(cluster_map(row_addr, k));
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            const float wk = __shfl_sync(0xFFFFFFFFu, w, k);
            if (k < cs && wk != 0.f) { acc.x += v[k].x * wk; acc.y += v[k].y * wk; acc.z += v[k].z * wk; acc.w += v[k].w * wk; }
        }
        const int i = (int)(((uint64_t)(uint32_t)(row0 + r) * p.row_div_magic) >> 32), h = g * G + (row0 + r) - i * G;
        const float inv = 1.f / l_all;
        uint2 packed;
        packed.x = pack_bf16(acc.x * inv, acc.y * inv);
        packed.y = pack_bf16(acc.z * inv, acc.w * inv);
        *(uint2*)((__nv_bfloat16*)p.out + ((long long)(sp.q_row0 + i) * p.hq + h) * 128 + lane * 4) = packed;
        if (p.lse && lane == 0) p.lse[(long long)(sp.q_row0 + i) * p.hq + h] = (m_all + log2f(l_all)) * 0.6931471805599453f;
    }
    cluster_sync();   // no CTA leaves while its rows may still be read
}

}  // namespace
}  // namespace agx
