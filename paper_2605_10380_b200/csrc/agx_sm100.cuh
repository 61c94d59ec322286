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
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
                 : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
// Bounded wait.  Returns false (and raises the CTA's abort flag) when the limit is hit or another
// role already gave up.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag, int* status,
                                          long long limit_cycles) {
    if (mbar_try_wait(bar, parity)) return true;
    const long long t0 = clock64();
    int spins = 0;
    for (;;) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((++spins & 63) == 0) {
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

// One lane of a converged warp.  Unlike `lane == 0` this tells the compiler that a single thread takes the branch, so the
// instructions that want their operands in uniform registers (tcgen05.mma, TMA copies) are issued without a loop over lanes.
__device__ __forceinline__ bool elect_one() {
    uint32_t p;
    asm volatile("{\n.reg .pred p;\nelect.sync _|p, 0xFFFFFFFF;\nselp.u32 %0, 1, 0, p;\n}\n" : "=r"(p));
    return p != 0;
}

// Programmatic dependent launch: a kernel lets the next launch in the stream start early (its CTAs then run
// their set-up and block in pdl_wait), and itself waits, before it touches global memory, until the launch
// before it has completed and its writes are visible.  Both are no-ops for launches without the attribute.
__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }

// Fused KV append (bf16, d = 128): the block's rows [i_lo, i_hi) of KV head g go into the sequence's pages (Sec. 2.3: the block's KV
// joins the cache).  Nothing in the same launch reads them there: the attention CTAs take the block's own rows from k_new / v_new,
// so there is nothing to wait for.
struct BlockRows {
    static constexpr int kBatch = 4;   // 16-byte units in flight per thread: idx0, idx0 + nthreads, ...
    uint4 v[kBatch];
    int id[kBatch];
    __device__ __forceinline__ void load(const AttnParams& p, const SeqPlan& sp, int g, int i_lo, int i_hi, int idx0, int nthreads) {
        const int* pt_row = p.page_table + (long long)sp.seq_index * p.pt_stride;
        const int units = (i_hi - i_lo) * 32;
#pragma unroll
        for (int j = 0; j < kBatch; ++j) {
            const int idx = idx0 + j * nthreads, i = i_lo + (idx >> 5), slot = (sp.prefix_len + i) >> 4;
            id[j] = -2;
            if (idx < units) {
                id[j] = slot < p.pt_stride ? __ldg(pt_row + slot) : -1;
                v[j] = __ldg((const uint4*)((const unsigned char*)((idx & 16) ? p.v_new : p.k_new) + (((long long)(sp.q_row0 + i) * p.hkv + g) * 256 + (idx & 15) * 16)));
            }
        }
    }
    __device__ __forceinline__ void store(const AttnParams& p, const SeqPlan& sp, int g, int i_lo, int i_hi, int idx0, int nthreads) {
#pragma unroll
        for (int j = 0; j < kBatch; ++j) {
            const int idx = idx0 + j * nthreads, tok = sp.prefix_len + i_lo + (idx >> 5);
            if (id[j] >= 0 && id[j] < p.num_pages)
                *(uint4*)((unsigned char*)((idx & 16) ? p.v_pool : p.k_pool) + ((((long long)id[j] * p.hkv + g) * kPage + (tok & 15)) * 256 + (idx & 15) * 16)) = v[j];
            else if (id[j] != -2) atomicOr(p.status, AGX_DEV_BAD_PAGE);
        }
    }
};

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

__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;\n" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&v);
}

}  // namespace
}  // namespace agx
