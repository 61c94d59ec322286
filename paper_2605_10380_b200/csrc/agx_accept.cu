// Greedy acceptance: per-row vocabulary argmax fused with the draft comparison and the length
// commit, in ONE launch (Sec. 2.3, speculative decoding: the first mismatching draft and all
// drafts after it are discarded; the accepted drafts plus the target's own token continue).
//
// HBM-bound scan: rows * vocab * elem bytes, read once with 128-bit loads.  Grid = (chunks, rows);
// every block reduces its slice of one row to a packed 64-bit (ordered value, inverted index) key
// whose unsigned maximum is "largest value, lowest index on ties", and folds it into the row's key
// with one 64-bit atomic maximum (order-independent, so the result is bit-reproducible).  The last
// block to finish (ticket counter) reads the row keys back, leaves them and the ticket at zero for
// the next launch, compares drafts and writes the results, so no second launch and no host round
// trip is needed.
#include <algorithm>

#include "agx_internal.cuh"
#include "agx_sm100.cuh"

namespace agx {

// Monotone map float -> uint32 with: NaN -> 0 (below everything), -0 == +0.
__device__ __forceinline__ unsigned int ordered_key(float x) {
    if (x != x) return 0u;
    unsigned int b = __float_as_uint(x);
    if (b == 0x80000000u) b = 0u;
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}

__device__ __forceinline__ unsigned long long pack_key(unsigned int key, unsigned int idx) {
    return ((unsigned long long)key << 32) | (unsigned long long)(0xFFFFFFFFu - idx);
}

__device__ __forceinline__ float bf16_bits_to_float(unsigned int lo16) { return __uint_as_float(lo16 << 16); }

// Running maximum of one thread over 16-byte vectors met in ascending order.  A vector costs a packed maximum of its elements and one
// comparison (NaN operands lose, and a NaN result compares false); only a vector that beats the maximum is kept, and which of its
// elements it was is worked out once at the end.  Ordering every element by an integer key instead took eight instructions each and
// bounded the scan of many rows (32 / 256 rows of 128256 bf16: 7.2 / 27.2 us before, 6.1 / 19.5 now; 8 rows 5.2).
template <bool kBf16>
struct VecMax {
    float best = -INFINITY;
    unsigned int base = 0;
    uint4 vec = make_uint4(0u, 0u, 0u, 0u);
    bool any = false;
    __device__ __forceinline__ void take(const uint4 a, unsigned int at) {
        float m;
        if (kBf16) {
            const __nv_bfloat162 x = __hmax2(__hmax2(*(const __nv_bfloat162*)&a.x, *(const __nv_bfloat162*)&a.y),
                                             __hmax2(*(const __nv_bfloat162*)&a.z, *(const __nv_bfloat162*)&a.w));
            m = fmaxf(__low2float(x), __high2float(x));
        } else {
            m = fmaxf(fmaxf(__uint_as_float(a.x), __uint_as_float(a.y)), fmaxf(__uint_as_float(a.z), __uint_as_float(a.w)));
        }
        if (m > best || (!any && m == m)) { best = m; base = at; vec = a; any = true; }
    }
    // Elements [at, end) at the end of a row whose length is not a multiple of the vector's: the rest counts as NaN.
    __device__ __forceinline__ void take_partial(const void* row, unsigned int at, unsigned int end) {
        unsigned int w[4] = {~0u, ~0u, ~0u, ~0u};   // (all ones is a NaN in both formats)
        for (unsigned int e = at; e < end; ++e) {
            if (kBf16) {
                const unsigned int x = ((const unsigned short*)row)[e], k = e - at;
                w[k >> 1] = (k & 1) ? (w[k >> 1] & 0xFFFFu) | (x << 16) : (w[k >> 1] & 0xFFFF0000u) | x;
            } else {
                w[e - at] = ((const unsigned int*)row)[e];
            }
        }
        take(make_uint4(w[0], w[1], w[2], w[3]), at);
    }
    // packed key of the maximum (lowest index on ties); 0 = no number seen
    __device__ __forceinline__ unsigned long long key() const {
        if (!any) return 0ull;
        const unsigned int w[4] = {vec.x, vec.y, vec.z, vec.w};
        unsigned int idx = base;
        bool found = false;
#pragma unroll
        for (int i = 0; i < (kBf16 ? 8 : 4); ++i) {
            const float x = kBf16 ? bf16_bits_to_float((i & 1) ? w[i >> 1] >> 16 : w[i >> 1] & 0xFFFFu) : __uint_as_float(w[i & 3]);
            if (!found && x == best) { idx = base + i; found = true; }
        }
        return pack_key(ordered_key(best), idx);
    }
};

__device__ __forceinline__ unsigned long long warp_max(unsigned long long v) {
    const unsigned int hi = (unsigned int)(v >> 32), top = __reduce_max_sync(0xFFFFFFFFu, hi);
    return ((unsigned long long)top << 32) | __reduce_max_sync(0xFFFFFFFFu, hi == top ? (unsigned int)v : 0u);
}

// What the comparison of a sequence needs besides the winners, fetched by a warp ahead of them: its rows, and of its drafts the first 32.
struct SeqHead {
    int r0 = 0, k = 0, len = 0, draft = 0;
    __device__ __forceinline__ void load_rows(int s, int B, const int* cu_q, const int* seq_lens) {
        if (s >= B) return;
        r0 = cu_q[s];
        k = cu_q[s + 1] - r0 - 1;
        if (seq_lens) len = seq_lens[s];
    }
    __device__ __forceinline__ void load_drafts(int s, int B, const int* drafts) {
        const int lane = threadIdx.x & 31;
        if (s < B && lane < k) draft = drafts[r0 - s + lane];
    }
};
// One warp compares a sequence's drafts, 32 at a time, with the winners of the rows before them and commits the result.
template <typename Token>
__device__ __forceinline__ void commit_sequence(int s, const SeqHead& h, const int* drafts, Token token, int* accept_len, int* next_token,
                                                int* seq_lens) {
    const int lane = threadIdx.x & 31;
    int a = 0;
    while (a < h.k) {
        const bool match = (a + lane < h.k) ? ((a == 0 ? h.draft : drafts[h.r0 - s + a + lane]) == token(h.r0 + a + lane)) : false;
        const unsigned int m = __ballot_sync(0xFFFFFFFFu, match);
        const int run = (m == 0xFFFFFFFFu) ? 32 : __ffs(~m) - 1;   // leading matches of this group of 32
        a += run;
        if (run < 32) break;
    }
    if (lane == 0) {
        accept_len[s] = a;
        next_token[s] = token(h.r0 + a);
        if (seq_lens) seq_lens[s] = h.len + a + 1;
    }
}

constexpr int kTokSmem = 2048;               // winners of up to this many rows stay in shared memory for the draft comparison

template <bool kBf16, bool kVec>
__global__ void __launch_bounds__(256, kAcceptCtas)
accept_kernel(const void* __restrict__ logits, long long row_stride, int vocab, int chunk_elems,
              const int* __restrict__ drafts, const int* __restrict__ cu_q, int B, int total_q,
              int* __restrict__ accept_len, int* __restrict__ next_token, int* __restrict__ argmax,
              int* __restrict__ seq_lens, unsigned long long* row_keys, int* tokens_global, unsigned int* ticket) {
    constexpr int kVecElems = kBf16 ? 8 : 4;
    pdl_launch_dependents();
    const int row = blockIdx.y;
    const int chunk = blockIdx.x;
    const char* row_ptr = (const char*)logits + (size_t)row * row_stride * (kBf16 ? 2 : 4);
    unsigned long long* row_key = row_keys + row;
    hold(row_ptr); hold(row_key); hold(cu_q); hold(drafts); hold(seq_lens); hold(ticket); hold(vocab); hold(B);
    asm volatile("" ::"l"(accept_len), "l"(next_token), "l"(argmax), "r"(total_q), "l"(tokens_global));   // (in the constant cache for the last block)
    pdl_wait();
    const unsigned int begin = (unsigned int)chunk * (unsigned int)chunk_elems;
    const unsigned int end = min((unsigned int)vocab, begin + (unsigned int)chunk_elems);

    // (every block fetches what only the last one will use: its two trips to memory lie under the scan and the ticket; 8 rows of 128256 bf16 in
    // a graph 4.58 -> 4.32 us, 4 rows of 1024 fp32 3.60 -> 3.41)
    const int warp = threadIdx.x >> 5;
    SeqHead head;
    head.load_rows(warp, B, cu_q, seq_lens);
    unsigned long long best = 0ull;  // "no element": loses to every real element
    if (kVec) {
        VecMax<kBf16> vm;
        // four independent 16-byte loads in flight per thread and trip, also in the last one
        const unsigned int stride = 256 * kVecElems;
        for (unsigned int i = begin + threadIdx.x * kVecElems; i < end; i += 4 * stride) {
            uint4 a[4];
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (i + u * stride + kVecElems <= end) a[u] = __ldg((const uint4*)(row_ptr + (size_t)(i + u * stride) * (kBf16 ? 2 : 4)));
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const unsigned int at = i + u * stride;
                if (at + kVecElems <= end) vm.take(a[u], at);
                else if (at < end) vm.take_partial(row_ptr, at, end);
            }
        }
        best = vm.key();
    } else {
        for (unsigned int e = begin + threadIdx.x; e < end; e += 256) {
            float x;
            if (kBf16) x = bf16_bits_to_float(((const unsigned short*)row_ptr)[e]);
            else x = ((const float*)row_ptr)[e];
            const unsigned long long k = pack_key(ordered_key(x), e);
            best = k > best ? k : best;
        }
    }

    best = warp_max(best);
    __shared__ unsigned long long warp_best[8];
    __shared__ bool is_last;
    if ((threadIdx.x & 31) == 0) warp_best[warp] = best;
    head.load_drafts(warp, B, drafts);
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long b = warp_best[0];
#pragma unroll
        for (int w = 1; w < 8; ++w) b = warp_best[w] > b ? warp_best[w] : b;
        if (b) atomicMax(row_key, b);   // (0: no number in this chunk)
        __threadfence();
        const unsigned int total = gridDim.x * gridDim.y;
        const unsigned int t = atomicAdd(ticket, 1u);
        is_last = (t == total - 1);
        if (is_last) *ticket = 0u;  // leave the counter ready for the next launch
    }
    __syncthreads();
    if (!is_last) return;
    __threadfence();

    // the rows' winners: read the keys back past the L1, zero them for the next launch; up to kTokSmem winners stay in
    // shared memory for the draft comparison, more go through global memory
    __shared__ int tokens_smem[kTokSmem];
    const bool in_smem = total_q <= kTokSmem;
    int* tokens = in_smem ? tokens_smem : tokens_global;
    for (int r = threadIdx.x; r < total_q; r += 256) {
        const unsigned long long b = __ldcg(row_keys + r);
        row_keys[r] = 0ull;
        const int t = b ? (int)(0xFFFFFFFFu - (unsigned int)(b & 0xFFFFFFFFull)) : 0;   // (a row of NaN only: 0)
        tokens[r] = t;
        if (argmax) argmax[r] = t;
    }
    __syncthreads();
    for (int s = warp; s < B; s += 8) {
        if (s != warp) { head.load_rows(s, B, cu_q, seq_lens); head.load_drafts(s, B, drafts); }
        commit_sequence(s, head, drafts, [&](int r) { return in_smem ? tokens[r] : __ldcg(tokens + r); }, accept_len, next_token, seq_lens);
    }
}

// The same for few, short rows, where the scan is nothing and the way of the winners from block to block is the time: one cluster of eight
// CTAs, whose keys meet through distributed shared memory instead of atomics, a fence, a ticket and a read back.  A row's elements are dealt to
// 8 / rows CTAs.  (In a graph, us a call, one launch with atomics / this: 4 x 1024 fp32 3.41 / 2.74, 8 x 4096 3.65 / 3.58, 8 x 8192 3.60 / 4.43,
// 1 x 32000 bf16 3.70 / 3.22, 2 x 128256 3.93 / 6.57: from 32 KB a CTA on, its SM's share of the bytes is the time.)
constexpr int kClusterCtas = 8;
constexpr int kClusterBytes = 16384;   // of a row per CTA, at most
template <bool kBf16>
__global__ void __cluster_dims__(kClusterCtas, 1, 1) __launch_bounds__(256)
accept_cluster_kernel(const void* __restrict__ logits, long long row_stride, int vocab, int chunks, int chunk_elems, const int* __restrict__ drafts,
                      const int* __restrict__ cu_q, int B, int total_q, int* __restrict__ accept_len, int* __restrict__ next_token,
                      int* __restrict__ argmax, int* __restrict__ seq_lens) {
    constexpr int kVecElems = kBf16 ? 8 : 4;
    __shared__ unsigned long long warp_best[8];
    __shared__ int tokens[kClusterCtas];
    pdl_launch_dependents();
    const int rank = blockIdx.x, row = rank / chunks, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned int begin = (unsigned int)(rank - row * chunks) * (unsigned int)chunk_elems, end = min((unsigned int)vocab, begin + (unsigned int)chunk_elems);
    const char* row_ptr = (const char*)logits + (size_t)row * row_stride * (kBf16 ? 2 : 4);
    hold(row_ptr); hold(cu_q); hold(drafts); hold(seq_lens); hold(accept_len); hold(next_token); hold(argmax); hold(B); hold(total_q);
    pdl_wait();
    SeqHead head;
    if (rank == 0) head.load_rows(warp, B, cu_q, seq_lens);
    VecMax<kBf16> vm;
    if (row < total_q) {
        for (unsigned int i = begin + threadIdx.x * kVecElems; i < end; i += 256 * kVecElems) {
            if (i + kVecElems <= end) vm.take(__ldg((const uint4*)(row_ptr + (size_t)i * (kBf16 ? 2 : 4))), i);
            else vm.take_partial(row_ptr, i, end);
        }
    }
    const unsigned long long best = warp_max(vm.key());
    if (lane == 0) warp_best[warp] = best;
    if (rank == 0) head.load_drafts(warp, B, drafts);
    cluster_sync();
    if (rank == 0) {
        if (warp < total_q) {   // warp r: the winner of row r, from the 8 * chunks keys of its CTAs
            unsigned long long b = 0ull;
            for (int i = lane; i < 8 * chunks; i += 32) {
                const uint32_t at = cluster_map(smem_u32(warp_best + (i & 7)), (uint32_t)(warp * chunks + (i >> 3)));
                unsigned long long x;
                asm volatile("ld.shared::cluster.u64 %0, [%1];\n" : "=l"(x) : "r"(at) : "memory");
                b = x > b ? x : b;
            }
            b = warp_max(b);
            const int t = b ? (int)(0xFFFFFFFFu - (unsigned int)(b & 0xFFFFFFFFull)) : 0;   // (a row of NaN only: 0)
            if (lane == 0) { tokens[warp] = t; if (argmax) argmax[warp] = t; }
        }
        __syncthreads();
        if (warp < B) commit_sequence(warp, head, drafts, [&](int r) { return tokens[r]; }, accept_len, next_token, seq_lens);
    }
    cluster_sync();   // no CTA leaves while its keys may still be read
}

cudaError_t launch_accept(const void* logits, int logits_dtype, long long row_stride, int vocab, const int* drafts,
                          const int* cu_q, int B, int total_q, int* accept_len, int* next_token, int* argmax,
                          int* seq_lens, unsigned long long* row_keys, int* tokens_global, int sm_count, unsigned int* ticket,
                          cudaStream_t stream) {
    const bool bf16 = logits_dtype == AGX_BF16;
    const int esz = bf16 ? 2 : 4;
    const int vec_elems = 16 / esz;
    const bool vec = ((uintptr_t)logits % 16 == 0) && ((row_stride * esz) % 16 == 0);
    // up to 8 rows whose CTAs have at most four vectors a thread each
    const int cluster_chunks = total_q <= kClusterCtas ? kClusterCtas / total_q : 0;
    if (vec && cluster_chunks && (long long)vocab * esz <= (long long)cluster_chunks * kClusterBytes) {
        int elems = (vocab + cluster_chunks - 1) / cluster_chunks;
        elems = (elems + vec_elems - 1) / vec_elems * vec_elems;
        return launch_chained(bf16 ? accept_cluster_kernel<true> : accept_cluster_kernel<false>, dim3(kClusterCtas), dim3(256), 0, stream, logits, row_stride, vocab,
                              cluster_chunks, elems, drafts, cu_q, B, total_q, accept_len, next_token, argmax, seq_lens);
    }
    const int chunks = accept_chunks(sm_count, total_q, vocab, esz, vec);
    int chunk_elems = (vocab + chunks - 1) / chunks;
    chunk_elems = (chunk_elems + vec_elems - 1) / vec_elems * vec_elems;  // chunk starts stay 16-byte aligned
    dim3 grid((vocab + chunk_elems - 1) / chunk_elems, total_q);
    cudaError_t err = cudaSuccess;
#define AGX_LAUNCH_ACCEPT(BF, VEC)                                                                              \
    err = launch_chained(accept_kernel<BF, VEC>, grid, dim3(256), 0, stream, logits, row_stride, vocab, chunk_elems,  \
                         drafts, cu_q, B, total_q, accept_len, next_token, argmax, seq_lens, row_keys, tokens_global, \
                         ticket)
    if (bf16) { if (vec) AGX_LAUNCH_ACCEPT(true, true); else AGX_LAUNCH_ACCEPT(true, false); }
    else      { if (vec) AGX_LAUNCH_ACCEPT(false, true); else AGX_LAUNCH_ACCEPT(false, false); }
#undef AGX_LAUNCH_ACCEPT
    return err;
}

}  // namespace agx

// --------------------------------------------------------------------------------------------
// Allocation-free variant of the accept step.
//
// Some callers cannot allocate device memory at the point where they verify drafts: code running
// inside a pre-sized serving arena or an embedded runtime whose memory is fixed at start-up, and
// code that must not disturb a caching allocator owned by someone else (a cudaMalloc there can
// synchronise the device or fail outright).  agx_accept_greedy needs a caller-provided workspace
// and a handle whose creation allocates; the entry point below needs neither.  Its scratch (the
// rows' argmax keys and the ticket counter) lives in a fixed array that is part of the loaded
// module, so every GPU that loads the library carries these 16 KB until the process exits.
#include <atomic>
#include <mutex>

namespace agx {
namespace {
constexpr int kStaticMaxRows = 2048;    // logits rows per call (their winners fit the kernel's shared memory)
constexpr int kStaticDevices = 64;
// layout: [0, 256) ticket counter | one 64-bit key per row
constexpr size_t kStaticBytes = 256 + (size_t)kStaticMaxRows * 8;
static_assert(kStaticMaxRows <= kTokSmem, "the allocation-free variant has no global buffer for the rows' winners");
static __device__ __align__(256) unsigned char g_accept_scratch[kStaticBytes];

struct StaticDeviceState {
    std::atomic<void*> scratch{nullptr};  // device address of g_accept_scratch on that device (NULL until resolved)
    int sm_count = 0;                     // written before `scratch` is published
};
StaticDeviceState g_static_state[kStaticDevices];
std::mutex g_static_init;                 // serialises the one-time set-up (several host threads may make the first call)

inline bool aligned_to(const void* p, size_t a) { return ((uintptr_t)p % a) == 0; }
}  // namespace
}  // namespace agx

extern "C" AGX_API agx_status agx_accept_greedy_static(const void* logits, int32_t logits_dtype, int64_t row_stride,
                                                       int32_t vocab, const int32_t* drafts, const int32_t* cu_q,
                                                       int32_t B, int32_t total_q, int32_t* accept_len,
                                                       int32_t* next_token, int32_t* argmax, int32_t* seq_lens,
                                                       void* stream) {
    using namespace agx;
    if (B < 0 || total_q < 0) return AGX_E_INVAL;
    if (B == 0) return AGX_OK;
    if (total_q < B) return AGX_E_INVAL;
    if (logits_dtype != AGX_BF16 && logits_dtype != AGX_F32) return AGX_E_UNSUPPORTED;
    if (vocab < 1 || row_stride < vocab) return AGX_E_RANGE;
    if (!logits || !cu_q || !accept_len || !next_token || (!drafts && total_q > B)) return AGX_E_INVAL;
    // the same alignment rules as the workspace variant: a misaligned pointer is an argument error, not a device fault
    if (!aligned_to(logits, logits_dtype == AGX_BF16 ? 2 : 4) || !aligned_to(drafts, 4) || !aligned_to(cu_q, 4) ||
        !aligned_to(accept_len, 4) || !aligned_to(next_token, 4) || !aligned_to(argmax, 4) || !aligned_to(seq_lens, 4))
        return AGX_E_INVAL;
    if (total_q > kStaticMaxRows) return AGX_E_RANGE;  // beyond the fixed scratch: use agx_accept_greedy

    int device = -1;
    if (cudaGetDevice(&device) != cudaSuccess || device < 0 || device >= kStaticDevices) return AGX_E_CUDA;
    StaticDeviceState& st = g_static_state[device];
    void* scratch = st.scratch.load(std::memory_order_acquire);
    if (!scratch) {
        // One-time set-up for this device, with it current.  In host code the array's name is only a
        // stand-in for the symbol; the address kernels can use has to be asked for.
        std::lock_guard<std::mutex> lock(g_static_init);
        scratch = st.scratch.load(std::memory_order_relaxed);
        if (!scratch) {
            void* ptr = nullptr;
            if (cudaGetSymbolAddress(&ptr, g_accept_scratch) != cudaSuccess || !ptr) return AGX_E_CUDA;
            int sms = 0;
            if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess || sms < 1) return AGX_E_CUDA;
            st.sm_count = sms;
            st.scratch.store(ptr, std::memory_order_release);
            scratch = ptr;
        }
    }
    unsigned char* base = (unsigned char*)scratch;
    // the array keeps whatever the previous call left: the ticket counter and the rows' keys must start at zero (the
    // kernel leaves them at zero itself; the clear makes the call independent of how an earlier one ended)
    if (cudaMemsetAsync(base, 0, 256 + (size_t)total_q * 8, (cudaStream_t)stream) != cudaSuccess) return AGX_E_CUDA;
    cudaError_t e = launch_accept(logits, logits_dtype, row_stride, vocab, drafts, cu_q, B, total_q, accept_len,
                                  next_token, argmax, seq_lens, (unsigned long long*)(base + 256), nullptr, st.sm_count,
                                  (unsigned int*)base, (cudaStream_t)stream);
    return e == cudaSuccess ? AGX_OK : AGX_E_CUDA;
}
