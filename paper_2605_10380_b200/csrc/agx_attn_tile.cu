// Large-q attention over a paged KV cache: the uncached suffix of a prompt attending over its cached
// prefix plus itself (Sec. 2.3, prefix caching; Sec. 4.2 makes the suffix a few hundred tokens over a
// prefix of thousands).  Here Q K^T and P V are dense contractions, so they run on the 5th-generation
// tensor cores: tcgen05.mma issued by one thread, operands staged in shared memory by TMA,
// accumulators in tensor memory (TMEM).
//
// What bounds it: the tensor pipe and the exponentials (2048 cycles each per KV tile), the instruction issue of the single-thread
// roles, whose warps share their schedulers with two softmax warps each (a KV tile took the TMA producer 3000 cycles while it
// divided by run-time stage counts and shuffled page ids; it is now two 16-byte loads and eight copies), and on long runs the power cap.
//
// Work item = (sequence, KV head g, chunk of 256 query rows, KV split).  The q * G rows of one KV
// head (row r = i * G + h % G) are cut into two 128-row tiles A and B that share every K/V tile.
// CTA = 12 warps:
//   warp 0      TMA producer (one elected thread): per 128-token tile, 8 pages x one 4 KB box for K and
//               for V (SWIZZLE_128B), page ids read through the page table.  One box per page instead of two
//               of 64 dims, issued without a loop over lanes: 4 x 32768 verify 107 -> 100 us, 16 x 8192 verify
//               116 -> 92 us, 16 decode blocks over 2k-14k tokens 83 -> 76 us.
//   warps 1, 2  MMA issuers, one elected thread each (elect.sync: behind `lane == 0` the issue of eight tcgen05.mma took up to
//               570 cycles), warp 1 also TMEM owner.  Warp 1 issues S = Q K^T, warp 2 O += P V:
//               S(A, 0) | S(B, 0) | S(A, 1)  O_A += P_A V(0) | S(B, 1)  O_B += P_B V(0) | ...
//               There is one S for both tiles: it is free as soon as the softmax warps hold the scores in registers, so
//               that S of the next unit is computed under the softmax of this one and under the PV of the one before.
//               (c3 29.8 -> 29.2 us, 16 x 8192 verify 100 -> 92, 16 decode blocks 78.5 -> 76.5 against the schedule in which P overwrote
//               S and the next S waited for PV.)  Long tensor-bound runs are at the board's power cap either way.
//   warps 4-7   softmax of tile A, warps 8-11 softmax of tile B: one thread per query row (TMEM lane).
//               The whole 128-column score row is held in registers (the two softmax warpgroups take
//               registers from warps 0-3 with setmaxnreg), so S is read from TMEM once: row maximum,
//               exponentials with packed f32x2 arithmetic, P written to TMEM as packed bf16 (the A
//               operand of the P V MMA comes from TMEM), O rescaled in TMEM only when the row maximum
//               grew by more than 2^8.
// The Q tiles arrive by TMA (warps 3 and 2) while warp 0 already streams K/V; results leave through a per-warp shared-memory staging area (the
// Q tiles, dead by then): split partials as they lie there, in bulk copies of 64 or 32 columns, finished rows as whole-row stores.  The block's own K/V rows go
// from the tiles into the pool by TMA.  What a CTA does once runs at five clocks and more an instruction and counts as much as its tiles where these
// are few (from the dependency wait to the first scores 3.1 -> 2.3 us, c3 29.2 -> 27.2 us, 3584 uncached tokens, 24/8 heads, 85.7 -> 79.9).
// TMEM columns: S [0,128) P_A [128,192) P_B [192,256) O_A [256,384) O_B [384,512).
// Every mbarrier wait is bounded: on time-out the CTA records AGX_DEV_WAIT_TIMEOUT and tears down.
#include <cuda.h>
#include <math.h>
#include <string.h>

#include "agx_internal.cuh"
#include "agx_sm100.cuh"

namespace agx {

namespace {

constexpr int kD = 128;
constexpr int kBN = 128;                    // KV tokens per tile
// Two schedules share the kernel (template parameter kStreams):
//   false  two 128-row Q tiles A and B per CTA (256 rows), both meet every KV tile;
//   true   ONE 128-row Q tile per CTA (verify blocks and short suffixes: q * G <= 128 rows, most of them
//          padding); the two softmax warpgroups take the even and the odd KV tiles of the same rows, each with
//          its own S and O accumulators in TMEM, and are merged inside the CTA at the end.  The step is
//          HBM-bound, so the padded MMA rows cost nothing that matters, while every K/V byte is read once
//          and the softmax of one tile hides behind the MMAs and copies of the next.
template <bool kStreams> struct Sched {
    static constexpr int kRows = kStreams ? 128 : 256;     // query rows per CTA
    static constexpr int kStagesK = kStreams ? 3 : 2;      // K is freed early (QK of a tile runs a unit ahead), V late
    static constexpr int kStagesV = 3;
};
constexpr int kThreads = 384;
constexpr uint32_t kTileBytes = 128 * 256;  // one operand tile: [2 halves of 64 dims][128 rows][128 B]
constexpr uint32_t kHalfBytes = 128 * 128;  // (Q tiles: [2 halves][128 rows][128 B])
constexpr uint32_t kPageBytes = kPage * 256; // K/V tiles: 8 pages of [2 row groups][2 halves of 64 dims][8 rows][128 B], as TMA writes them
constexpr uint32_t kOffQ = 0;
constexpr uint32_t kOffK = 2 * kTileBytes;
constexpr uint32_t kOffV = kOffK + 3 * kTileBytes;
constexpr uint32_t kOffBar = kOffV + 2 * kTileBytes;
// V stage s: the first two at kOffV, the third behind two K stages, or (kStreams: three K stages) in the unused second Q tile
template <bool kStreams>
__host__ __device__ constexpr uint32_t v_stage_off(int s) { return s < 2 ? kOffV + s * kTileBytes : kStreams ? kOffQ + kTileBytes : kOffK + 2 * kTileBytes; }
// kStreams epilogue: where stream 1's O row `rt` (512 bytes) waits for stream 0: in the K and the V stage that neither of the last two tiles is in, from
// which the block's own rows may still be on their way to the pool.
__device__ __forceinline__ uint32_t park_off(int rt, int n_tiles) {
    const int s = n_tiles % 3;
    return (rt < 64 ? kOffK + s * kTileBytes : v_stage_off<true>(s)) + (rt & 63) * 512;
}
constexpr uint32_t kOffCtx = kOffBar + 256;            // what the epilogue needs to know, parked at kernel start
constexpr uint32_t kOffPages = kOffBar + 512;          // row-group coordinates of the pages of up to 16 tiles
constexpr uint32_t kSmemBytes = kOffPages + 512 + 1024;   // + alignment slack
constexpr float kRescaleThreshold = 8.0f;              // log2 units
// Of every 8 column pairs, this many take the polynomial 2^x instead of the special-function unit (16 exponentials per clock
// and SM: the two Q tiles' 2 x 128 x 128 take as long as their MMAs).  0 / 1 / 2: c3 30.2 / 29.5 / 30.6 us, 3584 uncached
// tokens 89.5 / 88.7 / 91.5, 8000 + 700 tokens 107.2 / 106.8 / 109.2, the long prefill 1012 / 974 / 990 at the power cap.
constexpr int kPolyPairsOf8 = 1;

// barrier slots (8 bytes each)
enum { BAR_K_FULL = 0, BAR_K_EMPTY = 3, BAR_V_FULL = 6, BAR_V_EMPTY = 9, BAR_S_FULL = 12, BAR_P_READY = 14,
       BAR_O_FULL = 16, BAR_Q_FULL = 17, BAR_P_TAIL = 18, BAR_CTX = 20, BAR_P_FREE = 21, BAR_S_FREE = 23, BAR_Q_FULL_B = 24, BAR_O_FULL_B = 25, BAR_COUNT = 26 };
// P is handed to the MMA warp in two parts: the first kPvHeadSteps k-steps (16 tokens each) as soon as they are
// stored, so that their PV MMAs run while the softmax warpgroup still works on the last columns
constexpr int kPvHeadSteps = 6;
constexpr int kRegsLow = 96, kRegsHigh = 200; // 128 * 96 + 256 * 200 <= 384 * 168

constexpr uint32_t kTmemCols = 512;
constexpr uint32_t kColS = 0, kColP = 128, kColO = 256;  // one S for both; P + 64 * tile, O + 128 * tile

// tcgen05 instruction descriptor, kind::f16: D = f32, A = B = bf16, M = 128, N = 128
constexpr uint32_t kIdescBase = (1u << 4) | (1u << 7) | (1u << 10) | ((128u >> 3) << 17) | ((128u >> 4) << 24);
constexpr uint32_t kIdescQK = kIdescBase;              // A, B both K-major
constexpr uint32_t kIdescPV = kIdescBase | (1u << 16); // B (= V) is MN-major

__device__ __forceinline__ void tmem_st_x16(uint32_t taddr, const uint32_t* r) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};\n"
                 :: "r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]));
}
__device__ __forceinline__ void tmem_st_x32(uint32_t taddr, const uint32_t* r) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};\n"
                 :: "r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31]));
}


// Packed pairs of floats in one 64-bit register, for the f32x2 arithmetic instructions.
__device__ __forceinline__ uint64_t pk2(float lo, float hi) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};\n" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void upk2(uint64_t v, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;\n" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t fma2p(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;\n" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ uint64_t add2p(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("add.rn.f32x2 %0, %1, %2;\n" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ uint64_t mul2p(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("mul.rn.f32x2 %0, %1, %2;\n" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
// 2^x for a packed pair on the FMA pipes instead of the special-function unit: n = round(x) by the
// 1.5 * 2^23 trick, f = x - n in [-0.5, 0.5], 2^f by a polynomial of degree 5 fitted (Lawson's
// iteration) to minimise the maximum relative error on that interval (2.1e-7 evaluated in fp32, no more than the
// special-function unit's), times 2^n.  As with that unit a NaN stays a NaN and -inf, a masked score, gives exactly 0: x is clamped at -127
// by a maximum that passes NaN on, and the exponent field of 2^-127 is 0.
__device__ __forceinline__ float max_nan(float a, float b) {
    float d;
    asm("max.NaN.f32 %0, %1, %2;\n" : "=f"(d) : "f"(a), "f"(b));
    return d;
}
__device__ __forceinline__ void ex2_poly2(uint64_t x, float& p0, float& p1) {
    float x0, x1;
    upk2(x, x0, x1);
    x = pk2(max_nan(x0, -127.f), max_nan(x1, -127.f));
    const uint64_t magic = pk2(12582912.f, 12582912.f), neg_magic = pk2(-12582912.f, -12582912.f);
    const uint64_t t = add2p(x, magic);
    const uint64_t n = add2p(t, neg_magic);
    const uint64_t f = fma2p(n, pk2(-1.f, -1.f), x);
    auto c2 = [](float c) { return pk2(c, c); };
    uint64_t q = fma2p(f, c2(1.32764725e-3f), c2(9.67554096e-3f));
    q = fma2p(q, f, c2(5.55071309e-2f));
    q = fma2p(q, f, c2(2.40221202e-1f));
    q = fma2p(q, f, c2(6.93146944e-1f));
    q = fma2p(q, f, c2(1.00000012f));
    float t0, t1;
    upk2(t, t0, t1);   // (the low bits of t are n: shifted into the exponent field, on top of that of 1.0)
    upk2(mul2p(q, pk2(__int_as_float(__float_as_int(t0) * 8388608 + 0x3F800000), __int_as_float(__float_as_int(t1) * 8388608 + 0x3F800000))), p0, p1);
}
__device__ __forceinline__ void add2(float& d0, float& d1, float a0, float a1) {
    upk2(add2p(pk2(d0, d1), pk2(a0, a1)), d0, d1);
}
__device__ __forceinline__ float max3(float a, float b, float c) {
    float d;
    asm("max.f32 %0, %1, %2, %3;\n" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}
// What one CTA works on, derived from its block index alone.
struct TileItem {
    int g, G, P, q, rows, row0, split, nsplit, n_tiles, kv_begin, kv_end, vis_end, q_row0, seq_index;
};
// Everything the epilogue needs, kept in shared memory: kernel parameters reached through a pointer are
// slow to read, and registers are too precious across the main loop.
struct EpiCtx {
    TileItem it;
    int part_base, hq;
    unsigned char* part_tile;   // 256-row schedule: this CTA's tile of partials, or the first 32 columns of its rows (fp32)
    void* out;
    float* part_o;
    float2* part_ml;
    signed char* part_exp;
    float* lse;
    int* status;
    unsigned long long magic;   // (row * magic) >> 32 == row / G exactly for rows < 2^22
};
template <bool kStreams>
__device__ __forceinline__ TileItem locate_item(const AttnParams& p, int block) {
    constexpr int kRowsPerCta = Sched<kStreams>::kRows;
    const int si = find_seq(p, block);
    const SeqPlan& sp = p.seq[si];
    TileItem it;
    // work items reach the SMs in block order: the row chunks that see the most tokens (the last ones) go first.
    // block - item0 = ((g * row_chunks) + last - rc) * nsplit + split, or (((last - rc) * hkv) + g) * nsplit + split
    const unsigned item = block - sp.item0, group = item / (unsigned)sp.nsplit;   // (signed divisions take twice as long)
    it.nsplit = sp.nsplit;
    it.split = (int)(item - group * sp.nsplit);
    const int inner = sp.chunk_major ? p.hkv : sp.row_chunks;
    const int outer_idx = (int)(group / (unsigned)inner), inner_idx = (int)group - outer_idx * inner;
    it.g = sp.chunk_major ? inner_idx : outer_idx;
    const int rc = sp.row_chunks - 1 - (sp.chunk_major ? outer_idx : inner_idx);
    it.G = p.gqa;
    it.P = sp.prefix_len; it.q = sp.q_len;
    it.rows = it.q * it.G;
    it.row0 = rc * kRowsPerCta;
    it.vis_end = it.P + min(it.q - 1, (int)(((uint64_t)(uint32_t)(it.row0 + kRowsPerCta - 1) * p.row_div_magic) >> 32)) + 1;  // tokens the chunk's last row sees
    it.kv_begin = it.split * sp.split_tokens;
    it.kv_end = min(it.vis_end, it.kv_begin + sp.split_tokens);
    it.n_tiles = max(0, (it.kv_end - it.kv_begin + kBN - 1) / kBN);
    it.q_row0 = sp.q_row0; it.seq_index = sp.seq_index;
    return it;
}

// Epilogue of a softmax thread: the O row leaves TMEM through this warp's 8 KB of the (now idle) Q tiles (256-row schedule).
// With a single KV split the rows are normalised and written as bf16; otherwise partials and (m, l) go to the
// workspace for the combine kernel.  Kept out of line, and re-deriving its indices from the block index,
// so that nothing but its few arguments has to stay alive across the register-hungry main loop.
template <bool kStreams, bool kF32Part>
__device__ __noinline__ void tile_epilogue(unsigned char* smem, uint32_t tO, float m_ref, float l_run, bool ok) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    {   // the context is written by another warp at kernel start: wait for its arrival (long complete, normally)
        const uint32_t ctx_bar = smem_u32(smem) + kOffBar + 8u * BAR_CTX;
        volatile int* abort_flag = (volatile int*)(smem + kOffBar + BAR_COUNT * 8);
        if (!mbar_wait(ctx_bar, 0, abort_flag, nullptr, *(const long long*)(smem + kOffBar + BAR_COUNT * 8 + 16))) ok = false;
    }
    const EpiCtx cx = *(const EpiCtx*)(smem + kOffCtx);
    const TileItem& it = cx.it;
    const bool warp_has_rows = it.row0 + ((warp & 3) << 5) + (kStreams ? 0 : ((warp - 4) >> 2) * 128) < it.rows;
    float w_own = 1.f, w_other = 0.f;   // kStreams: weights of the two streams' accumulators
    if (kStreams) {
        // Stream 1 (warps 8-11) parks its rows in shared memory; stream 0 (warps 4-7) adds them to its own.
        const int rt = ((warp & 3) << 5) + lane;
        unsigned char* park = smem + park_off(rt, it.n_tiles);
        float2* park_ml = (float2*)(smem + kOffQ);   // (Q is dead)
        if (warp >= 8 && ok && warp_has_rows) {
            tc_fence_after();
            uint32_t oreg[32];
#pragma unroll
            for (int c4 = 0; c4 < 4; ++c4) {
                tmem_ld_x32(tO + c4 * 32, oreg);
                tmem_wait_ld();
#pragma unroll
                for (int v = 0; v < 8; ++v)
                    *(uint4*)(park + (((c4 * 8 + v) ^ lane) << 4)) = make_uint4(oreg[4 * v], oreg[4 * v + 1], oreg[4 * v + 2], oreg[4 * v + 3]);
            }
            park_ml[rt] = make_float2(m_ref, l_run);
        }
        // every softmax thread reaches this barrier, also after a bounded wait gave up somewhere in the CTA
        asm volatile("bar.sync 1, 256;\n" ::: "memory");
        if (warp >= 8 || !ok || !warp_has_rows || *(volatile int*)(smem + kOffBar + BAR_COUNT * 8)) return;
        const float2 other = park_ml[rt];
        const float m_new = fmaxf(m_ref, other.x);
        w_own = (m_ref == -INFINITY) ? 0.f : ex2(m_ref - m_new);
        w_other = (other.x == -INFINITY) ? 0.f : ex2(other.x - m_new);
        l_run = l_run * w_own + other.y * w_other;
        m_ref = m_new;
    }
    if (!warp_has_rows) return;
    unsigned char* stage = smem + kOffQ + (warp - 4) * 8192;     // [32 rows][256 B], 16-byte units XOR-swizzled by row (Q is dead)
    const int r_warp0 = it.row0 + (warp - 4) * 32;               // first row of this warp
    const uint64_t magic = cx.magic;                             // (row * magic) >> 32 == row / G exactly for rows < 2^22
    const bool single = it.nsplit == 1;
    const float inv = (l_run > 0.f) ? 1.f / l_run : 0.f;
    // per-row scalars, and the row's destination: lane j works them out for row j once, the copy loop below fetches
    // them by shuffle (a single warp doing the index arithmetic row by row took longer than the copies themselves)
    unsigned long long row_dst = 0;
    long long entry = -1;   // of this lane's partial
    {
        const int r = r_warp0 + lane;
        if (r < it.rows) {
            const int i = (int)(((uint64_t)(uint32_t)r * magic) >> 32), h = it.g * it.G + (r - i * it.G);
            if (single) {
                if (cx.lse) cx.lse[(long long)(it.q_row0 + i) * cx.hq + h] = (m_ref + log2f(l_run)) * 0.6931471805599453f;
                row_dst = (unsigned long long)((unsigned char*)cx.out + ((long long)(it.q_row0 + i) * cx.hq + h) * 256);
            } else {
                const long long e = (long long)cx.part_base + ((long long)i * cx.hq + h) * it.nsplit + it.split;
                cx.part_ml[e] = make_float2(m_ref, l_run);
                entry = e;
                if (kStreams) row_dst = (unsigned long long)(cx.part_o + e * kD);
            }
        }
    }
    // (the scalars above cost 0.4 us: they go under the last PV; 2 x 1200 uncached tokens 44.0 -> 43.1 us, 1000 + 128 13.5 -> 13.3)
    if (!kStreams && !mbar_wait(smem_u32(smem) + kOffBar + 8u * (warp < 8 ? BAR_O_FULL : BAR_O_FULL_B), 0, (volatile int*)(smem + kOffBar + BAR_COUNT * 8), cx.status,
                                *(const long long*)(smem + kOffBar + BAR_COUNT * 8 + 16))) return;
    tc_fence_after();
    // 128 bytes of each of the warp's rows, as they lie in a half of the staging area, to `at` of this CTA's partials
    auto leave = [&](const unsigned char* half, long long at) {
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
        __syncwarp();
        if (lane == 0) {
            asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;\n" ::"l"(cx.part_tile + at + (warp - 4) * 4096), "r"(smem_u32(half)), "r"(min(32, it.rows - r_warp0) * 128) : "memory");
            asm volatile("cp.async.bulk.commit_group;\n" ::: "memory");
        }
    };
    float top = 0.f;   // fp16 partials: the row's largest value
    {
        uint32_t oreg[64];   // two 32-column chunks per TMEM round trip
#pragma unroll 1
        for (int c8 = 0; c8 < 4; c8 += 2) {   // (code that runs once a CTA is fetched as it runs: not unrolled)
            tmem_ld_x32(tO + c8 * 32, oreg);
            tmem_ld_x32(tO + c8 * 32 + 32, oreg + 32);
            tmem_wait_ld();
            if (kStreams) {
                const unsigned char* park = smem + park_off(((warp & 3) << 5) + lane, it.n_tiles);
#pragma unroll
                for (int v = 0; v < 16; ++v) {
                    const float4 o1 = *(const float4*)(park + (((c8 * 8 + v) ^ lane) << 4));
                    oreg[4 * v + 0] = __float_as_uint(__uint_as_float(oreg[4 * v + 0]) * w_own + (w_other != 0.f ? o1.x * w_other : 0.f));
                    oreg[4 * v + 1] = __float_as_uint(__uint_as_float(oreg[4 * v + 1]) * w_own + (w_other != 0.f ? o1.y * w_other : 0.f));
                    oreg[4 * v + 2] = __float_as_uint(__uint_as_float(oreg[4 * v + 2]) * w_own + (w_other != 0.f ? o1.z * w_other : 0.f));
                    oreg[4 * v + 3] = __float_as_uint(__uint_as_float(oreg[4 * v + 3]) * w_own + (w_other != 0.f ? o1.w * w_other : 0.f));
                }
            }
            if (single || (!kStreams && !kF32Part)) {   // (the 256-row schedule normalises its fp16 partials too)
#pragma unroll
                for (int c = 0; c < 64; ++c) oreg[c] = __float_as_uint(__uint_as_float(oreg[c]) * inv);
            }
            if (kStreams) {
                // one warp with at most 32 rows: each lane stores its own row straight from registers (16 KB in all;
                // staging it through shared memory for whole-row stores took a single warp longer than these do)
                if (row_dst) {
#pragma unroll
                    for (int v = 0; v < 16; ++v) {
                        if (single) {
                            uint2 pk;
                            pk.x = pack_bf16(__uint_as_float(oreg[4 * v]), __uint_as_float(oreg[4 * v + 1]));
                            pk.y = pack_bf16(__uint_as_float(oreg[4 * v + 2]), __uint_as_float(oreg[4 * v + 3]));
                            *(uint2*)((unsigned char*)row_dst + (c8 * 8 + v) * 8) = pk;
                        } else {
                            __stcg((uint4*)((unsigned char*)row_dst + (c8 * 8 + v) * 16),
                                   make_uint4(oreg[4 * v], oreg[4 * v + 1], oreg[4 * v + 2], oreg[4 * v + 3]));
                        }
                    }
                }
            } else if (kF32Part && !single) {
                // fp32 partials the same way, 32 columns at a time through either half of the staging area
#pragma unroll
                for (int c4 = 0; c4 < 2; ++c4) {
                    unsigned char* half = stage + c4 * 4096;
                    if (c8) {
                        if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 1;\n" ::: "memory");
                        __syncwarp();
                    }
#pragma unroll
                    for (int v = 0; v < 8; ++v)
                        *(uint4*)(half + lane * 128 + ((v ^ (lane & 7)) << 4)) = make_uint4(oreg[32 * c4 + 4 * v], oreg[32 * c4 + 4 * v + 1], oreg[32 * c4 + 4 * v + 2], oreg[32 * c4 + 4 * v + 3]);
                    leave(half, (long long)(c8 + c4) * it.rows * 128);
                }
            } else if (!single) {
                // fp16 split partials, 64 columns of the warp's rows at a time: 128 bytes per row through the staging area, 16-byte units XOR-swizzled by row, and
                // on their way as they lie there, one bulk copy, while the other columns are read (128 rows
                // over 1000 tokens 11.5 -> 11.1 us, 250 over 900 with 16/2 heads 11.4 -> 11.0, 512 over 3072 with 24/8 25.7 -> 25.5 against one copy at the end)
                unsigned char* half = stage + (c8 >> 1) * 4096;
                float top1 = 0.f;
#pragma unroll
                for (int v = 0; v < 8; ++v) {
                    uint4 pk;
                    pk.x = pack_f16(__uint_as_float(oreg[8 * v + 0]), __uint_as_float(oreg[8 * v + 1]));
                    pk.y = pack_f16(__uint_as_float(oreg[8 * v + 2]), __uint_as_float(oreg[8 * v + 3]));
                    pk.z = pack_f16(__uint_as_float(oreg[8 * v + 4]), __uint_as_float(oreg[8 * v + 5]));
                    pk.w = pack_f16(__uint_as_float(oreg[8 * v + 6]), __uint_as_float(oreg[8 * v + 7]));
                    top = max3_abs(top, __uint_as_float(oreg[8 * v]), __uint_as_float(oreg[8 * v + 1]));
                    top1 = max3_abs(top1, __uint_as_float(oreg[8 * v + 2]), __uint_as_float(oreg[8 * v + 3]));
                    top = max3_abs(top, __uint_as_float(oreg[8 * v + 4]), __uint_as_float(oreg[8 * v + 5]));
                    top1 = max3_abs(top1, __uint_as_float(oreg[8 * v + 6]), __uint_as_float(oreg[8 * v + 7]));
                    *(uint4*)(half + lane * 128 + ((v ^ (lane & 7)) << 4)) = pk;
                }
                top = fmaxf(top, top1);
                leave(half, (c8 >> 1) * 32768);
            } else {
                // bf16 results: 256 bytes per row go through the staging area, 16-byte units XOR-swizzled by row
#pragma unroll
                for (int v = 0; v < 8; ++v) {
                    uint4 pk;
                    pk.x = pack_bf16(__uint_as_float(oreg[8 * v + 0]), __uint_as_float(oreg[8 * v + 1]));
                    pk.y = pack_bf16(__uint_as_float(oreg[8 * v + 2]), __uint_as_float(oreg[8 * v + 3]));
                    pk.z = pack_bf16(__uint_as_float(oreg[8 * v + 4]), __uint_as_float(oreg[8 * v + 5]));
                    pk.w = pack_bf16(__uint_as_float(oreg[8 * v + 6]), __uint_as_float(oreg[8 * v + 7]));
                    *(uint4*)(stage + lane * 256 + ((((c8 >> 1) * 8 + v) ^ (lane & 15)) << 4)) = pk;
                }
            }
        }
    }
    // fp16 rows that need more than its range.  (The loops are rolled up: in line and unrolled, never taken, this cost 0.2 to 0.5 us.)
    const bool again = !kStreams && !kF32Part && !single && __any_sync(0xFFFFFFFFu, entry >= 0 && (top < kFp16Least || top > kFp16Most));
    const int n_valid = min(32, it.rows - r_warp0);
    if (!again) {
        if (kStreams) return;
        if (!single) {
            if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;\n" ::: "memory");   // (the staging area is read before the CTA ends)
            return;
        }
        __syncwarp();
        // a half-warp writes one 256-byte row per instruction (lane j moves 16-byte unit j % 16 of row 2 u + j / 16); eight
        // row pairs' loads are in flight before the first store
        for (int rl0 = 0; rl0 < n_valid; rl0 += 16) {
            uint4 v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int rl = rl0 + 2 * u + (lane >> 4);
                v[u] = *(const uint4*)(stage + rl * 256 + (((lane & 15) ^ (rl & 15)) << 4));
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int rl = rl0 + 2 * u + (lane >> 4);
                const unsigned long long dst = __shfl_sync(0xFFFFFFFFu, row_dst, rl & 31);
                if (rl < n_valid) *(uint4*)((unsigned char*)dst + (lane & 15) * 16) = v[u];
            }
        }
        return;
    }
    auto piece = [&](int c, float (&x)[16]) {   // columns [c, c + 16)
        tmem_ld<16>(tO + c, (uint32_t*)x);
        tmem_wait_ld();
#pragma unroll
        for (int k = 0; k < 16; ++k) x[k] *= inv;
    };
    float x[16];
    top = 0.f;
#pragma unroll 1
    for (int c = 0; c < kD; c += 16) {
        piece(c, x);
#pragma unroll
        for (int k = 0; k < 16; ++k) top = fmaxf(top, finite_abs(x[k]));
    }
    const int e = entry >= 0 ? fp16_exponent(top) : 0;
    if (__any_sync(0xFFFFFFFFu, e)) {
        if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;\n" ::: "memory");   // (the rows are on their way as they were)
        __syncwarp();
        if (e) {
            cx.part_ml[entry] = make_float2(m_ref, -l_run);
            cx.part_exp[entry] = (signed char)e;
        }
        const float f = pow2(-e);
#pragma unroll 1
        for (int c = 0; c < kD; c += 16) {
            piece(c, x);
#pragma unroll
            for (int k = 0; k < 16; k += 8) {
                const uint4 pk = make_uint4(pack_f16(x[k] * f, x[k + 1] * f), pack_f16(x[k + 2] * f, x[k + 3] * f), pack_f16(x[k + 4] * f, x[k + 5] * f),
                                            pack_f16(x[k + 6] * f, x[k + 7] * f));
                const int unit = (c + k) / 8;
                *(uint4*)(stage + (unit >> 3) * 4096 + lane * 128 + (((unit ^ lane) & 7) << 4)) = pk;
            }
        }
        leave(stage, 0);
        leave(stage + 4096, 32768);
    }
    if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;\n" ::: "memory");
}

// K or V of a tile that holds block rows or ends inside a page, by the whole producer warp.  Tokens [0, pool_end) come from the pool,
// with a fused append the block's own from k_new / v_new: pages from the pool; a tile of nothing but block rows as one copy where
// 128 rows are there; else row groups of 8 tokens from k_new / v_new; and by hand the groups that mix prefix and block or, for V,
// reach beyond the last token (zeros: P is 0 there, but 0 * NaN is not).  The copies are on their way before the loads by hand are waited for, and
// with `waited` false (a fused append whose cached-prefix pages may be fetched early) those of the pool's pages before the dependency wait.
// Out of line: inlined twice into the producer's loop it cost the other warps 7 % on a long prefill that never takes it (instruction fetch).
__device__ __noinline__ void load_mixed(const AttnParams& p, const CUtensorMap* pool_map, const CUtensorMap* rows8, const CUtensorMap* rows128,
                                        const unsigned char* pool, const unsigned char* rows, bool is_v, int g, int P, int L, int q_row0,
                                        unsigned char* dst, uint32_t full_bar, int tok0, int npg, int group, bool waited) {
    const int lane = threadIdx.x & 31, hkv = p.hkv;
    const int pool_end = rows ? P : L, pool_full = pool_end & ~(kPage - 1);
    const int pool_pg = min(npg, max(0, (pool_full - tok0) >> 4));        // pages of the tile that come from the pool; lane l holds the first row group of page l
    const int own0 = tok0 + pool_pg * kPage, own1 = tok0 + npg * kPage;   // tokens of the pages that do not
    const int rows0 = min(own1, max(own0, (pool_end + 7) & ~7));          // row groups by TMA: [rows0, rows1)
    const int rows1 = rows ? max(rows0, min(own1, is_v ? (L & ~7) : ((L + 7) & ~7))) : rows0;
    const int own_group = __shfl_sync(0xFFFFFFFFu, group, pool_pg & 31);
    // (the whole-tile copy may bring in rows of the next sequence: for V none of them may be met by the MMAs, 16 tokens at a time)
    const int row0_new = q_row0 + tok0 - P;
    const bool big = rows && tok0 >= P && row0_new + kBN <= p.total_rows && (!is_v || own1 <= L);
    const uint32_t d = smem_u32(dst);
    if (lane == 0) mbar_expect_tx(full_bar, big ? kTileBytes : pool_pg * kPageBytes + (rows1 - rows0) * 256);
    __syncwarp();
    if (!big && lane < pool_pg) tma_load_page(d + lane * kPageBytes, pool_map, group, full_bar);
    __syncwarp();
    if (!waited) pdl_wait();
    if (big) {
        if (lane == 0) tma_load_rows128(d, rows128, row0_new, g, full_bar);
    } else {
        const int base = rows0 + lane * 8;
        if (base < rows1) tma_load_rows8(d + (base - tok0) * 256, rows8, q_row0 + base - P, g, full_bar);
    }
    __syncwarp();
    bool by_hand = false;
    for (int base = own0; base < own1 && !big; base += 8) {
        if (base == rows0) base = rows1;
        if (base >= own1 || (!is_v && base >= rows1)) break;   // (K rows beyond the last token are masked, whatever they are)
        by_hand = true;
        // half a warp a row, rows r0, r0 + 2, r0 + 4, r0 + 6 of the group
        const int r0 = lane >> 4, u0 = lane & 15;
        const unsigned char* in_pool = pool + ((long long)own_group * 8 + (base & 15) + r0) * 256 + u0 * 16;
        const unsigned char* in_rows = rows + ((long long)(q_row0 + base + r0 - P) * hkv + g) * 256 + u0 * 16;
        uint4 u[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int tok = base + r0 + 2 * j;
            const unsigned char* src = tok < pool_end ? in_pool + j * 512 : in_rows + j * hkv * 512;
            u[j] = make_uint4(0, 0, 0, 0);
            if (tok < L) u[j] = __ldcg((const uint4*)src);
        }
        unsigned char* at = dst + (base - tok0) * 256 + (u0 >> 3) * 1024;
#pragma unroll
        for (int j = 0; j < 4; ++j) { const int r = r0 + 2 * j; *(uint4*)(at + r * 128 + (((u0 & 7) ^ r) << 4)) = u[j]; }
    }
    if (by_hand) asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    __syncwarp();
    if (lane == 0) mbar_arrive(full_bar);
    __syncwarp();
}

// The block's own row groups of K tile `tok0` ahead of its stage's next tile: a chunk of 256 tokens (one head a group) lies in up to three tiles, and K
// has two stages.  Row groups from `lo` on, see the end of warp 0.
__device__ __noinline__ void store_k_groups(const AttnParams& p, const CUtensorMap* map, const int* pt_row, int g, int L, int lo, int tok0, uint32_t tile) {
    const int lane = threadIdx.x & 31, tok = tok0 + lane * 8;
    if (lane < kBN / 8 && tok >= lo && tok + 8 <= L) {
        const int id = tok / kPage < p.pt_stride ? __ldg(pt_row + tok / kPage) : -1;   // (a bad one is reported with V's)
        if (id >= 0 && id < p.num_pages) tma_store_group(map, (id * p.hkv + g) * (kPage / 8) + ((tok >> 3) & 1), tile + lane * 8 * 256);
        asm volatile("cp.async.bulk.commit_group;\n" ::: "memory");
        asm volatile("cp.async.bulk.wait_group.read 0;\n" ::: "memory");
    }
    __syncwarp();
}

// Rows of the block that are in no whole group of eight, from k_new / v_new to the pool by one warp, half a warp a row: of the groups that the block
// begins and ends in those whose first block row is in [own_lo, own_hi).
__device__ __forceinline__ void store_ends(const AttnParams& p, const SeqPlan& sp, int g, int L, int own_lo, int own_hi) {
    const int lane = threadIdx.x & 31, r0 = lane >> 4, P = sp.prefix_len;
#pragma unroll 1
    for (int end = 0; end < 2; ++end) {
        const int t0 = (end ? L : P) & ~7, first = max(t0, P);
        if (t0 == (end ? L : P) || (end && t0 < P) || first < own_lo || first >= own_hi) continue;   // (whole, the other one's, or another CTA's)
        const int id = t0 / kPage < p.pt_stride ? __ldg(p.page_table + (long long)sp.seq_index * p.pt_stride + t0 / kPage) : -1;
        const long long from = ((long long)(sp.q_row0 + t0 + r0 - P) * p.hkv + g) * 256 + (lane & 15) * 16;
        auto mine = [&](int j) { const int tok = t0 + r0 + 2 * j; return tok >= P && tok < L; };
        uint4 k[4], v[4];
#pragma unroll
        for (int j = 0; j < 4; ++j)   // (in one trip with the page id)
            if (mine(j)) {
                k[j] = __ldg((const uint4*)((const unsigned char*)p.k_new + from + j * p.hkv * 512));
                v[j] = __ldg((const uint4*)((const unsigned char*)p.v_new + from + j * p.hkv * 512));
            }
        if (id < 0 || id >= p.num_pages) { atomicOr(p.status, AGX_DEV_BAD_PAGE); continue; }
        const long long to = (((long long)id * p.hkv + g) * kPage + (t0 & 15) + r0) * 256 + (lane & 15) * 16;
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (mine(j)) {
                *(uint4*)((unsigned char*)p.k_pool + to + j * 512) = k[j];
                *(uint4*)((unsigned char*)p.v_pool + to + j * 512) = v[j];
            }
    }
    __syncwarp();
}

// A Q tile's rows [row0, row0 + n) of KV head g, n <= 128, by one thread: single rows up to the next whole token, boxes of q_tokens tokens
// while they fit the tile (the last one may bring rows nobody looks at), single rows again.  Where G divides 128 that is one box per half.
struct QTile {
    int n, i0, hh0, front, boxed;   // rows; token and head of the first; rows [front, boxed) come in boxes
    __device__ __forceinline__ QTile(int row0, int rows, int G, int box, unsigned long long magic) {
        n = max(0, min(128, rows - row0));
        i0 = (int)(((uint64_t)(uint32_t)row0 * magic) >> 32);
        hh0 = row0 - i0 * G;
        front = boxed = hh0 ? min(n, G - hh0) : 0;
        while (box > 0 && boxed < n && boxed + box <= 128) boxed += box;
    }
    __device__ __forceinline__ void load(const RowsMaps& maps, uint32_t tile, uint32_t bar, int G, int q_row0, int g) const {
        mbar_arrive_expect_tx(bar, 256u * (uint32_t)max(n, boxed));
        int token = q_row0 + i0, hh = hh0, r = 0;
        auto copy = [&](const CUtensorMap* map) {
            tma_load_q(tile + r * 128, map, hh, token, 0, g, bar);
            tma_load_q(tile + r * 128 + kHalfBytes, map, hh, token, 1, g, bar);
        };
#pragma unroll 1
        for (; r < front; ++r, ++hh) copy(&maps.q_row);
        if (hh0) { hh = 0; ++token; }
#pragma unroll 1
        for (; r < boxed; r += maps.q_tokens * G, token += maps.q_tokens) copy(&maps.q_box);
#pragma unroll 1
        for (; r < n; ++r) {
            copy(&maps.q_row);
            if (++hh == G) { hh = 0; ++token; }
        }
    }
};

}  // namespace

template <bool kStreams, bool kF32Part>
__global__ void __launch_bounds__(kThreads, 1)
attn_tile_bf16_kernel(const __grid_constant__ AttnParams p, const __grid_constant__ CUtensorMap map_k,
                      const __grid_constant__ CUtensorMap map_v, const __grid_constant__ RowsMaps maps_new) {
    extern __shared__ unsigned char smem_raw[];
    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    unsigned char* smem = smem_raw + (smem_base - smem_u32(smem_raw));
    volatile int* abort_flag = (volatile int*)(smem + kOffBar + BAR_COUNT * 8);
    uint32_t* tmem_slot = (uint32_t*)(smem + kOffBar + BAR_COUNT * 8 + 8);
    auto bar = [&](int i) { return smem_base + kOffBar + 8u * i; };

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

    constexpr int kRowsPerCta = Sched<kStreams>::kRows;
    constexpr int kStagesK = Sched<kStreams>::kStagesK, kStagesV = Sched<kStreams>::kStagesV;
    // ---- work item
    const TileItem it = locate_item<kStreams>(p, blockIdx.x);
    const SeqPlan& sp = p.seq[find_seq(p, blockIdx.x)];
    const int split = it.split, g = it.g, G = it.G, P = it.P, q = it.q, L = P + q, rows = it.rows, row0 = it.row0;
    const int kv_begin = it.kv_begin, kv_end = it.kv_end, n_tiles = it.n_tiles;

    pdl_launch_dependents();
    if (n_tiles == 0) {  // nothing visible in this split (nsplit > 1 by construction): publish (m, l) = (-inf, 0);
                         // the combine kernel does not read the O rows of such entries
        pdl_wait();
        for (int rl = tid; rl < kRowsPerCta; rl += kThreads) {
            const int r = row0 + rl;
            if (r >= rows) break;
            const int i = r / G, h = g * G + (r - i * G);
            p.part_ml[(long long)sp.part_base + ((long long)i * p.hq + h) * sp.nsplit + split] = make_float2(-INFINITY, 0.f);
        }
        return;
    }

    // ---- setup: barriers, TMEM, Q tiles
    // Early loads: with p.early_prefix the caller vouches that the page table and the K/V pages below the cached-prefix
    // length are not written by any launch still in flight, so the producer warp may fetch them while the launch in
    // front of this one drains.  Its first page ids are on their way while it sets the barriers up.
    const int stable_end = P & ~(kPage - 1);   // tokens below this sit in pages no append of this block touches
    const bool early_ids = p.early_prefix;
    const int n_pool_pages = max(0, (min(kv_end, p.k_new ? P : L) - kv_begin + kPage - 1) / kPage);   // pages of this CTA that the pool is read for
    int first_id = -1;
    const int* const first_id_at = p.page_table + (long long)sp.seq_index * p.pt_stride + kv_begin / kPage + lane;
    if (warp == 0 && early_ids && lane < n_pool_pages) first_id = __ldg(first_id_at);
    if (tid == 0) {
        for (int i = 0; i < BAR_COUNT; ++i)
            if (i != BAR_Q_FULL && i != BAR_Q_FULL_B && i != BAR_CTX) mbar_init(bar(i), (i == BAR_P_READY || i == BAR_P_READY + 1 || i == BAR_P_TAIL || i == BAR_P_TAIL + 1 || i == BAR_S_FREE) ? 4u : 1u);
        *abort_flag = 0;
        *(long long*)(smem + kOffBar + BAR_COUNT * 8 + 16) = p.wait_limit_cycles;   // for the out-of-line epilogue
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        asm volatile("prefetch.tensormap [%0];\n" ::"l"(&map_k) : "memory");
        asm volatile("prefetch.tensormap [%0];\n" ::"l"(&map_v) : "memory");
        if (p.k_new && kv_end > stable_end) {
            asm volatile("prefetch.tensormap [%0];\n" ::"l"(&maps_new.k128) : "memory");
            asm volatile("prefetch.tensormap [%0];\n" ::"l"(&maps_new.k8) : "memory");
            asm volatile("prefetch.tensormap [%0];\n" ::"l"(&maps_new.v128) : "memory");
            asm volatile("prefetch.tensormap [%0];\n" ::"l"(&maps_new.v8) : "memory");
        }
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(tmem_slot)), "r"(kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    if (warp == 3 && elect_one()) {
        mbar_init(bar(BAR_Q_FULL), 1);
        mbar_init(bar(BAR_Q_FULL_B), 1);
        mbar_init(bar(BAR_CTX), 1);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        asm volatile("prefetch.tensormap [%0];\n" ::"l"(maps_new.q_tokens ? &maps_new.q_box : &maps_new.q_row) : "memory");
    }
    // One Q tile: its rows of padding (most of them) are zeros, in Q here and in P below.  The MMAs work on them all the same, but zeros take less
    // of the board's power than whatever lay there: 16 x 8192 verify, for seconds on end, 208 us with neither, 201 with Q, 197 with both.
    if (kStreams && warp >= 4) {
        const QTile qt(row0, rows, G, maps_new.q_tokens * G, p.row_div_magic);
        for (int c = tid - 128 + max(qt.n, qt.boxed) * 8; c < 128 * 8; c += kThreads - 128) {
            *(uint4*)(smem + kOffQ + c * 16) = make_uint4(0, 0, 0, 0);
            *(uint4*)(smem + kOffQ + kHalfBytes + c * 16) = make_uint4(0, 0, 0, 0);
        }
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    }
    // Barriers initialised, TMEM address published.  Warps 0 and 3 only signal and go straight to their first copies: each of them has set up
    // all the barriers that it uses itself, and needs nothing else from the others.  No warp has waited for the launch in front yet: what follows such a wait (warps 0, 2 and 3 have one
    // each; whatever else the CTA reads or writes comes behind the Q tiles) is a chain of latencies with as little code as can be.
    tc_fence_before();
    if (warp == 0 || warp == 3) { __syncwarp(); asm volatile("bar.arrive 2, %0;\n" ::"n"(kThreads) : "memory"); }
    else asm volatile("bar.sync 2, %0;\n" ::"n"(kThreads) : "memory");
    tc_fence_after();
    const uint32_t tmem_base = (warp == 0 || warp == 3) ? 0u : *tmem_slot;
    // Fused append: a row group (eight tokens of half a page) is stored by the CTA whose row chunk's first query rows and whose split its first
    // block token lies in.  That CTA has the group in one of its last K and V tiles, and a whole one leaves from there by TMA (by_tma).
    const int own_lo = max(kv_begin, P + (int)(((uint64_t)(uint32_t)(row0 + G - 1) * p.row_div_magic) >> 32));
    const int own_hi = p.k_new ? min(kv_end, kv_begin + sp.split_tokens) : 0;
    auto by_tma = [&](int tok) { return tok >= P && tok + 8 <= L; };
    const int own_group0 = (max(own_lo, P) + 7) & ~7;   // the first that may be a whole one
    auto pages_in_tile = [&](int t) { return min(8, (kv_end - (kv_begin + t * kBN) + kPage - 1) / kPage); };

    // the softmax warpgroups keep a whole score row in registers: warps 0-3 hand registers over to them
    if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;\n" ::"n"(kRegsLow));
    if (warp == 0) {
        // ================= TMA producer =================
        if (!early_ids) {
            pdl_wait();
            if (lane < n_pool_pages) first_id = __ldg(first_id_at);
        }
        const int* pt_row = p.page_table + (long long)sp.seq_index * p.pt_stride;
        const int page0 = kv_begin / kPage;
        // Page ids are read 32 (four tiles) at a time and two groups ahead of the copies that need them; their row-group coordinates wait in
        // shared memory, so that the thread that issues the copies of a tile has them with two loads.
        int* const page_ring = (int*)(smem + kOffPages);   // [4 groups][32]
        auto load_ids = [&](int group) {   // (by the whole warp)
            const int pi = group * 32 + lane;
            return pi < n_pool_pages ? __ldg(pt_row + page0 + pi) : -1;
        };
        auto check_ids = [&](int group, int id) {
            if (group * 32 + lane < n_pool_pages && (id < 0 || id >= p.num_pages)) { id = 0; atomicOr(p.status, AGX_DEV_BAD_PAGE); }
            return id;
        };
        auto fetch_ids = [&](int group) { return check_ids(group, load_ids(group)); };
        auto put_ids = [&](int group, int id) { page_ring[(group & 3) * 32 + lane] = (id * p.hkv + g) * (kPage / 8); __syncwarp(); };
        bool ok = true;
        bool waited = !early_ids;            // has this warp passed the dependency wait?
        // tokens [0, pool_end) come from the pool; a tile wholly inside the pool's full pages is eight page copies, see load_mixed for others
        const int pool_full = (p.k_new ? P : L) & ~(kPage - 1);
        int last_k = -1, last_v = -1;   // last tiles whose copies were armed (for the drain below)
        const int n_groups = (n_pool_pages + 31) >> 5;
        if (n_groups > 0) put_ids(0, check_ids(0, first_id));
        int ids_ahead = 0, ahead = -1;       // group `ahead` has been read (its ids are in ids_ahead), groups below it are in page_ring
        int ks = 0, vs = 0;
        uint32_t kph = 1, vph = 1;
        // in the order of need: K(0), K(1), V(0), K(2), V(1), ..., V(n - 1)
        for (int i = 0; i <= n_tiles; ++i) {
#pragma unroll
            for (int is_v = 0; is_v < 2; ++is_v) {
                const int t = is_v ? i - 1 : i;
                if (t < 0 || t >= n_tiles || !ok) continue;
                const int tok0 = kv_begin + t * kBN;
                const bool whole = tok0 + kBN <= pool_full && tok0 + kBN <= kv_end;
                // tiles inside the cached prefix, as far as free stages go, may be requested before the wait, also part of a tile (load_mixed)
                if (!waited && !((tok0 + kBN <= stable_end || (!whole && p.k_new)) && t < (is_v ? kStagesV : kStagesK))) { pdl_wait(); waited = true; }
                if (!is_v && (t & 3) == 0) {
                    const int group = t >> 2;
                    if (group > 0 && group < n_groups) put_ids(group, ahead == group ? ids_ahead : fetch_ids(group));
                    if (waited && group + 1 < n_groups) { ids_ahead = fetch_ids(group + 1); ahead = group + 1; }
                }
                if (t == p.drop_stage) {   // test hook: this tile never arrives, its consumers' waits run out
                    if (is_v) { if (++vs == kStagesV) { vs = 0; vph ^= 1; } } else if (++ks == kStagesK) { ks = 0; kph ^= 1; }
                    continue;
                }
                const int s = is_v ? vs : ks;
                const uint32_t full = bar((is_v ? BAR_V_FULL : BAR_K_FULL) + s), empty = bar((is_v ? BAR_V_EMPTY : BAR_K_EMPTY) + s);
                const uint32_t off = is_v ? v_stage_off<kStreams>(s) : kOffK + s * kTileBytes;
                ok = mbar_wait(empty, is_v ? vph : kph, abort_flag, p.status, p.wait_limit_cycles);
                if (!ok) continue;
                if (is_v) last_v = t; else last_k = t;
                if (!kStreams && !is_v && p.k_new && p.drop_stage < 0 && tok0 - (kStagesK - 1) * kBN > own_group0)
                    store_k_groups(p, &maps_new.k_pool8, pt_row, g, L, own_group0, tok0 - kStagesK * kBN, smem_base + off);
                if (whole) {
                    if (elect_one()) {
                        const int4 c0 = *(const int4*)(page_ring + ((t * 8) & 127)), c1 = *(const int4*)(page_ring + ((t * 8) & 127) + 4);
                        const CUtensorMap* map = is_v ? &map_v : &map_k;
                        const uint32_t dst = smem_base + off;
                        mbar_arrive_expect_tx(full, kTileBytes);
                        tma_load_page(dst, map, c0.x, full);
                        tma_load_page(dst + kPageBytes, map, c0.y, full);
                        tma_load_page(dst + 2 * kPageBytes, map, c0.z, full);
                        tma_load_page(dst + 3 * kPageBytes, map, c0.w, full);
                        tma_load_page(dst + 4 * kPageBytes, map, c1.x, full);
                        tma_load_page(dst + 5 * kPageBytes, map, c1.y, full);
                        tma_load_page(dst + 6 * kPageBytes, map, c1.z, full);
                        tma_load_page(dst + 7 * kPageBytes, map, c1.w, full);
                    }
                } else {
                    load_mixed(p, is_v ? &map_v : &map_k, is_v ? &maps_new.v8 : &maps_new.k8, is_v ? &maps_new.v128 : &maps_new.k128,
                               (const unsigned char*)(is_v ? p.v_pool : p.k_pool), (const unsigned char*)(is_v ? p.v_new : p.k_new), is_v, g, P, L,
                               sp.q_row0, smem + off, full, tok0, pages_in_tile(t), page_ring[(t * 8 + (lane & 7)) & 127], waited);
                    waited = true;
                }
                __syncwarp();
                if (is_v) { if (++vs == kStagesV) { vs = 0; vph ^= 1; } } else if (++ks == kStagesK) { ks = 0; kph ^= 1; }
            }
        }
        // The block's own row groups go from the tiles into the pool, a lane per group (a chunk has 32 at most).  Through registers it was 85 tokens' worth of
        // loads and stores a CTA (3584 uncached tokens, 24/8 heads): in front of the softmax warps' loop 3 us of their way to the first scores; on warp 3
        // beside the loop its instructions slowed the softmax warps of its scheduler, and with them the CTA, by a quarter.
        // With one Q tile they went through registers of warp 3, eight tokens a trip to memory: 8/8 heads, 128 rows over 100 tokens 27.3 us, now 10.8 (12.5 by
        // ten warps in front of their loops).
        const int own_tok = own_group0 + lane * 8, own_t = (own_tok - kv_begin) / kBN;
        const bool leaves = ok && p.drop_stage < 0 && own_tok < own_hi && by_tma(own_tok);
        int own_id = -1;
        if (leaves) {
            if (own_tok / kPage < p.pt_stride) own_id = __ldg(pt_row + own_tok / kPage);   // (under the last copies)
            if (own_id >= p.num_pages) own_id = -1;
            if (own_id < 0) atomicOr(p.status, AGX_DEV_BAD_PAGE);
        }
        const int own_at = ((own_tok - kv_begin) & (kBN - 1)) * 256, own_group = (own_id * p.hkv + g) * (kPage / 8) + ((own_tok >> 3) & 1);
        // drain: the copies this warp started must land before the CTA's shared memory goes away.  Bounded by the
        // clock alone: after a time-out elsewhere in the CTA the abort flag is up, and the copies still have to land.
        if (lane == 0)
            for (int t = max(0, last_k - kStagesK + 1); t <= last_k; ++t)
                if (t != p.drop_stage) mbar_drain(bar(BAR_K_FULL + t % kStagesK), (t / kStagesK) & 1, p.wait_limit_cycles);
        __syncwarp();
        if (own_id >= 0 && own_t >= n_tiles - kStagesK) tma_store_group(&maps_new.k_pool8, own_group, smem_base + kOffK + (own_t % kStagesK) * kTileBytes + own_at);
        __syncwarp();
        if (lane == 0)
            for (int t = max(0, last_v - kStagesV + 1); t <= last_v; ++t)
                if (t != p.drop_stage) mbar_drain(bar(BAR_V_FULL + t % kStagesV), (t / kStagesV) & 1, p.wait_limit_cycles);
        __syncwarp();
        if (own_id >= 0) tma_store_group(&maps_new.v_pool8, own_group, smem_base + v_stage_off<kStreams>(own_t % kStagesV) + own_at);
        // (they are read before the CTA's shared memory goes away)
        asm volatile("cp.async.bulk.commit_group;\n" ::: "memory");
        asm volatile("cp.async.bulk.wait_group.read 0;\n" ::: "memory");
        __syncwarp();
    } else if (warp == 1 || warp == 2) {
        // ================= MMA issuers: one thread of warp 1 for S = Q K^T, one of warp 2 for O += P V =================
        // Units of work u = 0, 1, ...: a KV tile against tile A or B (x = u & 1); with kStreams one KV tile each.  S holds one unit's scores: it
        // is free again as soon as the softmax warps have them in registers, so QK of unit u + 1 runs under the softmax of unit u and
        // beside PV of unit u - 1.  Two issuing threads, because one was busy all the time: every wait of a warp that shares its scheduler
        // with two softmax warps costs it 90 cycles and more, also when there is nothing to wait for.
        const int n_units = kStreams ? n_tiles : 2 * n_tiles;
        if (!kStreams && warp == 2) {
            const QTile b(row0 + 128, rows, G, maps_new.q_tokens * G, p.row_div_magic);
            if (elect_one()) {
                pdl_wait();
                if (b.n > 0) b.load(maps_new, smem_base + kOffQ + kTileBytes, bar(BAR_Q_FULL_B), G, sp.q_row0, g);
                else mbar_arrive(bar(BAR_Q_FULL_B));   // (a tile of padding only: whatever is there)
            }
            __syncwarp();
        }
        if (warp == 1 && elect_one()) {
            const uint32_t tS = tmem_base + kColS;
            // descriptors differ only in the start address: add (byte offset >> 4) to a base descriptor
            const uint64_t q_desc0 = make_desc(smem_base + kOffQ, 16, 1024);
            const uint64_t k_desc0 = make_desc(smem_base + kOffK, 16, 2048);
            bool ok = mbar_wait(bar(BAR_Q_FULL), 0, abort_flag, p.status, p.wait_limit_cycles);
            int ks = 0;
            uint32_t kph = 0;
            for (int u = 0; u < n_units && ok; ++u) {
                const int x = u & 1;
                if (kStreams || x == 0) ok = mbar_wait(bar(BAR_K_FULL + ks), kph, abort_flag, p.status, p.wait_limit_cycles);
                if (!kStreams && ok && u == 1) ok = mbar_wait(bar(BAR_Q_FULL_B), 0, abort_flag, p.status, p.wait_limit_cycles);
                if (ok && u > 0) ok = mbar_wait(bar(BAR_S_FREE), x ^ 1, abort_flag, p.status, p.wait_limit_cycles);   // unit u - 1 is in registers
                if (!ok) break;
                tc_fence_after();
                const uint64_t qd = q_desc0 + (uint64_t)((kStreams ? 0 : x * kTileBytes) >> 4);
                const uint64_t kd = k_desc0 + (uint64_t)((ks * kTileBytes) >> 4);
#pragma unroll
                for (int s = 0; s < 8; ++s) {   // 8 k-steps of 16 dims
                    const uint64_t q_off = (uint64_t)(((s >> 2) * kHalfBytes + (s & 3) * 32) >> 4);
                    const uint64_t k_off = (uint64_t)(((s >> 2) * 1024 + (s & 3) * 32) >> 4);
                    umma_ss(tS, qd + q_off, kd + k_off, kIdescQK, s > 0);
                }
                umma_commit(bar(BAR_S_FULL + x));
                if (kStreams || x) {
                    umma_commit(bar(BAR_K_EMPTY + ks));
                    if (++ks == kStagesK) { ks = 0; kph ^= 1; }
                }
            }
        } else if (warp == 2 && elect_one()) {
            bool ok = true;
            int vs = 0;
            uint32_t vph = 0;
            for (int u = 0; u < n_units && ok; ++u) {
                const int x = u & 1, t = kStreams ? u : u >> 1, npg = pages_in_tile(t);
                const uint32_t ph = (u >> 1) & 1;
                const uint32_t tP = tmem_base + kColP + x * 64, tO = tmem_base + kColO + x * 128;
                const uint64_t vd = make_desc(smem_base + v_stage_off<kStreams>(vs), 1024, 2048);
                if (kStreams || x == 0) ok = mbar_wait(bar(BAR_V_FULL + vs), vph, abort_flag, p.status, p.wait_limit_cycles);
                // one k-step per page: the first kPvHeadSteps once P_READY says those columns of P are stored, the rest after P_TAIL
                if (ok) ok = mbar_wait(bar(BAR_P_READY + x), ph, abort_flag, p.status, p.wait_limit_cycles);
                if (!ok) break;
                tc_fence_after();
                if (npg == 8) {
#pragma unroll
                    for (int s = 0; s < kPvHeadSteps; ++s) umma_ts(tO, tP + s * 8, vd + (uint64_t)((s * kPageBytes) >> 4), kIdescPV, u >= 2 || s > 0);
                } else {
                    for (int s = 0; s < min(npg, kPvHeadSteps); ++s) umma_ts(tO, tP + s * 8, vd + (uint64_t)((s * kPageBytes) >> 4), kIdescPV, u >= 2 || s > 0);
                }
                ok = mbar_wait(bar(BAR_P_TAIL + x), ph, abort_flag, p.status, p.wait_limit_cycles);
                if (!ok) break;
                tc_fence_after();
                if (npg == 8) {
#pragma unroll
                    for (int s = kPvHeadSteps; s < 8; ++s) umma_ts(tO, tP + s * 8, vd + (uint64_t)((s * kPageBytes) >> 4), kIdescPV, true);
                } else {
                    for (int s = kPvHeadSteps; s < npg; ++s) umma_ts(tO, tP + s * 8, vd + (uint64_t)((s * kPageBytes) >> 4), kIdescPV, true);
                }
                umma_commit(bar(BAR_P_FREE + x));
                // (tile A's epilogue does not wait for tile B's last tile: 8 x 300 uncached tokens 30.5 -> 28.8 us, 256 9.41 -> 8.92, 128 over 1000 11.8 ->
                // 11.5, 512 over 3072 with 24/8 heads 26.0 -> 25.7)
                if (!kStreams && u == n_units - 2) umma_commit(bar(BAR_O_FULL));
                if (kStreams || x) {
                    umma_commit(bar(BAR_V_EMPTY + vs));
                    if (++vs == kStagesV) { vs = 0; vph ^= 1; }
                }
            }
            constexpr int kLast = kStreams ? BAR_O_FULL : BAR_O_FULL_B;
            umma_commit(bar(kLast));  // arrives when every MMA issued above has completed
            mbar_wait(bar(kLast), 0, abort_flag, p.status, p.wait_limit_cycles);
            // (the copies must land before the CTA's shared memory goes away, also after a time-out elsewhere)
            if (!kStreams) mbar_drain(bar(BAR_Q_FULL_B), 0, p.wait_limit_cycles);
        }
        __syncwarp();
    } else {   // warp 3
        // Q by TMA, with everything worked out before the dependency wait (a single thread takes five clocks and more an instruction).  cp.async of
        // one row by 16 threads took 2.1-2.7 us from the wait to the last byte, addresses and LSU; this 1.2.
        const QTile a(row0, rows, G, maps_new.q_tokens * G, p.row_div_magic);
        if (elect_one()) {
            pdl_wait();
            a.load(maps_new, smem_base + kOffQ, bar(BAR_Q_FULL), G, sp.q_row0, g);
        }
        __syncwarp();
        if (lane == 0) {   // park the epilogue's context
            EpiCtx* cx = (EpiCtx*)(smem + kOffCtx);
            cx->it = locate_item<kStreams>(p, blockIdx.x);
            cx->part_base = sp.part_base; cx->hq = p.hq;
            cx->out = p.out; cx->part_o = p.part_o; cx->part_ml = p.part_ml; cx->part_exp = p.part_exp; cx->lse = p.lse;
            cx->magic = p.row_div_magic; cx->status = p.status;
            const int rc = row0 / kRowsPerCta;
            cx->part_tile = (unsigned char*)p.part_o + (long long)sp.part_base * 512 +
                            (kF32Part ? ((long long)g * sp.nsplit + split) * rows * 512 + row0 * 128
                                      : (((long long)g * sp.row_chunks + rc) * sp.nsplit + split) * 65536);
            mbar_arrive(bar(BAR_CTX));   // (release) the epilogue waits on this before it reads the context
        }
        // what of the fused append is no whole row group (see the end of warp 0): the groups that the block begins and ends in
        if (p.k_new) {
            pdl_wait();
            store_ends(p, sp, g, L, own_lo, own_hi);
        }
        // (the copies must land before the CTA's shared memory goes away, also after a time-out elsewhere)
        if (lane == 0) mbar_drain(bar(BAR_Q_FULL), 0, p.wait_limit_cycles);
    }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;\n" ::"n"(kRegsHigh));
        pdl_wait();
        // ================= softmax + epilogue: one thread per query row =================
        const int x = (warp - 4) >> 2;                       // tile A / B
        const int rt = ((warp & 3) << 5) + lane;             // row in tile == TMEM lane
        const uint32_t lane_addr = (uint32_t)((warp & 3) << 5) << 16;
        const uint32_t tS = tmem_base + lane_addr + kColS;
        const uint32_t tP = tmem_base + lane_addr + kColP + x * 64;
        const uint32_t tO = tmem_base + lane_addr + kColO + x * 128;
        const int q_tile_row0 = row0 + (kStreams ? 0 : x * 128);   // kStreams: both warpgroups hold the same rows
        const int r = q_tile_row0 + rt;
        const int limit = P + min(r / G, q - 1);             // last token this row sees
        const int tile_i_min = min(q_tile_row0 / G, q - 1);
        const bool warp_has_rows = q_tile_row0 + ((warp & 3) << 5) < rows;
        const float sc = p.scale_log2;
        float m_ref = -INFINITY;
        float l_run = 0.f;                                   // running row sum, relative to m_ref
        bool ok = true;
        constexpr int kStep = kStreams ? 2 : 1;
        const int t_first = kStreams ? x : 0;
        if (!warp_has_rows) {   // a warp whose 32 rows are all padding keeps the barriers in step, nothing else
            if (kStreams) {
                uint32_t zero[32];
#pragma unroll
                for (int c = 0; c < 32; ++c) zero[c] = 0;
                tmem_st_x32(tP, zero);
                tmem_st_x32(tP + 32, zero);
                tmem_wait_st();
                tc_fence_before();
            }
            for (int t = t_first; t < n_tiles && ok; t += kStep) {
                const int j = (t - t_first) / kStep;
                ok = mbar_wait(bar(BAR_S_FULL + x), j & 1, abort_flag, p.status, p.wait_limit_cycles);
                if (ok && j > 0) ok = mbar_wait(bar(BAR_P_FREE + x), (j - 1) & 1, abort_flag, p.status, p.wait_limit_cycles);
                __syncwarp();
                if (ok && lane == 0) { mbar_arrive(bar(BAR_S_FREE)); mbar_arrive(bar(BAR_P_READY + x)); mbar_arrive(bar(BAR_P_TAIL + x)); }
            }
        } else
        for (int t = t_first; t < n_tiles; t += kStep) {
            const int j = (t - t_first) / kStep;             // this warpgroup's j-th tile
            ok = mbar_wait(bar(BAR_S_FULL + x), j & 1, abort_flag, p.status, p.wait_limit_cycles);
            if (!ok) break;
            tc_fence_after();
            uint32_t sreg[128];
#pragma unroll
            for (int c4 = 0; c4 < 4; ++c4) tmem_ld_x32(tS + c4 * 32, sreg + c4 * 32);
            tmem_wait_ld();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(BAR_S_FREE));   // (one arrival per warp: 32 on one barrier take turns)
            const int tok0 = kv_begin + t * kBN;
            const bool masked = (tok0 + kBN - 1 > P + tile_i_min) || (tok0 + kBN > kv_end);  // uniform per tile
            float lt0 = 0.f, lt1 = 0.f, lt2 = 0.f, lt3 = 0.f;   // this tile's row sum, four partial sums
            if (masked) {
                const int nvis = max(0, min(min(limit + 1, kv_end) - tok0, kBN));        // visible columns: [0, nvis)
#pragma unroll
                for (int c = 0; c < 128; ++c)
                    if (c >= nvis) sreg[c] = 0xFF800000u;  // -inf: its exponential is exactly 0
            }
            // ---- row maximum (four independent chains of 3-input max).  The exponentials below are taken against the
            //      running reference m_ref (the maximum of earlier tiles, so P may exceed 1); only if this tile's
            //      maximum tops it by more than 2^8 is the reference moved and O rescaled.
            float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
            for (int c = 0; c < 128; c += 8) {
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    mx[k] = max3(mx[k], __uint_as_float(sreg[c + 2 * k]), __uint_as_float(sreg[c + 2 * k + 1]));
            }
            const float m_tile = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])) * sc;
            const bool need = m_tile > m_ref + kRescaleThreshold;
            // P and O of this tile belong to the MMAs of its previous unit until these are done (long since, normally)
            auto wait_p_free = [&]() {
                if (j > 0) ok = mbar_wait(bar(BAR_P_FREE + x), (j - 1) & 1, abort_flag, p.status, p.wait_limit_cycles);
                tc_fence_after();
                return ok;
            };
            if (__any_sync(0xFFFFFFFFu, need)) {
                if (!wait_p_free()) break;
                const float m_new = need ? m_tile : m_ref;
                const float factor = need ? ex2(m_ref - m_new) : 1.f;   // m_ref = -inf gives 0
                if (j > 0) {
                    uint32_t oreg[32];
#pragma unroll
                    for (int c4 = 0; c4 < 4; ++c4) {
                        tmem_ld_x32(tO + c4 * 32, oreg);
                        tmem_wait_ld();
#pragma unroll
                        for (int c = 0; c < 32; ++c) oreg[c] = __float_as_uint(__uint_as_float(oreg[c]) * factor);
                        tmem_st_x32(tO + c4 * 32, oreg);
                    }
                    tmem_wait_st();
                }
                l_run *= factor;
                m_ref = m_new;
            }
            // ---- P = 2^(S * scale - m_ref) as packed bf16 pairs, in place: sreg[c / 2] <- (p[c], p[c + 1]); the
            //      first kPvHeadSteps * 16 columns are stored and handed over before the rest is computed
            const float neg_m = (m_ref == -INFINITY) ? 0.f : -m_ref;
            const uint64_t sc2 = pk2(sc, sc), nm2 = pk2(neg_m, neg_m);
            auto sweep = [&](const int c_lo, const int c_hi) {
#pragma unroll
                for (int c = c_lo; c < c_hi; c += 4) {
                    const uint64_t xa = fma2p(pk2(__uint_as_float(sreg[c]), __uint_as_float(sreg[c + 1])), sc2, nm2);
                    const uint64_t xb = fma2p(pk2(__uint_as_float(sreg[c + 2]), __uint_as_float(sreg[c + 3])), sc2, nm2);
                    float a0, a1, b0, b1;
                    if (((c >> 1) & 7) < kPolyPairsOf8) ex2_poly2(xa, a0, a1);
                    else { upk2(xa, a0, a1); a0 = ex2(a0); a1 = ex2(a1); }
                    if ((((c >> 1) + 1) & 7) < kPolyPairsOf8) ex2_poly2(xb, b0, b1);
                    else { upk2(xb, b0, b1); b0 = ex2(b0); b1 = ex2(b1); }
                    add2(lt0, lt1, a0, a1);
                    add2(lt2, lt3, b0, b1);
                    sreg[c >> 1] = pack_bf16(a0, a1);
                    sreg[(c >> 1) + 1] = pack_bf16(b0, b1);
                }
            };
            constexpr int kHeadCols = kPvHeadSteps * 16;   // 96 score columns = 48 packed registers
            sweep(0, kHeadCols);
            if (!wait_p_free()) break;
            tmem_st_x32(tP, sreg);
            tmem_st_x16(tP + 32, sreg + 32);
            tmem_wait_st();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(BAR_P_READY + x));
            sweep(kHeadCols, 128);
            l_run += (lt0 + lt1) + (lt2 + lt3);
            tmem_st_x16(tP + 48, sreg + 48);
            tmem_wait_st();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(BAR_P_TAIL + x));
        }
        if (kStreams && ok) ok = mbar_wait(bar(BAR_O_FULL), 0, abort_flag, p.status, p.wait_limit_cycles);   // (else waited for in the epilogue)
        if (ok || kStreams) tile_epilogue<kStreams, kF32Part>(smem, tO, m_ref, l_run, ok);
    }
    // ---- teardown
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem_base), "r"(kTmemCols) : "memory");
    }
}

// --------------------------------------------------------------------------------------------
namespace {
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn get_encode_fn() {
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void* ptr = nullptr;
        cudaDriverEntryPointQueryResult qres;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &qres) == cudaSuccess &&
            qres == cudaDriverEntryPointSuccess)
            fn = (EncodeTiledFn)ptr;
    }
    return fn;
}
// View of a pool [num_pages * Hkv * 16 rows][128 dims] bf16 as [row groups of 8][halves of 64 dims][8 rows][64 dims]; a box is two row
// groups = the 4 KB of one page and KV head, or one of them, 128-byte swizzle
bool make_pool_map_impl(CUtensorMap* map, const void* pool, long long num_pages, int hkv, int groups) {
    EncodeTiledFn fn = get_encode_fn();
    if (!fn) return false;
    const cuuint64_t dims[4] = {64, 8, 2, (cuuint64_t)num_pages * hkv * (kPage / 8)};
    const cuuint64_t strides[3] = {(cuuint64_t)kD * 2, 128, (cuuint64_t)kD * 2 * 8};
    const cuuint32_t box[4] = {64, 8, 2, (cuuint32_t)groups};
    const cuuint32_t estr[4] = {1, 1, 1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(pool), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
}  // namespace

bool make_pool_map(CUtensorMap* map, const void* pool, long long num_pages, int hkv) {
    return make_pool_map_impl(map, pool, num_pages, hkv, kPage / 8);
}

// [KV heads][row groups of 8][halves of 64 dims][rows][64 dims]; the row and the row-group dimension overlap (a box of 16 groups from any
// row on), so the bounds of the map do not protect a box of `groups` > 1: its 8 * groups rows have to exist
static bool make_rows_map(CUtensorMap* map, const void* rows, long long total_q, int hkv, int groups) {
    EncodeTiledFn fn = get_encode_fn();
    if (!fn) return false;
    const cuuint64_t row = (cuuint64_t)hkv * kD * 2;
    const cuuint64_t dims[5] = {64, (cuuint64_t)total_q, 2, (cuuint64_t)groups, (cuuint64_t)hkv};
    const cuuint64_t strides[4] = {row, 128, row * 8, (cuuint64_t)kD * 2};
    const cuuint32_t box[5] = {64, 8, 2, (cuuint32_t)groups, 1};
    const cuuint32_t estr[5] = {1, 1, 1, 1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void*>(rows), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
bool make_rows_maps(RowsMaps* m, const void* k_new, const void* v_new, long long total_q, const void* k_pool, const void* v_pool, long long num_pages,
                    int hkv) {
    return make_pool_map_impl(&m->k_pool8, k_pool, num_pages, hkv, 1) && make_pool_map_impl(&m->v_pool8, v_pool, num_pages, hkv, 1) &&
           make_rows_map(&m->k8, k_new, total_q, hkv, 1) && make_rows_map(&m->v8, v_new, total_q, hkv, 1) &&
           make_rows_map(&m->k128, k_new, total_q, hkv, 16) && make_rows_map(&m->v128, v_new, total_q, hkv, 16);
}

// [KV heads][halves of 64 dims][tokens][heads of the group][64 dims]; a box is all heads of q_tokens tokens, or one row
bool make_q_maps(RowsMaps* m, const void* q, long long total_q, int hq, int hkv, int q_tokens) {
    EncodeTiledFn fn = get_encode_fn();
    if (!fn) return false;
    const cuuint32_t G = (cuuint32_t)(hq / hkv);
    const cuuint64_t dims[5] = {64, G, (cuuint64_t)total_q, 2, (cuuint64_t)hkv};
    const cuuint64_t strides[4] = {(cuuint64_t)kD * 2, (cuuint64_t)hq * kD * 2, 128, (cuuint64_t)G * kD * 2};
    const cuuint32_t one[5] = {64, 1, 1, 1, 1}, box[5] = {64, G, (cuuint32_t)q_tokens, 1, 1}, estr[5] = {1, 1, 1, 1, 1};
    auto make = [&](CUtensorMap* map, const cuuint32_t* b) {
        return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void*>(q), dims, strides, b, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                  CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
    };
    m->q_tokens = q_tokens;
    if (q_tokens == 0) memset(&m->q_box, 0, sizeof m->q_box);
    return make(&m->q_row, one) && (q_tokens == 0 || make(&m->q_box, box));
}

namespace {
template <bool kStreams, bool kF32Part>
cudaError_t launch_tile(const AttnParams& p, const CUtensorMap& map_k, const CUtensorMap& map_v, const RowsMaps& maps_new,
                        cudaStream_t stream) {
    // the attribute is per device: remember which devices have it (a process normally drives one GPU)
    static bool configured_on[64] = {false};
    int device = 0;
    if (cudaGetDevice(&device) != cudaSuccess || device < 0 || device >= 64) return cudaErrorInvalidDevice;
    bool& configured = configured_on[device];
    if (!configured) {
        cudaError_t e = cudaFuncSetAttribute(attn_tile_bf16_kernel<kStreams, kF32Part>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBytes);
        if (e != cudaSuccess) return e;
        configured = true;
    }
    return launch_chained(attn_tile_bf16_kernel<kStreams, kF32Part>, dim3(p.num_items), dim3(kThreads), kSmemBytes, stream, p, map_k, map_v, maps_new);
}
}  // namespace

cudaError_t launch_attn_tile_bf16(const AttnParams& p, bool streams, const CUtensorMap& map_k, const CUtensorMap& map_v,
                                  const RowsMaps& maps_new, cudaStream_t stream) {
    if (p.num_items == 0) return cudaSuccess;
    if (streams) return launch_tile<true, false>(p, map_k, map_v, maps_new, stream);
    // (fp32 partials as a case of the same kernel: 512-row prefills 0.8 % slower, for the code at the end of a CTA)
    return p.part_half == PART_F32_TILES ? launch_tile<false, true>(p, map_k, map_v, maps_new, stream) : launch_tile<false, false>(p, map_k, map_v, maps_new, stream);
}

}  // namespace agx

