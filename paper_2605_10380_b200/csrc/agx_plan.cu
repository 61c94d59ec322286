#include "agx_plan.cuh"

#include <stdio.h>
#include <stdlib.h>

#include <algorithm>
#include <climits>

namespace agx {

namespace {

constexpr long long kMaxTokens = 0x7FFFFFFFll - 4096;   // of one sequence: rounded up to tiles they still fit an int

inline int ceil_div(int a, int b) { return (int)(((unsigned)a + (unsigned)b - 1u) / (unsigned)b); }   // (of two positive numbers)
inline int round_up(long long v, int m) { return (int)((v + m - 1) / m * m); }

// What a launch of one of the attention kernels costs (us), fitted to sweeps over split lengths and batches (GQA 32/8; worst errors 2-3 us at
// 20-130): CTAs go to the SMs (or to their halves) longest first; a step of `unit` tokens takes per_add + max(per_min, per_busy * A) while
// A CTAs are at work (per_busy: HBM, or the mma.sync rate, shared by all of them), the start and end of the first CTA `base`, those of
// others behind it on an SM `overhead` steps.
struct SplitModel {
    int unit, slots, overhead;
    double base, per_add, per_min, per_busy;
    double merge, merge_mb, merge_mb_beyond_16;   // merge launch, per MB of partials up to 16 (they stay in L2) and beyond
    int part_row_bytes;
    double lean;            // > 0: one-wave launches with few (row, head) pairs leave SMs to their merge kernel, which costs this and 0.2 per MB
    bool in_order;          // up to 16 waves: CTAs dealt out as the grid has them instead of longest first
    double crowd;           // launches of one wave and more: the next call's CTAs find no free SMs to start on (all of it; nothing up to half of the SMs)
    double merge_many;      // a merge of more than four splits
};
// Fitted to 340 launches of one to eight blocks, each in all splits that make sense: the split chosen is 1.0 % slower than the best of them on
// average (with 1.9 us a tile, 2.2 + 0.38 us per MB: 1.4 %).  The grid's order counts where a launch is little more than
// one wave: 152 CTAs dealt out longest first fit 148 SMs as if the short ones were stacked, but the last ones to start are long ones (256 tokens behind
// 3000, 32/8 heads, 5 / 4 splits: 31.1 / 21.7 us a layer; 931 behind 3086, 24/8: 66.7 -> 60.2; 598 behind 5293: 76 -> 68.3; verify blocks with three to
// eight prefills 5 to 10 %).  (Sequences whose K/V exceed 48 MB have the KV head outermost in the grid and are dealt out here like the others: 50 plans that
// the order makes different were 0.2 % slower together with it, single ones 13 % faster to 13 % slower.)
// For one block or two, merge, merge_mb, crowd and merge_many are from 185 lone blocks of 97 to 1500 rows, each in all splits that make sense, with the merge of half
// a warp a pair: the split chosen is 0.75 % slower than the best of them on average (1.5 % with a merge of 1.5 + 0.45 us per MB and neither of the two others;
// 72 drawn blocks whose plans the two make different: 3.3 % faster together, single ones 18 % faster to 11 % slower; 23 drawn batches with one or two prefills
// beside decode and verify blocks 3.5 %, 11 % faster to 1 % slower).  Three and more blocks keep the other constants: with these 50 drawn batches were 1.6 %
// slower together, 10 % faster to 10 % slower.
// It replaced waves x (tiles + 3), which took every CTA of a launch for as long as its longest: 48 decode blocks over 700-6000 tokens 129 ->
// 101 us (no split at all), 400 uncached tokens 15.8 -> 13.3, 4 x (32768, 8) 98 -> 93, a ragged prefill batch 512 -> 473.
SplitModel tile_model(const PlanConfig& c, size_t blocks, bool f32_partials = false) {
    if (f32_partials) return {128, c.sm_count, 3, 6.0, 1.3, 0.17, 0.0047, 1.9, 0.3, 0.3, 520, 0, true, 0, 0};
    if (blocks > 2) return {128, c.sm_count, 3, 6.0, 1.3, 0.17, 0.0047, 1.5, 0.45, 0.3, 264, 0, true, 0, 0};
    return {128, c.sm_count, 3, 6.0, 1.3, 0.17, 0.0047, 1.1, 0.35, 0.3, 264, 0, true, 0.5, 0.4};
}
// (a tile of 64 KB takes 0.85 us and more per SM, 1.25 with more than 32 rows; HBM is busy with about 90 of them.  40 rows over 300 / 450 / 600
// tokens, 40/8 heads, take 9.0 / 9.8 / 10.5 us whole and 10.5 / 10.1 / 9.9 in splits of 256 tokens: the merge behind two tiles costs as much as two)
SplitModel stream_model(const PlanConfig& c, bool wide) {
    return {128, c.sm_count, 7, 7.5, 0, wide ? 1.25 : 0.85, 0.0093, wide ? 2.5 : 4.5, wide ? 0.4 : 0.6, 0.3, 520, wide ? 2.2 : 1.0, false, 0, 0};
}
// warp-MMA kernel with 4-page stages, two CTAs per SM: HBM-bound with one 16-row tile, bounded by its own chain with two (mma.sync)
SplitModel small4_model(const PlanConfig& c, int mt) {
    return {64, 2 * c.sm_count, mt == 1 ? 3 : 2, 4.0, 0, mt == 1 ? 1.1 : 1.6, mt == 1 ? 0.00537 : 0.0055, 3.0, 0.38, 0.3, 520, 0, false, 0, 0};
}

// Steps (of md.unit tokens) per KV split: the candidate with the smallest estimated time, and that time.  A server's lengths change with every
// step, so this is host time of every step; what all candidates share is worked out once, and the CTAs of one that cannot win are not dealt out.
struct SplitChoice {
    int tiles = 0;        // 0: not asked for
    double time = 0;
};
SplitChoice choose_split(const PlanConfig& c, const SplitModel& md, const std::vector<int>& seqs, const int32_t* P, const int32_t* Q, int G,
                         int rows_per_chunk, int min_tiles, long long base_items) {
    const int sms = md.slots, hkv = c.num_kv_heads, kOverhead = md.overhead;
    int max_tiles = 1;
    long long pairs = 0;      // (row, query head)
    bool equal = true;
    struct Seq { int tiles, seen_end; double rows_heads; };
    struct Seen { int tiles; long long n; };   // n (row chunk, KV head) pairs that see this many tiles
    std::vector<Seq> work;
    std::vector<Seen> seen;
    work.reserve(seqs.size());
    seen.reserve(seqs.size());
    for (int s : seqs) {
        const int lt = (P[s] + Q[s] + md.unit - 1) / md.unit;
        equal &= s == seqs[0] || lt == max_tiles;
        pairs += (long long)Q[s] * c.num_q_heads;
        max_tiles = std::max(max_tiles, lt);
        const int chunks = (Q[s] * G + rows_per_chunk - 1) / rows_per_chunk, first = (int)seen.size();
        auto add = [&](int last_row, long long n) {
            const int tiles = (P[s] + std::min(Q[s] - 1, last_row / G) + md.unit) / md.unit;
            if ((int)seen.size() > first && seen.back().tiles == tiles) seen.back().n += n;
            else seen.push_back({tiles, n});
        };
        if (chunks <= 32) {
            for (int rc = 0; rc < chunks; ++rc) add((rc + 1) * rows_per_chunk - 1, hkv);
        } else {   // in 32 groups of chunks with the tiles of the group's last one
            for (int k = 0; k < 32; ++k) {
                const int rc0 = (int)((long long)chunks * k / 32), rc1 = (int)((long long)chunks * (k + 1) / 32);
                add(rc1 * rows_per_chunk - 1, (long long)hkv * (rc1 - rc0));
            }
        }
        work.push_back({lt, (int)seen.size(), (double)Q[s] * c.num_q_heads});
    }
    // calls item(tiles, n) for the CTAs of a candidate
    auto deal = [&](int split_tiles, auto item) {
        int i = 0;
        for (const Seq& w : work) {
            const unsigned ns = ((unsigned)w.tiles + split_tiles - 1) / (unsigned)split_tiles, per = ((unsigned)w.tiles + ns - 1) / ns;
            for (; i < w.seen_end; ++i) {
                const unsigned full = (unsigned)seen[i].tiles / per;
                item(seen[i], (int)per, (int)full, (int)((unsigned)seen[i].tiles - full * per));
            }
        }
    };
    struct Cand { int tiles, longest; double bound, merge; long long sum, count; };   // merge: what follows the last tile, and what the next call waits for
    struct Chunks { long long n; int per, full, rest; };
    std::vector<Cand> cands;
    const int n_max = (int)std::min<long long>((max_tiles + min_tiles - 1) / min_tiles, std::max<long long>(32, 2 * sms / std::max<long long>(base_items, 1)));
    cands.reserve(n_max);
    for (int n = 1, last = 0; n <= n_max; ++n) {
        const int t = std::max(min_tiles, (max_tiles + n - 1) / n);
        if (t == last) continue;
        last = t;
        long long sum = 0, count = 0;
        int longest = 0, ns_max = 1;
        double mb = 0;
        for (const Seq& w : work) {
            const int ns = (w.tiles + t - 1) / t;
            ns_max = std::max(ns_max, ns);
            if (ns > 1) mb += w.rows_heads * ns * md.part_row_bytes * 1e-6;
        }
        deal(t, [&](const Seen& v, int per, int full, int rest) {
            const int starts = full + (rest != 0);
            sum += v.n * (v.tiles + kOverhead * starts);
            count += v.n * starts;
            longest = std::max(longest, full ? per : rest);
        });
        const double load = std::max<double>((double)sum / sms, longest + kOverhead);
        Cand cd;
        cd.tiles = t;
        cd.longest = longest;
        cd.sum = sum;
        cd.count = count;
        cd.merge = mb == 0 ? 0 : md.lean > 0 && count <= sms * 15 / 16 && pairs <= 3 * sms ? md.lean + 0.2 * mb
                   : md.unit == 64 && equal && n <= 16 ? (count <= sms ? 0.5 : 4.0)   // (merged inside clusters)
                   : md.merge + md.merge_mb * std::min(mb, 16.0) + md.merge_mb_beyond_16 * std::max(mb - 16.0, 0.0);
        cd.merge += md.crowd * std::min(1.0, std::max(0.0, (double)(count - sms / 2) / (sms / 2))) + (ns_max > 4 ? md.merge_many : 0.0);
        // (a step takes per_add, and beyond it per_min or what all CTAs at work share of per_busy)
        cd.bound = md.base + cd.merge + (load - kOverhead) * md.per_add +
                   std::max((load - kOverhead) * md.per_min, (sum - (double)kOverhead * std::min<long long>(count, sms)) * md.per_busy);
        cands.push_back(cd);
    }
    std::stable_sort(cands.begin(), cands.end(), [](const Cand& a, const Cand& b) { return a.bound < b.bound; });
    SplitChoice best;
    std::vector<int> load;
    std::vector<long long> of_size;   // CTAs with that many tiles
    std::vector<Chunks> in_order;
    for (const Cand& cd : cands) {
        if (best.tiles && cd.bound >= best.time) break;   // (bounds ascend)
        // load[x]: SMs with x tiles (and starts) so far; a CTA goes to an SM with the least
        load.assign((size_t)(cd.sum / sms) + cd.longest + kOverhead + 2, 0);
        load[0] = sms;
        size_t lo = 0, hi = 0;
        auto place = [&](int size, long long left) {
            while (left > 0) {
                while (load[lo] == 0) ++lo;
                const int k = (int)std::min<long long>(load[lo], left);
                load[lo] -= k;
                load[lo + size + kOverhead] += k;
                hi = std::max(hi, lo + size + kOverhead);
                left -= k;
            }
        };
        if (md.in_order && cd.count <= 16 * sms) {
            in_order.clear();
            deal(cd.tiles, [&](const Seen& v, int per, int full, int rest) { in_order.push_back({v.n, per, full, rest}); });
            size_t first = 0;
            for (const Seq& w : work) {   // a sequence's row chunks last to first, a chunk's splits first to last
                for (size_t at = w.seen_end; at-- > first;) {
                    const Chunks& v = in_order[at];
                    if (v.rest == 0) place(v.per, v.full * v.n);
                    else if (v.full == 0) place(v.rest, v.n);
                    else for (long long left = v.n; left > 0;) {
                        // as many (chunk, head) pairs as the SMs of the least load can take whole go there together, one that they cannot by itself
                        while (load[lo] == 0) ++lo;
                        const int k = (int)std::min<long long>(load[lo] / (v.full + 1), left);
                        load[lo] -= k * (v.full + 1);
                        load[lo + v.per + kOverhead] += k * v.full;
                        load[lo + v.rest + kOverhead] += k;
                        if (k > 0) hi = std::max(hi, lo + v.per + kOverhead);   // (the rest is shorter)
                        left -= k;
                        if (k == 0) { place(v.per, v.full); place(v.rest, 1); --left; }
                    }
                }
                first = w.seen_end;
            }
        } else {
            of_size.assign(cd.longest + 1, 0);
            deal(cd.tiles, [&](const Seen& v, int per, int full, int rest) {
                if (full) of_size[per] += v.n * full;
                of_size[rest] += v.n;   // (of_size[0] is not looked at)
            });
            for (int size = cd.longest; size > 0; --size) place(size, of_size[size]);
        }
        double t = md.base;
        size_t prev = kOverhead;
        int busy = sms;
        for (size_t x = 0; x <= hi; ++x) {
            if (load[x] == 0) continue;
            if (x > prev) { t += (x - prev) * (md.per_add + std::max(md.per_min, md.per_busy * busy)); prev = x; }
            busy -= load[x];
        }
        t += cd.merge;
        if (!best.tiles || t < best.time) best = {cd.tiles, t};
    }
    return best;
}

// Tokens per KV split (a multiple of `unit`) with which the sequences' items are one wave of `target` CTAs, at least about min_split.
int one_wave_split(const PlanConfig& c, const std::vector<int>& seqs, const int32_t* P, const int32_t* Q, int G, int rows_per_chunk, int unit, int min_split,
                   int target, bool shrink) {
    long long work = 0, base = 0;
    auto items_of = [&](int s) { return (long long)c.num_kv_heads * ((Q[s] * G + rows_per_chunk - 1) / rows_per_chunk); };
    for (int s : seqs) { base += items_of(s); work += items_of(s) * (P[s] + Q[s]); }
    const int even = round_up((work + target - 1) / target, unit);
    // (splits only a little shorter than the minimum are taken where they are one wave: they fill more SMs)
    int C = shrink && even < min_split && even * 20 >= min_split * 17 ? even : std::max(min_split, even);
    for (;; C += unit) {
        long long n = 0;
        for (int s : seqs) n += items_of(s) * ceil_div(P[s] + Q[s], C);
        if (n <= std::max<long long>(target, base)) return C;
    }
}

}  // namespace

// Chunks that the accept kernel cuts a row of logits into, a CTA each.
// Rows read 16 bytes a load: one wave of CTAs, as long as every thread has two loads to do.  (Rounded up, the last CTAs were a second wave: rows of 128256 bf16,
// eight CTAs of two loads a thread per SM rounded up / six of four loads rounded down, us: 33 rows 6.3 / 6.0, 64 9.0 / 7.8, 128 12.6 / 10.4, 256 20.1 / 16.5, 300
// 20.8 / 16.8, 445 26.5 / 23.6, 512 33.7 / 31.7, 600 43.8 / 35.4, 800 49.3 / 44.3, 888 52.5 / 48.8.)  More whole rows than a wave holds are cut in two where the last
// wave is half empty or more: 128256 bf16, one chunk / two, 889 rows 49.5 / 44.8, 1000 61.9 / 57.3, 1184 67.4 / 64.4, 2000 109 / 106, but 1500 64.1 / 67.1;
// 32000 f32 889 27.9 / 24.8, 2000 71.3 / 69.9; shorter rows, 32000 bf16, 1000 25.5 / 25.5, 2000 51.1 / 52.2, 3000 84 / 89.
// Other rows, one element a load, wait longer for each and want the CTAs that an SM can hold, rounded up (one wave as above / this, us: 32003 bf16, 256 rows 18.0
// / 14.5, 445 34.7 / 19.1, 600 41.8 / 30.3, 889 39.4 / 34.3; 128257 bf16 300 61.7 / 45.1, 600 113 / 92; 32003 f32 256 17.9 / 14.7, 64 7.2 / 7.4).
int accept_chunks(int sm_count, int total_q, int vocab, int elem_bytes, bool aligned) {
    const int vec = 16 / elem_bytes, rows = std::max(total_q, 1);
    const int max_chunks = (vocab + 256 * vec * 2 - 1) / (256 * vec * 2);
    const int wave = kAcceptCtas * sm_count;
    int want = wave / rows;
    if (!aligned) want = (8 * sm_count + rows - 1) / rows;
    else if (want == 0 && rows % wave * 2 <= wave && (long long)vocab * elem_bytes >= 128000) want = 2;
    want = std::max(1, std::min(want, max_chunks));
    int chunk_elems = (vocab + want - 1) / want;
    chunk_elems = (chunk_elems + vec - 1) / vec * vec;
    return (vocab + chunk_elems - 1) / chunk_elems;
}

PlanConfig plan_config(const agx_config& cfg, int sm_count, int (*max_clusters)(int mt, int kw, int cluster)) {
    auto number = [](const char* name, int otherwise) { const char* v = getenv(name); return v ? atoi(v) : otherwise; };
    PlanConfig c;
    c.num_q_heads = cfg.num_q_heads; c.num_kv_heads = cfg.num_kv_heads; c.head_dim = cfg.head_dim; c.dtype = cfg.dtype;
    c.sm_count = sm_count;
    c.max_clusters = max_clusters;
    c.small_min_split = std::max(64, number("AGX_SMALL_MIN_SPLIT", 256) / 64 * 64);
    c.force_mma_sync = number("AGX_FORCE_MMA_SYNC", 0);
    c.debug_plan = number("AGX_DEBUG_PLAN", 0);
    const int kw = number("AGX_SMALL_KW", 0);
    c.small_kw = kw == 4 || kw == 8 ? kw : 0;
    c.batch_stream_tokens = number("AGX_BATCH_STREAM_TOKENS", -1);   // -1: by the estimates of both kernels
    c.longest_first = number("AGX_LONGEST_FIRST", 1) != 0;
    c.merge_sms = number("AGX_MERGE_SMS", 1) != 0;
    c.cluster_merge = !getenv("AGX_CLUSTER_MERGE") ? 1 : number("AGX_CLUSTER_MERGE", 0) ? 2 : 0;
    c.stream_max_rows = number("AGX_STREAM_MAX_ROWS", 384);
    c.stream_rows_estimated = getenv("AGX_STREAM_MAX_ROWS") == nullptr;
    c.stream_min_tokens = number("AGX_STREAM_MIN_TOKENS", -1);
    return c;
}

agx_status build_plan(const PlanConfig& c, int B, const int32_t* P, const int32_t* Q, int pt_stride, Plan& plan, char* err, size_t err_bytes) {
    auto fail = [&](agx_status code, const char* fmt, auto... args) { snprintf(err, err_bytes, fmt, args...); return code; };
    const int G = c.num_q_heads / c.num_kv_heads;
    std::vector<int> row0(B + 1, 0);
    for (int s = 0; s < B; ++s) {
        if (Q[s] < 1) return fail(AGX_E_INVAL, "q_len[%d] = %d < 1", s, Q[s]);
        if (P[s] < 0) return fail(AGX_E_INVAL, "prefix_len[%d] = %d < 0", s, P[s]);
        if (pt_stride >= 0 && (long long)P[s] + Q[s] > (long long)pt_stride * kPage)
            return fail(AGX_E_RANGE, "sequence %d: %d + %d tokens exceed the page table (%d pages)", s, P[s], Q[s], pt_stride);
        if ((long long)P[s] + Q[s] > kMaxTokens) return fail(AGX_E_RANGE, "sequence %d: %d + %d tokens", s, P[s], Q[s]);
        if ((long long)row0[s] + Q[s] > (1 << 30)) return fail(AGX_E_RANGE, "too many rows");
        row0[s + 1] = row0[s] + Q[s];
    }
    plan.total_rows = row0[B];
    // Blocks of at most 32 rows go to the warp-MMA kernel or to the one-Q-tile tensor-core schedule, all of a batch together: to the one whose
    // estimate is lower (SplitModel; for the small-q kernels with 8-page stages, one CTA per SM, k thousand tokens at 8 KV heads take
    // 4.1 + 0.69 k us up to 16 rows, 5.6 + 0.8 k above in splits that an SM holds whole, max(8.8, 5.8 + 1.06 k) otherwise.  The ground of these
    // lines is narrow: one to eight blocks with 32/8 heads, where one block over 1000-12000 tokens takes up to 0.9 us less or more than they say;
    // other KV head counts only scale k.  7.9: on 148 SMs, from about there two CTAs per SM with 4-page stages are the faster form for several blocks).
    // What it decides against the fixed thresholds it replaces (24576 tokens in all; 7168 / 10240 for one sequence): 32 decode blocks over 1000
    // tokens 38.3 -> 25.3 us, 24 over 2000 54 -> 43, 16 over 4000 48.3 -> 46, one over 20000 20.5 -> 17.5, 32 verify blocks over 1500 53 -> 43;
    // 8 verify blocks over 8000 stay at 50 (55 the other way).
    double small_k = 0;
    int small_rows = 0;
    std::vector<int> small_seqs, wide_seqs;   // up to 32 rows | others that take the schedule in any case
    const bool scalar_path = c.dtype == AGX_F32 || c.head_dim != 128;   // fp32 pools, and bf16 with head_dim 64
    if (!scalar_path)
        for (int s = 0; s < B; ++s) {
            const int rows = Q[s] * G;
            if (rows <= 32) { small_k += (P[s] + Q[s]) * 1e-3 * c.num_kv_heads / 8; small_rows = std::max(small_rows, rows); small_seqs.push_back(s); }
            else if (rows <= c.stream_max_rows) wide_seqs.push_back(s);
        }
    // One block of 65 to 384 rows: the 256-row schedule reads K/V half as often as 128-row chunks do and takes fewer splits, but one KV tile at a
    // time, so that it loses where HBM is the bound.  By the estimates of both, with a margin for what they miss; its partials are fp32 here, as
    // those of the other schedule.  120 such blocks, up to 384 rows over 200 to 16000 tokens: 10 % faster together than all of them in 128-row chunks, single
    // ones up to 5 % slower.  A layer in us: (693, 37) 14.4 -> 9.1, (1687, 70) 19.5 -> 12.6 with 24/8 heads, (2110, 42) 16.7 -> 11.7 with 32/8.
    // (Batches: gains and losses of 20 %, which the estimates do not tell apart.  One query head per KV head: not measured.)
    bool wide_tiles = false;
    SplitChoice tile_choice, stream_choice, small_choice[2];   // splits that the estimates were made with, where they were
    if (c.stream_rows_estimated && B == 1 && wide_seqs.size() == 1 && Q[0] * G > kSmallRowsMax && G > 1 && !c.force_mma_sync) {
        auto estimate = [&](const SplitModel& md, int chunk, int min_tiles) {
            return choose_split(c, md, wide_seqs, P, Q, G, chunk, min_tiles, (long long)c.num_kv_heads * ((Q[0] * G + chunk - 1) / chunk));
        };
        tile_choice = estimate(tile_model(c, 1, true), 256, 1);
        stream_choice = estimate(stream_model(c, true), 128, 2);
        wide_tiles = tile_choice.time < (Q[0] * G <= 128 ? 0.86 : 0.89) * stream_choice.time;
        if (c.debug_plan) fprintf(stderr, "agx plan: %d rows, 256-row schedule %.1f us, 128-row chunks %.1f us\n", Q[0] * G, tile_choice.time, stream_choice.time);
    }
    bool batch_streams = false;
    if (!small_seqs.empty()) {
        if (c.batch_stream_tokens >= 0) {
            batch_streams = small_seqs.size() >= 2 && small_k * 1e3 >= c.batch_stream_tokens;
        } else if (c.stream_min_tokens < 0) {
            auto estimate = [&](const SplitModel& md, int chunk, const std::vector<int>& seqs) {
                long long items = 0;
                for (int s : seqs) items += (long long)c.num_kv_heads * ((Q[s] * G + chunk - 1) / chunk);
                return seqs.empty() ? SplitChoice() : choose_split(c, md, seqs, P, Q, G, chunk, md.unit == 64 ? 4 : 2, items);
            };
            const bool one = small_seqs.size() == 1;
            double warp_mma;
            std::vector<int> mt1, mt2;
            for (int s : small_seqs) (Q[s] * G <= 16 ? mt1 : mt2).push_back(s);
            if (one || small_k < 7.9) {
                const bool whole = mt2.empty() || one_wave_split(c, mt2, P, Q, G, 32, 16, c.small_min_split, c.sm_count, true) <= kSwapMaxTokens;
                warp_mma = small_rows <= 16 ? 4.1 + 0.69 * small_k : whole ? 5.6 + 0.8 * small_k : std::max(8.8, 5.8 + 1.06 * small_k);
            } else {
                small_choice[0] = estimate(small4_model(c, 1), 16, mt1);
                small_choice[1] = estimate(small4_model(c, 2), 32, mt2);
                warp_mma = small_choice[0].time + small_choice[1].time;
            }
            std::vector<int> all = wide_seqs;
            all.insert(all.end(), small_seqs.begin(), small_seqs.end());
            // (with one 16-row tile the warp-MMA kernel was never more than 2 % slower than the schedule in the sweeps of equal and ragged decode
            // batches behind the models, though its estimate is up to 15 % higher there: 0.87 takes that out)
            if (!one && small_k >= 7.9 && small_rows <= 16) warp_mma *= 0.87;
            const SplitModel sm = stream_model(c, !wide_seqs.empty());
            if (!wide_seqs.empty() || warp_mma > sm.base) {   // (no launch of the schedule is estimated below its base)
                const SplitChoice together = estimate(sm, 128, all), wide = estimate(sm, 128, wide_seqs);
                batch_streams = together.time < warp_mma + wide.time;
                stream_choice = batch_streams ? together : wide;
            }
        }
    }
    long long warp_mma_tokens = 0;
    int warp_mma_seqs = 0;
    std::vector<int> groups[KIND_COUNT];
    for (int s = 0; s < B; ++s) {
        Kind k;
        if (scalar_path) k = KIND_SIMT;
        else {
            const int rows = Q[s] * G;
            const bool tile_ok = !c.force_mma_sync;
            // up to 128 rows: one Q tile per CTA, KV tiles alternating between two softmax warpgroups (HBM-bound
            // streaming on the tcgen05 pipe); blocks of at most 32 rows over short contexts stay with the warp-MMA
            // kernel, whose fixed costs are lower (none above 32 rows)
            // (with the batch rule forced the estimates are not asked, and a sequence of its own keeps the cross-over between the two kernels)
            const int cross = c.stream_min_tokens >= 0 ? c.stream_min_tokens : c.batch_stream_tokens < 0 ? INT_MAX : rows > 8 ? 7168 : 10240;
            const bool forced = P[s] + Q[s] >= cross;
            if (wide_tiles) k = KIND_TILE;
            else if (tile_ok && rows <= c.stream_max_rows && (rows > 32 || batch_streams || forced)) k = KIND_STREAM;
            else if (rows <= 16) k = KIND_SMALL1;
            else if (rows <= 32) k = KIND_SMALL2;
            else if (rows <= kSmallRowsMax || c.force_mma_sync) k = KIND_SMALL4;
            else k = KIND_TILE;
            if (k == KIND_SMALL1 || k == KIND_SMALL2) { warp_mma_tokens += P[s] + Q[s]; ++warp_mma_seqs; }
        }
        groups[k].push_back(s);
    }
    const int small_kw = c.small_kw ? c.small_kw : (warp_mma_seqs >= 2 && warp_mma_tokens * c.num_kv_heads / 8 >= 7900) ? 4 : 8;
    // Work items are handed to the SMs in launch order: the sequences with the longest contexts go first, so that the
    // longest items of a ragged batch are not the ones left over for the last wave (env AGX_LONGEST_FIRST=0 keeps the batch order).
    if (c.longest_first)
        for (int k = 0; k < KIND_COUNT; ++k)
            std::stable_sort(groups[k].begin(), groups[k].end(), [&](int a, int b) { return P[a] + Q[a] > P[b] + Q[b]; });
    for (int k = 0; k < KIND_COUNT; ++k) {
        const std::vector<int>& seqs = groups[k];
        if (seqs.empty()) continue;
        // ---- choose the split length C (tokens) so that one wave of CTAs covers the group
        int unit, min_split, target;
        long long base_items = 0;  // items per split, summed over sequences
        std::vector<long long> per_seq_items(seqs.size());
        if (k == KIND_SIMT) { unit = 64; min_split = 64; target = c.sm_count * 2; }
        else if (k == KIND_TILE || k == KIND_STREAM) { unit = 128; min_split = k == KIND_TILE ? 128 : 256; target = c.sm_count; }
        else { unit = 16; min_split = c.small_min_split; target = c.sm_count; }
        const int rows_per_chunk = (k == KIND_SIMT) ? 8 : (k == KIND_SMALL1) ? 16 : (k == KIND_SMALL2) ? 32 : (k == KIND_SMALL4) ? 64 : (k == KIND_STREAM) ? 128 : 256;
        for (size_t n = 0; n < seqs.size(); ++n) {
            const int s = seqs[n];
            const long long items = (long long)c.num_kv_heads * ((Q[s] * G + rows_per_chunk - 1) / rows_per_chunk);
            per_seq_items[n] = items;
            base_items += items;
        }
        const bool small_kind = k == KIND_SMALL1 || k == KIND_SMALL2;
        int C = min_split, kw = k == KIND_SMALL4 ? 4 : small_kw;
        if (k != KIND_TILE && k != KIND_STREAM && !(small_kind && kw == 4)) {
            C = one_wave_split(c, seqs, P, Q, G, rows_per_chunk, unit, min_split, target, k != KIND_SIMT);
            // fp32-arithmetic kernel: a CTA's tiles are a chain of 2.5-8 us each, so that where one wave would take chains of more than eight, several
            // waves of four are faster (32/8 heads, fp32, d 128 / 64: one row over 20000 + 30 x 40 tokens 364 -> 107 / 200 -> 62 us, 6 x 8000
            // 330 -> 201 / 185 -> 113; in chains of eight 16 x 1000 74 / 41 us, of four 79 / 45)
            if (k == KIND_SIMT && C > 512) C = std::min(C, one_wave_split(c, seqs, P, Q, G, rows_per_chunk, unit, 256, 16 * c.sm_count, false));
            // several verify blocks whose splits no SM holds whole: two CTAs per SM with 4-page stages where the lengths are alike (7 x 1000
            // tokens 14.3 -> 12.3 us, 8 x 900 14.3 -> 11.8, 2 x 3500 12.5 -> 11.4, 3700 + 3900 12.7 -> 12.3; but 1500 + 2500 + 3500 12.9 -> 13.4.
            // Up to 16 rows: 7 x 1000 10.7 / 11.4, 8 x 900 10.8 / 10.2)
            int longest = 0, shortest = INT_MAX;
            for (int s : seqs) { longest = std::max(longest, P[s] + Q[s]); shortest = std::min(shortest, P[s] + Q[s]); }
            if (k == KIND_SMALL2 && seqs.size() >= 2 && C > kSwapMaxTokens && longest < 2 * shortest && !c.small_kw) kw = 4;
        }
        // one CTA per SM that holds its split whole (agx_attn_swap.cu)
        const bool whole = small_kind && kw == 8 && C <= kSwapMaxTokens;
        auto count_items = [&](int c_tokens) {
            long long items = 0;
            for (size_t n = 0; n < seqs.size(); ++n) {
                const int L = P[seqs[n]] + Q[seqs[n]];
                items += per_seq_items[n] * ceil_div(L, c_tokens);
            }
            return items;
        };
        if (k == KIND_TILE || k == KIND_STREAM) {
            int max_len = 0;
            for (int s : seqs) max_len = std::max(max_len, P[s] + Q[s]);
            SplitChoice choice = k == KIND_STREAM ? stream_choice : tile_choice;
            if (!choice.tiles) {
                const bool wide = std::any_of(seqs.begin(), seqs.end(), [&](int s) { return Q[s] * G > 32; });
                choice = choose_split(c, k == KIND_STREAM ? stream_model(c, wide) : tile_model(c, seqs.size()), seqs, P, Q, G, rows_per_chunk, min_split / unit, base_items);
            }
            C = unit * choice.tiles;
            if (const char* force = getenv("AGX_TILE_SPLIT_TOKENS")) { if (atoi(force) >= unit) C = atoi(force) / unit * unit; }
            if (c.debug_plan)
                fprintf(stderr, "agx plan: tile kernel, %lld row chunks, longest sequence %d tokens -> KV splits of %d tokens, %lld CTAs\n",
                        base_items, max_len, C, count_items(C));
        } else if (small_kind && kw == 4) {
            const SplitModel md = small4_model(c, k == KIND_SMALL1 ? 1 : 2);
            const int least = std::max(1, min_split / md.unit);
            const SplitChoice& known = small_choice[k == KIND_SMALL1 ? 0 : 1];
            C = md.unit * (known.tiles && least == 4 ? known : choose_split(c, md, seqs, P, Q, G, rows_per_chunk, least, base_items)).tiles;
            // One wave: the shortest splits that are one, in pages instead of the model's steps of four (4 x (2500, 1) 12.2 -> 11.0 us, 6 x (2500, 4)
            // 16.4 -> 14.7, 4 x (2500, 8) 15.0 -> 13.2, 4650 + 4650 11.4 -> 11.1).
            bool splits = false;
            for (int s : seqs) splits |= P[s] + Q[s] > C;
            if (splits && count_items(C) <= md.slots) C = std::min(C, one_wave_split(c, seqs, P, Q, G, rows_per_chunk, unit, min_split, md.slots, true));
        }
        // ---- small-q kernel: when every sequence has one row chunk and the same number of KV splits (2..16), the
        //      splits of a (sequence, KV head) form a thread-block cluster and are merged through distributed shared
        //      memory: no partials in global memory, no combine launch.  17..20 splits are squeezed into 16.
        //      Not where a CTA holds its split whole: a CTA that waits for its cluster keeps an SM from the next call, whose K/V then come late
        //      (8 rows over 300 / 700 / 2000 tokens 8.3 / 8.7 / 7.2 us, through memory 6.9 / 7.1 / 6.3; 4 x 500 7.8 / 6.4; one row over 3 x 700
        //      5.9 / 5.0).  One block of one row or two keeps the clusters: as fast, and a launch fewer for the host (6.0 / 6.2 us a call).
        int cluster = 0;
        bool memory_merge = false;   // (fp32 partials, as the clusters' are)
        if ((small_kind || k == KIND_SMALL4) && c.cluster_merge && seqs.size() <= (size_t)kMaxSeqs) {
            int common = -1;
            bool ok = true;
            for (size_t n = 0; n < seqs.size() && ok; ++n) {
                const int L = P[seqs[n]] + Q[seqs[n]];
                int ns = ceil_div(L, C);
                ns = ceil_div(L, round_up(ceil_div(L, ns), unit));
                if (ns > 16 && ns <= 20) ns = 16;
                ok = per_seq_items[n] == c.num_kv_heads && (common < 0 || ns == common);
                common = ns;
            }
            if (ok && common >= 2 && common <= 16) {
                const int mt = k == KIND_SMALL1 ? 1 : k == KIND_SMALL2 ? 2 : 4;
                const int fit = c.max_clusters(mt, kw, common);
                if (fit >= base_items) {
                    memory_merge = whole && !(seqs.size() == 1 && Q[seqs[0]] <= 2) && c.cluster_merge != 2;
                    if (!memory_merge) cluster = common;
                }
                if (c.debug_plan) fprintf(stderr, "agx plan: clusters of %d: %d fit the device, %lld needed\n", common, fit, base_items);
            }
        }
        // One block in splits that an SM holds whole: as long as two or three KV tiles allow, and the last one a tile shorter than the others, since its
        // CTA also puts the block's own pages together by hand.  At most 16 of them, with fp32 partials; two tiles up to 12 splits at 8 KV heads, where the
        // launch leaves SMs to the next one's CTAs.  32/8 heads, a layer, equal splits / these: 8 rows over 700 tokens 7.2 / 6.6 us, 1550 7.1 / 6.6, 2750
        // 7.7 / 7.2, 3500 9.2 / 7.8, 4096 8.3 / 8.1, 5100 11.0 / 9.0; one row over 4096 6.6 / 6.4, 5100 8.0 / 6.8.  (Up to 16 rows over 3100 to 3840
        // tokens 15 equal splits of two tiles are faster: three rows over 3660 6.4 / 7.3.  From 17 splits of three tiles on nothing is gained.
        // Up to 256 tokens are one CTA's, without a merge: one row over 160 / 200 / 250 tokens 3.9 / 4.0 / 4.0 us, in two splits 5.6; 8 rows 5.3 / 6.0.)
        bool last_shorter = false;
        if (whole && !cluster && seqs.size() == 1 && c.merge_sms) {
            const int L = P[seqs[0]] + Q[seqs[0]], twos = ceil_div(L, 256) * c.num_kv_heads, tiles = twos * 10 <= c.sm_count * 7 ? 2 : 3;
            const bool equal_twos = tiles == 3 && k == KIND_SMALL1 && twos * 6 <= c.sm_count * 5, is_split = L > C;
            for (int t = tiles * 128; t > tiles * 128 - 128 && !last_shorter && !equal_twos && is_split; t -= unit) {
                const int n = ceil_div(L, t);
                if (n < 2 || n > 16 || n * c.num_kv_heads > c.sm_count || L - (n - 1) * t > (tiles - 1) * 128) continue;
                C = t;
                last_shorter = memory_merge = true;
            }
        }
        // One block over more than 16 such splits: 16 or fewer, of 320 tokens or more, are faster than 17 to 24 with SMs left to
        // the merge (of fp16 rows when this was measured; 32/8 heads, 8 rows over 4096 / 4400 / 6000 tokens 8.05 -> 7.66 / 9.43 -> 7.89 / 10.07 -> 9.32 us, one row
        // 6.14 -> 5.91 over 4096, 7.82 -> 7.36 over 6000); not for few rows on a third of the SMs (16/2, one row over 6000 5.71 -> 5.96).  (All of it from 14 shapes.)
        if (whole && !cluster && !memory_merge && seqs.size() == 1 && c.merge_sms && (k == KIND_SMALL2 || count_items(C) * 2 > c.sm_count)) {
            const int L = P[seqs[0]] + Q[seqs[0]], longer = std::max(320, round_up((L + 15) / 16, unit));
            if (ceil_div(L, C) > 16 && longer <= kSwapMaxTokens) { C = std::max(C, longer); memory_merge = true; }
        }
        // ---- fp32-arithmetic kernel: up to 16 splits of an item form a cluster, as many for all sequences; more leave partials
        if (k == KIND_SIMT && c.cluster_merge) {
            int max_len = 0;
            for (int s : seqs) max_len = std::max(max_len, P[s] + Q[s]);
            const int ns = ceil_div(max_len, C);
            if (ns <= 16) {
                cluster = ns;
                C = round_up(ceil_div(max_len, ns), kPage);
            }
        }
        // ---- small-q kernel, one wave of one CTA per SM, splits merged by the merge kernel: leave that kernel SMs of its own.
        //      An attention CTA takes a whole SM, so merge CTAs that find no free SM sit on SMs the next call's attention CTAs
        //      need, and those CTAs then start (and fetch their K/V) only after the merge instead of under it.  With a few SMs
        //      left out of the attention grid the merge CTAs are resident there from the start and the next call's grid
        //      follows this one without a gap.  24 (row, head) pairs an SM, 16 with more than 20 splits.  More of them fit, but what the merge leaves is where
        //      the next call's CTAs start (counted as 96 and 64 pairs, up to 8 splits, 70 batches of one to eight blocks whose plans that changes: 2.9 % slower
        //      together, 9 % faster to 15 % slower; 4 verify blocks 7.7 -> 8.9 us, five of 800 to 2700 tokens 14.5 -> 16.6).
        bool lean_merge = false;
        const bool small_one_per_sm = k == KIND_SMALL4 || (small_kind && kw == 8);
        // (the one-Q-tile tensor-core schedule as well: a single long sequence is one wave of whole-SM CTAs too)
        if (!cluster && !memory_merge && (small_one_per_sm || k == KIND_STREAM) && seqs.size() <= (size_t)kMaxSeqs && c.merge_sms) {
            long long pairs = 0;
            for (int s : seqs) pairs += (long long)Q[s] * c.num_q_heads;
            for (;;) {
                const long long items = count_items(C);
                int ns_max = 1;
                for (int s : seqs) ns_max = std::max(ns_max, ceil_div(P[s] + Q[s], C));
                if (ns_max == 1 || items > c.sm_count) break;   // no merge, or more than one wave anyway
                const long long reserve = (pairs + (ns_max <= 20 ? 24 : 16) - 1) / (ns_max <= 20 ? 24 : 16);
                if (reserve > c.sm_count / 8) break;   // a merge that large needs the whole device anyway
                lean_merge = true;
                if (items <= c.sm_count - reserve || items <= base_items) break;
                if (whole && C + unit > kSwapMaxTokens) break;   // (6 x 1000 tokens, one row, 10.1 -> 8.1 us; 8 rows over 6700 12.7 -> 11.5)
                C += unit;
            }
        }
        // ---- emit launches of at most kMaxSeqs sequences
        for (size_t a = 0; a < seqs.size(); a += kMaxSeqs) {
            Launch ln;
            ln.kind = (Kind)k;
            plan.tensor_core |= k == KIND_TILE || k == KIND_STREAM;
            ln.total_rows = 0;
            ln.num_items = 0;
            ln.cluster = cluster;
            ln.lean_merge = lean_merge;
            ln.f32_partials = wide_tiles;
            ln.kw = kw;
            for (size_t n = a; n < std::min(seqs.size(), a + kMaxSeqs); ++n) {
                const int s = seqs[n];
                const int L = P[s] + Q[s];
                SeqPlan sp;
                sp.prefix_len = P[s];
                sp.q_len = Q[s];
                sp.q_row0 = row0[s];
                sp.seq_index = s;
                sp.nsplit = ceil_div(L, C);
                sp.split_tokens = last_shorter ? C : round_up(ceil_div(L, sp.nsplit), unit);
                sp.nsplit = ceil_div(L, sp.split_tokens);
                if (cluster) { sp.nsplit = cluster; sp.split_tokens = round_up(ceil_div(L, cluster), kPage); }
                sp.row_chunks = (Q[s] * G + rows_per_chunk - 1) / rows_per_chunk;
                // Row chunks of one KV head side by side share its K/V tiles through L2 (a whole long-context sequence does not fit
                // there); where the sequence's K/V fits with room to spare, all heads' longest chunks go first instead, so that the
                // short chunks of a causal block fill the last wave (3584 uncached tokens 114.7 -> 89.5 us, 2 x 1200 50.0 -> 43.0).
                sp.chunk_major = (long long)L * c.num_kv_heads * c.head_dim * 4 <= (48ll << 20);
                sp.item0 = ln.num_items;
                sp.part_base = 0;
                if (sp.nsplit > 1 && !cluster) {
                    long long entries = (long long)Q[s] * c.num_q_heads * sp.nsplit;
                    // (a tile of fp16 partials is 128 slots: more than the slots of its rows only where one chunk has fewer than 128 of them)
                    if (k == KIND_TILE && !wide_tiles) entries = std::max(entries, per_seq_items[n] * sp.nsplit * 128);
                    if (plan.part_entries + entries > 0x7FFFFFFFll) return fail(AGX_E_RANGE, "split partials exceed 2^31 entries");
                    sp.part_base = (int)plan.part_entries;
                    plan.part_entries += entries;
                    plan.any_split = true;
                }
                const long long items = per_seq_items[n] * sp.nsplit;
                if (ln.num_items + items > 0x7FFFFFFFll) return fail(AGX_E_RANGE, "too many work items");
                ln.num_items += (int)items;
                ln.total_rows += Q[s];
                ln.seqs.push_back(sp);
            }
            if (c.debug_plan && k != KIND_TILE && k != KIND_STREAM)
                fprintf(stderr, "agx plan: kind %d (stages of %d pages), %zu sequences, %d CTAs, first sequence %d splits of %d tokens%s\n", k,
                        ln.kw, ln.seqs.size(), ln.num_items, ln.seqs[0].nsplit, ln.seqs[0].split_tokens,
                        cluster ? ", merged in clusters" : "");
            plan.launches.push_back(std::move(ln));
        }
    }
    return AGX_OK;
}

}  // namespace agx
