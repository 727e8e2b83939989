// Host planner: turns the per-sequence lengths of one mixed batch into work items for the
// split-K decode kernel, the combine kernel and the chunked-prefill kernel.
// The batch is the one the paper's decode worker builds from its resident decode sequences plus
// its local prefill queue (Section 5); the planner only partitions work, it does no arithmetic
// on tensor data.
#pragma once
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <vector>

#include "../../include/crossflow_attn.h"

namespace cf {

struct DecodeItem {        // one (decode sequence, KV chunk); the kernel adds the KV-head index
    int32_t seq;
    int32_t q_row;         // packed row of the sequence's single query token
    int32_t kv_begin;      // first visible token of the chunk (multiple of block_size)
    int32_t kv_end;        // one past the last token (== context_len for the last chunk)
    int32_t part_slot;     // partial slot to write, or -1: the only chunk, write `out` directly
    int32_t chunk;         // index of this chunk within its sequence
    int32_t n_chunks;      // chunks of the sequence (its partial slots are part_slot - chunk + [0, n_chunks))
    int32_t kv_lo;         // first visible token of the sequence (left edge of a sliding window; 0 without one):
                           // tokens of this chunk below it are masked (only the first chunk can hold any)
};

// Shared prefix (radix-cache reuse, Section 4.4: a lookup tells how much of a prompt is already resident; agent
// turns share long prefixes): decode sequences of one share group point at the same physical pages for the first
// `shared_len` tokens.  Those pages are streamed once per KV chunk for a whole set of members, whose query heads
// ride along as extra MMA columns; every member gets a partial per shared chunk, merged with the partials of
// its own suffix by the usual split-K merge.
struct SharedDecodeItem {  // one (share group, shared KV chunk, member set); the kernel adds the KV-head index
    int32_t seq;           // the member whose block-table row is read for the shared pages
    int32_t kv_begin;      // whole pages of the shared prefix: [kv_begin, kv_end)
    int32_t kv_end;
    int32_t chunk;         // index of this chunk in every member's chunk list (shared chunks come first)
    int32_t member_first;  // first entry of this set in the member list
    int32_t n_members;     // members in the set (n_members * G <= kSharedColumns)
    int32_t pad[2];
};
struct ShareMember {       // one member of a set
    int32_t q_row;         // packed row of its query token
    int32_t part_first;    // first partial slot of the sequence (its chunk c writes slot part_first + c)
    int32_t pad[2];
};
constexpr int32_t kSharedColumns = 64;      // query-head columns a shared-prefix CTA carries (two 8-wide MMA operands per warp)
constexpr int32_t kSharedMembers = 32;      // and sequences
constexpr int32_t kMinSharedPages = 16;     // shorter shared prefixes are not worth a separate pass

struct CombineItem {       // one decode sequence that was split
    int32_t q_row;
    int32_t part_first;    // its chunks occupy slots [part_first, part_first + n_chunks)
    int32_t n_chunks;
};

// tcgen05 kernel: two q tiles of one KV head (tile 1 may be absent).  A q tile is 128 / G tokens x the G heads of the
// group; for the kernel on pairs of SMs it is 128 tokens of one head.
struct PrefillTcItem {
    int32_t seq;
    int32_t kvh;
    int32_t q_row0[2];     // packed row of each tile's first token
    int32_t row0[2];       // index of that token inside the chunk
    int32_t n_rows[2];     // tokens of the tile; 0 = tile absent
    int32_t head[2];       // first query head of each tile
    // KV split: this item covers KV tiles [j_begin, j_end) (128-token tiles; j_end clamps to the item's
    // own extent).  part_slot[t] >= 0: tile t writes an fp32 partial for row r (token * heads + head) into slot
    // part_slot[t] + r * part_k + part_c instead of the final output.
    int32_t j_begin, j_end;
    int32_t part_slot[2];
    int32_t part_k, part_c;
    int32_t prefix, ctx_len;   // of the sequence (copied here so that a role needs one load per item)
    int32_t page_lo;           // first page of the sequence any row of the item can see (sliding window; 0 without
                               // one): pages below it are neither fetched nor multiplied
    int32_t pad;               // pair items (two CTAs, four q tiles): offset of the second CTA's partial slots from
                               // part_slot[]; 0 otherwise.  80 bytes: five 16-byte words
};
static_assert(sizeof(PrefillTcItem) == 80, "PrefillTcItem is copied as five 16-byte words");

struct PrefillCombineItem { // one KV-split tcgen05 item: merges its part_k partials per row
    int32_t q_row0[2];
    int32_t n_rows[2];     // tokens
    int32_t head[2];       // first head
    int32_t part_slot[2];
    int32_t part_k;
    int32_t pack;          // heads of a tile: row r is token r / pack, head head[t] + r % pack
};

struct PlanConfig {
    int32_t num_sms = 148;
    int32_t decode_waves = 4;         // most CTA waves that the decode chunks are sized for
    int32_t decode_min_chunk_pages = 8;
    int32_t decode_page_quantum = 4;  // chunk lengths are multiples of this many pages (warps per CTA)
    int32_t prefill_sms_mixed = 0;    // > 0: SMs the prefill items are balanced over when the batch also holds decode
                                      // work (spatial launch sequence: the first prefill grid's share); 0: num_sms
    int32_t prefill_force_split = 0;  // >= 2: split every tcgen05 item that many ways (tests); 1: none, and one plan for both launch
                                      // sequences; 0: cost model decides
    int64_t part_bytes = INT64_MAX;   // bytes that the fp32 partials of split sequences and items may take (fixed workspace)
    bool prefill_pair = false;        // plan for the two-CTA kernel where the geometry allows it (head_dim 128, group
                                      // size a multiple of 4): an item carries four heads, the machine has num_sms / 2 slots
};

struct Plan {
    std::vector<int32_t> q_start;     // [S+1] exclusive prefix sum of query_len
    std::vector<int32_t> prefix;      // [S] context_len - query_len (filled by the callers that append)
    std::vector<DecodeItem> decode;   // longest chunk first
    std::vector<CombineItem> combine;
    std::vector<SharedDecodeItem> shared_decode;   // shared-prefix chunks (empty unless the caller described sharing)
    std::vector<ShareMember> share_members;
    std::vector<PrefillTcItem> prefill_tc;   // longest KV extent first (tcgen05 kernel); KV-split items appear part_k times
    std::vector<PrefillCombineItem> prefill_combine;   // one per KV-split item
    int32_t n_pre_slots = 0;          // fp32 partial rows of KV-split prefill items (compact, D floats each)
    int32_t n_part_slots = 0;
    int32_t total_q = 0;
    int32_t n_decode_seqs = 0;
    int32_t n_prefill_seqs = 0;
    bool pair = false;                // prefill_tc items are pair items (four q tiles, two CTAs)
    int32_t front_sms = 0;            // mixed batch of the spatial sequence: SMs that the first prefill grid takes (at most
                                      // cfg.prefill_sms_mixed; fewer when they need no more rounds for items of like length)
};

// Validates geometry (supported head_dim / block_size / group / strides).
cf_status validate_desc(const cf_cache_desc* d);
// Validates lengths against the block-table width; fills q_start/total_q.
cf_status validate_lengths(const cf_cache_desc* d, const int32_t* context_len, const int32_t* query_len,
                           int32_t num_seqs, int32_t max_blocks_per_seq, Plan* plan);
// Decode chunking, shared by build_plan and by the allocation-free entry point (plain loops over the
// caller's arrays: nothing here allocates).  `lc_of(s)` returns the context length of sequence s if it is
// a decode sequence and a negative number otherwise.
//   decode_target_pages: the chunk length (in pages) with the smallest predicted time among those that fill the resident
//     CTA slots exactly one, two, ... `decode_waves` times, a ladder of longer ones, and no split at all, of those whose partials
//     fit the budget: cfg.part_bytes, and the limits of the allocation-free entry point, which plans with this routine (no
//     split needs none).
//   decode_split: near-equal chunks of at most `target` pages, each a multiple of the page quantum.
// The prediction, in microseconds, was fitted to 800 (batch, chunk length) pairs: batches of 2 to 256 sequences of 100 to 20,000
// tokens on all geometries, measured on a B200.  Streaming at full bandwidth (B) and one CTA's way through the longest chunk (g per page)
// add up in the 1.7-norm, 2.5 for a split (partials, ticket, merge; fp8 cache: 3.2), 1.2 for every further eight chunks of a
// sequence (the merge takes eight at a time), 2.2 (fp8: 3.5) for every further wave.  Against chunks of at least 32 pages
// in four waves, decode kernel alone: 40 sequences of 400 tokens, 64 over 8 heads 18.2 -> 14.2 us; 100 of 600 tokens 54 -> 47 us,
// with head_dim 64 31 -> 23 us; 16 of 600 tokens (head_dim 64) 9.3 -> 7.8 us; 64 of 1500 tokens on an fp8 cache 54 -> 47 us;
// 64 of 4000 tokens, which four waves fitted, 167 -> 168 us; all of them 1.06 in the mean.
constexpr int64_t kStaticPartBytes = (16ll << 20) - (128ll << 10);      // partials of the allocation-free entry point
constexpr int32_t kStaticMaxItems = 3584;                              // and its chunks
constexpr int32_t kTargetSeqs = 2048;               // larger batches: whole sequences are chunks enough
// `pages`: scratch of kTargetSeqs floats
template <class LcOf>
inline int64_t decode_target_pages(int32_t num_seqs, LcOf lc_of, int32_t B, int32_t Hq, int32_t Hkv, int32_t D, bool fp8,
                                   const PlanConfig& cfg, float* pages, int64_t extra_pages = 0)
{
    int32_t n = 0;
    int64_t total = extra_pages, longest = 1;           // extra: pages streamed by shared-prefix items
    for (int32_t s = 0; s < num_seqs; ++s) {
        const int64_t lc = lc_of(s);
        if (lc < 0) continue;
        const int64_t pg = (lc + B - 1) / B;
        total += pg;
        longest = pg > longest ? pg : longest;
        if (n < kTargetSeqs) pages[n] = (float)pg;
        ++n;
    }
    const int64_t quantum = cfg.decode_page_quantum > 1 ? cfg.decode_page_quantum : 1;
    const int64_t lo = ((cfg.decode_min_chunk_pages > 1 ? cfg.decode_min_chunk_pages : 1) + quantum - 1) / quantum * quantum;
    const int64_t sms = cfg.num_sms > 1 ? cfg.num_sms : 1;      // those that the grid starts on
    const int64_t slots = sms * (D == 64 || fp8 ? 3 : 2);      // resident CTAs: 64 KB of shared memory each, or 96 KB
    const int32_t waves = cfg.decode_waves > 1 ? cfg.decode_waves : 1;
    auto round_up = [&](int64_t c) { return (c + quantum - 1) / quantum * quantum; };
    const int64_t full = round_up((total * Hkv + 2 * sms * waves - 1) / (2 * sms * waves));      // fills `waves` waves of two CTAs per SM
    const int64_t slot_bytes = (int64_t)Hq * (D + 2) * 4, budget = std::min(cfg.part_bytes, kStaticPartBytes);
    if (n > kTargetSeqs || extra_pages > 0) {
        int64_t c = round_up((total * Hkv + slots * waves - 1) / (slots * waves));
        c = extra_pages > 0 ? (c > 32 ? c : c > lo ? 32 : lo) : (c > lo ? c : lo);
        if (cfg.part_bytes != INT64_MAX) {
            int64_t parts = 0;
            for (int32_t s = 0; s < num_seqs; ++s) {
                const int64_t pg = (lc_of(s) + B - 1) / B;
                if (pg > c) parts += (pg + c - 1) / c;
            }
            if (parts * slot_bytes > cfg.part_bytes) c = std::max(c, std::max<int64_t>(full, 32));
        }
        return c;
    }
    // chunks of all sequences, and of those that have more than one: upper bounds (near-equal chunks are rounded up later, and
    // the slack covers the reciprocal's rounding)
    auto chunks = [&](int64_t c) -> int64_t {
        const float inv = 1.000001f / (float)c, up = (float)(c - 1);
        int32_t sum = 0;
        for (int32_t i = 0; i < n; ++i) sum += (int32_t)((pages[i] + up) * inv + 1e-4f);
        return sum > n ? sum : n;
    };
    auto parts = [&](int64_t c) -> int64_t {
        const float inv = 1.000001f / (float)c, up = (float)(c - 1);
        int32_t sum = 0;
        for (int32_t i = 0; i < n; ++i) {
            const int32_t k = (int32_t)((pages[i] + up) * inv + 1e-4f);
            sum += k > 1 ? k : 0;
        }
        return sum;
    };
    const double page_bytes = 2.0 * B * D * (fp8 ? 1.0 : 2.0), g = fp8 ? 0.15 : D == 64 ? 0.077 : 0.113;
    const double rate = (fp8 ? 6.3e6 : 7.6e6) * (double)sms / 148.0;
    const double bytes_us = std::pow((double)total * Hkv * page_bytes / rate, 1.7);
    double best = 1e30;
    int64_t best_c = std::max(std::max(lo, full), round_up(128));      // for a budget that none of the candidates fits
    // Chunks longer than 192 pages unbalance the end of the grid, except where there is so much to stream that even
    // `decode_waves` waves of two CTAs per SM hold longer ones (`full`): there a chunk's start, its partials and its share of the merge
    // weigh more.  Decode kernel alone, at most 192 pages -> with this limit: 256 ragged sequences around 5000 tokens 759 ->
    // 741 us (64 over 8 heads 771 -> 743, head_dim 64 389 -> 381), 600 around 3000 1553 -> 1533 us, one of 1 M tokens 654 -> 634
    // us (head_dim 64 357 -> 329, fp8 cache 411 -> 367).
    const int64_t hi = std::max(std::max(lo, full), (int64_t)192);
    auto consider = [&](int64_t c) {
        c = round_up(c < lo ? lo : c);
        if (c > hi && c < longest) c = hi / quantum * quantum;
        const int64_t all = chunks(c);
        if (all > kStaticMaxItems && all > n) return;
        if (all * slot_bytes + 256 > budget && parts(c) * slot_bytes + 256 > budget) return;
        const int64_t ctas = all * Hkv, len = c < longest ? c : longest, of_longest = (longest + c - 1) / c;
        // further waves: a whole one for any remainder when the chunks are alike, the remainder's part of one when most
        // are shorter than the longest (they leave their slots early)
        const double w = (double)ctas / (double)slots, alike = (double)total * Hkv / ((double)ctas * (double)len);
        const double more = w > 1.0 ? (w - 1.0) + (std::ceil(w) - w) * alike * alike * alike : 0.0;
        const double t = std::pow(bytes_us + std::pow(g * (double)len, 1.7), 1.0 / 1.7) +
                         (of_longest > 1 ? (fp8 ? 3.2 : 2.5) + 1.2 * (double)((of_longest - 1) / 8) : 0.0) + (fp8 ? 3.5 : 2.2) * more;
        if (t < best - 1e-3) { best = t; best_c = c; }
    };
    for (int32_t k = 1; k <= waves; ++k) {
        // the shortest chunk with at most k waves of CTAs (none when even whole sequences are more)
        int64_t a = lo / quantum, z = round_up(longest > lo ? longest : lo) / quantum;
        if (chunks(z * quantum) * Hkv <= k * slots) {
            while (a < z) {
                const int64_t m = (a + z) / 2;
                if (chunks(m * quantum) * Hkv <= k * slots) z = m; else a = m + 1;
            }
            consider(a * quantum);
            if (k == 1)
                for (int64_t f : {5, 6, 8, 12}) consider(a * quantum * f / 4);
        }
    }
    if (longest > 64)
        for (int64_t c : {32, 64, 96, 128, 160}) consider(c);
    if (full > 192) {
        for (int64_t c : {192, 256, 384, 512, 768, 1024})
            if (c < full) consider(c);
        consider(full);
    }
    if (longest <= hi) consider(longest);
    return best_c;
}
inline void decode_split(int64_t pages, int64_t target, int32_t quantum, int64_t* n_chunks, int64_t* pages_per_chunk)
{
    const int64_t qn = quantum > 1 ? quantum : 1;
    int64_t n = (pages + target - 1) / target;
    if (n < 1) n = 1;
    int64_t per = (pages + n - 1) / n;
    per = (per + qn - 1) / qn * qn;
    if (per < qn) per = qn;
    *n_chunks = (pages + per - 1) / per > 0 ? (pages + per - 1) / per : 1;
    *pages_per_chunk = per;
}

// Full plan (calls validate_lengths).
// share_group / shared_len (both or neither; HOST [num_seqs]): share_group[s] >= 0 names the group of sequence s,
// whose members have identical block-table entries for the first shared_len[s] tokens; < 0: shares nothing.
cf_status build_plan(const cf_cache_desc* d, const int32_t* context_len, const int32_t* query_len,
                     int32_t num_seqs, int32_t max_blocks_per_seq, const PlanConfig& cfg, Plan* plan,
                     const int32_t* share_group = nullptr, const int32_t* shared_len = nullptr);

// The prefill items of a plan for inspection, in launch order: one entry per (rows of a 128-row block, query head, KV range).
// Tiles of packed items that carry consecutive rows of one block over the same KV range are listed as one run of rows; what
// does not fit together - a missing tile, another row, another range - shows as runs of their own.
struct PrefillEntry {
    int32_t seq, q_row, row0, n_rows, head, kvh, j_begin, j_end;
};
std::vector<PrefillEntry> list_prefill(const cf_cache_desc* d, const Plan& plan);

// The plans of consecutive parts of one batch (part i: sequences from seqs[i] on, packed rows from rows[i] on) as one plan of
// the batch: the same items, chunks and KV ranges, so every row has the bits that its part gives it, queued as build_plan
// queues them.
void join_plans(const cf_cache_desc* d, const std::vector<const Plan*>& parts, const std::vector<int32_t>& seqs,
                const std::vector<int64_t>& rows, Plan* plan);

// Predicted device time of one cf_mixed_attention call, in microseconds, from a model fitted to this
// library's measured kernel times on B200 (decode: fixed cost + bytes at the sustained split-K rate;
// prefill: work items scheduled longest-first onto the SMs, each costing a fixed part plus a time per
// 128-token KV tile).  Meant for deriving a lease's compute credit from a latency headroom (Section 4.2).
struct Estimate {
    float us_decode = 0.f, us_combine = 0.f, us_prefill = 0.f;
};
// Spatial launch sequence: how many SMs the first prefill grid takes when a batch holds decode and prefill work
// (0 when either part is absent).  Computed from the lengths alone, before the plan exists, because the planner
// balances the prefill items over this many SMs.  Decode gets what it needs to be done when the prefill is, and no
// more: it saturates HBM from k_sat SMs (about 65 with up to four heads per KV head, about 100 with eight, where the
// MMAs per byte double), so over a call of length T it needs k_sat * t_decode / T of them, taken with a margin of 1.15;
// the share of the prefill grid is clamped to [3/5, 7/8] of the SMs.  t_decode and the prefill work come from constants of
// its own (decode beside prefill, not on its own).  Fitted against sweeps of the share on the bench configurations (within a few per
// cent of the best share on each).
int32_t spatial_front_sms(const cf_cache_desc* d, const int32_t* context_len, const int32_t* query_len, int32_t num_seqs,
                          int32_t num_sms);
Estimate estimate_us(const cf_cache_desc* d, const int32_t* context_len, const int32_t* query_len, const Plan& plan,
                     int32_t num_sms);

}  // namespace cf
