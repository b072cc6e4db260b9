// How the launchers cut their work: host rules on sizes alone, in plain C++, so that they can be
// checked without a device.
#pragma once
#include <math.h>
#include <stdint.h>

#ifdef __CUDACC__
#define ESTP_RULE __host__ __device__ __forceinline__
#else
#define ESTP_RULE inline
#endif

namespace estp {

ESTP_RULE int64_t div_up(int64_t a, int64_t b) { return (a + b - 1) / b; }

// --------------------------------------------------------------- attention importance items
// Items of one group of a prompt of n tiles, cut into chunks of qc query tiles (importance_plan.cuh).
ESTP_RULE int64_t items_f(int64_t n, int qc) {
    const int64_t a = n / qc, r = n % qc;
    return (int64_t)qc * a * (a + 1) / 2 + r * (a + 1);
}

// Number of chunks of key tile kt of a prompt with nt tiles.
ESTP_RULE int chunks_of(int nt, int kt, int qc) { return (nt - kt + qc - 1) / qc; }

// Tiles of a prompt of mean length: the lengths themselves stay on the device.
inline int64_t mean_tiles(int B, int64_t sumT, int rows) {
    return div_up(B > 0 ? div_up(sumT, B) : 0, rows);
}

// Pairs of query tiles per column-sum item of bf16 inputs (tiles are pairs of `pair` rows): the
// largest of 16, 8, 4 and 2 that still gives about kImpItemsPerSm items an SM.  Longer items cost
// fewer item hand-offs; too few items leave SMs idle at the end of a launch.  One pair per item where
// every SM then has at most one: one prompt of 1000 tokens, 28/4 heads, 33.0 -> 22.8 us, of 2000
// 34.8 -> 25.1, three of 1000 35.0 -> 24.8.  Where one pair makes more items than SMs, two are as
// good or better (fewer partials to add): one prompt of 1000, 16/16 heads, 18.5 for one pair and
// 16.6 for two, of 2300, 28/4 heads, 37.0 and 35.1, of 1500, 32/8 heads, 28.3 and 26.8.
constexpr int kImpItemsPerSm = 16;
inline int imp_pairs(int B, int64_t sumT, int n_groups, int pair, int num_sms) {
    const int64_t lists = (int64_t)B * n_groups, nt = mean_tiles(B, sumT, pair);
    for (int qc = 16; qc >= 2; qc /= 2)
        if (lists * items_f(nt, qc) >= (int64_t)kImpItemsPerSm * num_sms) return qc;
    return lists * items_f(nt, 1) <= num_sms ? 1 : 2;
}

// Chunk slots of the partial column sums, for prompts of up to `longest` tokens.
inline int chunk_slots(int64_t longest, int tile, int qc) { return (int)div_up(div_up(longest, tile), qc); }

// fp32 inputs.  Items per SM below which the split gets finer.  4 prompts of 300 to 1500 tokens, 16
// heads, d 128 (2.5 items of 128 rows per SM): row normalisers 158 us with 128 rows, 171 with 64.
// Column sums at 4 and at 8 items per SM: 164 and 162 us there, 432 and 369 on 32 prompts of 100 to 1000.
constexpr int kFLseItemsPerSm = 2, kFImpItemsPerSm = 8;

inline int f32_rows(int B, int64_t sumT, int n_heads, int num_sms) {
    return (int64_t)B * n_heads * mean_tiles(B, sumT, 128) >= (int64_t)kFLseItemsPerSm * num_sms ? 128 : 64;
}

// Rows of an item's fixed side, query tiles per column-sum item, and whether each head gets
// column-sum items of its own (else a KV group's heads share them).
struct F32Split {
    int rows, qc;
    bool per_head;
};

// Finer splits keep more partial sums (a slot per chunk of query tiles and list of items): they are
// taken while those fit kFPartBytes, or what chunks of 512 queries and one list per KV group would
// take.  Without a limit a batch of many short prompts beside a long one, or a loose bound on their
// length, takes up to 8 x heads per group as much as that.
constexpr int64_t kFPartBytes = 64ll << 20;
inline int64_t f32_part_bytes(const F32Split& s, int64_t sumT, int64_t longest, int n_heads, int n_groups) {
    return 4 * (int64_t)chunk_slots(longest, s.rows, s.qc) * (s.per_head ? n_heads : n_groups) * sumT;
}
inline F32Split f32_split(int B, int64_t sumT, int64_t longest, int n_heads, int n_groups, int num_sms) {
    F32Split s{128, 8, false};
    const int64_t coarse = f32_part_bytes({64, 8, false}, sumT, longest, n_heads, n_groups);
    const int64_t limit = coarse > kFPartBytes ? coarse : kFPartBytes;
    // takes the split t if more items are wanted and it fits
    const auto finer = [&](F32Split t) {
        const int64_t lists = (int64_t)B * (s.per_head ? n_heads : n_groups);
        if (lists * items_f(mean_tiles(B, sumT, s.rows), s.qc) >= (int64_t)kFImpItemsPerSm * num_sms) return false;
        if (f32_part_bytes(t, sumT, longest, n_heads, n_groups) > limit) return false;
        s = t;
        return true;
    };
    finer({s.rows, s.qc, true});
    while (s.qc > 1 && finer({s.rows, s.qc / 2, s.per_head})) {
    }
    finer({64, s.qc, s.per_head});
    return s;
}

// ---------------------------------------------------------------- entropy from hidden states
// n_rb row blocks x S vocabulary splits are dealt round-robin to one CTA an SM.  A split is cut in
// cuts of `gran` units (32 entries), 8 (a whole tile) or 1, and worked off in tiles of kLmTileUnits.
constexpr int kLmTileUnits = 8;

struct LmSplit {
    int64_t S;
    int gran;
};

// Time of an item of u units, in tenths of a full tile's unit.  A tile of r < 8 units loads a box of
// W for each of them beside its box of hidden states, which one thread issues: about 2 + 1.6 r units'
// time (from items of 2 to 10 tiles with S forced; 5 units cost more than a whole tile).
inline int64_t lm_item_cost(int64_t u) {
    const int64_t r = u % kLmTileUnits;
    return 10 * (u - r) + (r ? 20 + 16 * r : 0);
}

// Of the cuts in units and in whole tiles, and of the numbers of splits that give the busiest SM w
// items (the largest S of each, up to 16 items or four times the fewest), the one that is least for
// that SM: its items plus, for each, 1 / kLmPassShare of the vocabulary.  That is what an item costs
// beside its tiles, its share of one more pass of W through L2 (a 40th to a 100th of the vocabulary
// with S forced; from a 40th to an 80th the rule's choices are equally good).  A single row block is cut in units: streaming W is the bound there and the
// shares have to be equal (one row, V 128256: 176.6 us, 180.7 in whole tiles).
// Measured sustained over 37 sizes (129 to 21663 rows, D 896 to 4096, V 5000 to 152064) with 8 to 10
// S each: whole tiles with the rule's S are within 1.8 % of the best S.  A rule that took the first S
// in units whose last round is 97 % full, of at most four times the fewest, left SMs idle or took
// rounds that cost more than they filled: 14848 rows, D 896, V 128256 2374 us for S = 1 against 2123
// for 5; 20000 rows, D 4096, V 8000 1005 against 843; 5888 rows, D 4096, V 128256 3937 for S = 13
// against 3801 for 6.
constexpr int kLmPassShare = 80;

// s_min: at least as many splits as keep the row blocks in flight in L2.
inline LmSplit lm_split(int64_t n_rb, int64_t n_unit, int64_t s_min, int64_t num_sms) {
    const int64_t n_tile = div_up(n_unit, kLmTileUnits);
    LmSplit best{1, 1};
    int64_t best_cost = INT64_MAX;
    for (int gran = n_rb > 1 ? kLmTileUnits : 1; gran >= 1; gran -= kLmTileUnits - 1) {
        const int64_t n = gran > 1 ? n_tile : n_unit;
        const int64_t w0 = div_up(n_rb * (n < s_min ? n : s_min), num_sms);  // items of the busiest SM
        const int64_t w1 = 4 * w0 > 16 ? 4 * w0 : 16;
        for (int64_t w = w0; w <= w1; ++w) {
            const int64_t S = w * num_sms / n_rb < n ? w * num_sms / n_rb : n;
            int64_t cost = div_up(n_rb * S, num_sms) *
                           (lm_item_cost(div_up(n, S) * gran) + 10 * n_unit / kLmPassShare);
            if (gran == 1) cost += cost / 50;  // units only for a gain beyond the model's error
            if (cost < best_cost) {
                best_cost = cost;
                best = LmSplit{S, gran};
            }
            if (S == n) break;
        }
    }
    return best;
}

// ------------------------------------------------------------------------------------ pooling
// Token ranges of the pooling stream, each streamed by one CTA per column slice; `full` ranges
// (full x n_slices CTAs) are one wave.  G ranges of a batch of B prompts take about
// bytes / (G x 54 GB/s) to stream below the memory's rate (one CTA's loads in flight) and G / B slots
// a prompt, 75 ns each, to merge: the sum is least at G^2 = bytes B / kPoolRangeBytes.  One wave
// against this, pooling and head: one prompt of 128 x 1024 fp32 15.4 -> 10.4 us, 300 x 4096 bf16
// 29.8 -> 13.4, 2048 x 3584 29.3 -> 18.3, 8192 x 4096 34.5 -> 26.0.
// CTAs of which an SM holds two (rows of 7 KB and more) are one on each SM or a wave: between the two
// the SMs with two set the pace.  16 prompts of 16 to 100 tokens x 4096 bf16 24.7 us with 177 CTAs,
// 20.7 with 152, 22.9 with 304; 8 x 700 x 4096 26.9 with 303, 22.6 with 152, 24.7 with 304.  (Smaller
// CTAs are limited by their own loads: 16 x 256..2048 x 512 bf16 20.7 us with 281, 25.5 with 152.)  A
// wave that would be five sixths full is filled: 64 x 512 x 512 fp32 18.9 us with 1036, 18.6 with 1216.
// Up to kPoolTokens tokens each have a range of their own, as a second row in one costs more than its
// slot: 16 x 4096 bf16, cold, 18.4 us with 15 ranges or 6, 16.9 with 16.
constexpr double kPoolRangeBytes = 4000.0;
constexpr int64_t kPoolTokens = 16;
inline int64_t pool_ranges(int64_t sumT, int64_t row_bytes, int B, int64_t full, int n_slices, int num_sms) {
    int64_t G = full;
    const double few = sqrt((double)sumT * (double)row_bytes * B / kPoolRangeBytes);
    if (sumT > kPoolTokens && (double)G > few) {
        G = (int64_t)few;
        const int64_t two = 2 * (int64_t)num_sms;
        if (full * n_slices <= two && G * n_slices > num_sms && G * n_slices < two) G = num_sms / n_slices;
        else if (6 * G >= 5 * full) G = full;
    }
    if (G > sumT) G = sumT;
    return G > 1 ? G : 1;  // every range holds >= 1 token
}

// --------------------------------------------------------------------- wide products of the MLP
// First value of rank `rank`'s share of a contraction of n_k values in slices of bk: whole slices,
// as even as they go, so the longest share is one slice longer than the shortest at most.
ESTP_RULE int64_t rank_begin(int64_t n_k, int bk, int rank, int ranks) {
    const int64_t k = div_up(n_k, bk) * rank / ranks * bk;
    return k < n_k ? k : n_k;
}

// Ranks (a power of two up to 8) along the contraction for `tiles` output tiles: as many as keep the
// grid within two blocks an SM and every rank kRankValues values of the contraction.
constexpr int kRankValues = 128;
inline int wide_ranks(int64_t tiles, int64_t n_k, int num_sms) {
    int S = 8;
    while (S > 1 && (tiles * S > 2 * (int64_t)num_sms || n_k / S < kRankValues)) S /= 2;
    return S;
}

}  // namespace estp
