// How the LM-head passes with soft-max statistics (draft_batch.cuh, draft_few.cuh) are cut.  Host code on plain sizes, so that a
// test without a GPU can go through them.
#pragma once

#include <algorithm>

namespace disco {

constexpr int kDbEpiWarps = 8;
constexpr int kDbFinWarps = 2;
constexpr int kDbBoundSlots = 12;      // words of the shared bound per row

// CTAs that finish rows and do nothing else: a warp for each row.  (us per step, any CTA may finish -> CTAs of their own: one row of
// 32000 x 768 14.7 -> 11.4, 7 rows of 40011 x 768 17.5 -> 14.3, 64 rows of 32000 x 768 17.1 -> 16.7, 126 rows 18.4 -> 18.1, of 49152 x
// 768 24.1 -> 23.2.)
inline int draft_finishers(int sms, int R) {
    constexpr int per_cta = kDbEpiWarps + kDbFinWarps;
    return std::max(1, std::min((R + per_cta - 1) / per_cta, sms / 4));
}

// Pairs of CTAs that share their vocabulary tiles, for passes over MT tiles of 128 hidden rows: where the operands' way from L2 is the
// bound, which takes a long contraction.  kept: the logits are written; stats: no lists of the ten largest.  us, single CTAs ->
// pairs, under continuous load (a few launches in a row differ by as much):
//   an even number of tiles, d = 2048, kept (both heads of a feature extraction), 200 / 450 / 700 / 1000 rows: V = 5000 42 / 54 / 69 /
//   83 -> 43 / 55 / 68 / 83, 17000 77 / 123 / 170 / 220 -> 74 / 116 / 159 / 210, 32000 119 / 208 / 285 / 376 -> 111 / 194 / 260 / 340; not
//   kept: 5000 16.5 / 19.7 / 23.8 / 27.3 -> 17.8 / 20.6 / 25.3 / 28.1, 17000 26.7 / 40.6 / 54.5 / 69.9 -> 26.4 / 40.3 / 53.2 / 67.0, 32000
//   43.5 / 69.8 / 101 / 120 -> 40.7 / 65.7 / 93 / 115;
//   an odd one, where a pair works on a tile of nothing, kept, 600 / 850 rows: 5000 x 2048 63 / 76 -> 66 / 77, 17000 x 2048 153 / 198 -> 149 /
//   197, 32000 x 5120 475 / 645 -> 458 / 600; not kept: 32000 x 2048 88 / 106 -> 92 / 113, x 5120 165 / 228 -> 174 / 236; three tiles lose
//   wherever they are narrower than 49152;
//   narrow heads, 700 / 1000 rows kept: 32000 x 768 182 / 229 -> 187 / 245, x 1024 199 / 252 -> 200 / 260, x 1536 240 / 314 -> 229 / 298, 17000 x
//   1536 142 / 184 -> 145 / 190; statistics only, 1006 rows of 32000 x 1024 169 -> 164, of 17000 x 1024 108 -> 112.
inline bool draft_in_pairs(int V, int d, int MT, bool kept, bool stats, int sms) {
    if (MT < 2 || ((MT + 1) & ~1) > sms) return false;
    const long long head = (long long)V * d;
    if (d < 2048) return kept && MT >= 6 && MT % 2 == 0 && V >= 24000 && d >= (stats ? 1024 : 1536);
    if (MT % 2) return kept && MT >= 5 && head >= 25000000;
    return kept ? MT >= 6 || head >= 16000000 : head >= 32000000;
}

// MT tiles of 128 hidden rows (an even number by pairs of CTAs), CN CTAs (or pairs' halves) for each, TPC tiles of TR vocabulary rows
// for each of those, TRN what the MMA takes.
struct DraftTiling {
    int MT, finishers, CN, TPC, TR, TRN;
    // One tile of hidden rows: CTAs of their own finish the rows, unless the others would need a vocabulary tile more for it, or one
    // that is too large to do without the shared bound.
    static DraftTiling cut(int V, int R, bool kept, bool pair, int sms, int target) {
        DraftTiling t;
        t.MT = (R + 127) / 128;
        if (pair) t.MT = (t.MT + 1) & ~1;
        auto tiles_each = [&](int CN) { return (V + target * CN - 1) / (target * CN); };
        const int without = sms / t.MT, with = t.MT == 1 ? without - draft_finishers(sms, R) : without;
        t.CN = with < 1 || tiles_each(with) > tiles_each(without) || (V > 32 * with && V <= 32 * without) ? without : with;
        t.finishers = without - t.CN;
        t.TPC = std::max(1, tiles_each(t.CN));
        t.TR = (V + t.CN * t.TPC - 1) / (t.CN * t.TPC);
        if (kept) t.TR = (t.TR + 3) & ~3;   // rows of logits are stored 16 bytes at a time
        t.TRN = std::max(16, (t.TR + 15) / 16 * 16);
        return t;
    }
    // One tile of hidden rows: the LM head arrives slower than the tensor pipe works, so the vocabulary tiles are small and the
    // epilogue of one runs under the loads of the next.  More tiles of rows: the rows' tile is loaded again for every
    // vocabulary tile, and that traffic (L2 to shared memory) is the bound, so the vocabulary tiles are the widest.
    // Heads of more than two small tiles for each CTA that there is in the end: three narrow tiles take longer than two wide ones
    // (40 / 64 / 100 / 128 rows of 40000 x 768 20.6 / 20.9 / 21.6 / 22.0 -> 19.1 / 20.0 / 20.8 / 21.9 us; of 32000 x 768, two or one, 15.8 /
    // 16.9 / 17.5 / 18.4 -> 17.6 / 18.7 / 20.2 / 20.0).  Two narrow ones without CTAs for the finishing, for which they are too full, still
    // beat a wide one (37000 x 768 20.7 / 20.9 / 21.6 / 21.9 -> 18.7 / 19.0 / 19.4 / 19.8; 36000 x 512 18.5 -> 17.3 at 100 rows, x 384 16.1 ->
    // 15.5), but for short contractions, whose tile is done before the epilogue (x 256 14.7 -> 16.0).
    static DraftTiling make(int V, int d, int R, bool kept, bool pair, int sms) {
        const DraftTiling narrow = cut(V, R, kept, pair, sms, 128);
        if (R > 128) return cut(V, R, kept, pair, sms, 256);
        if (kept || narrow.TPC < 2 || (narrow.TPC == 2 && (narrow.finishers > 0 || d > 320))) return narrow;
        return cut(V, R, kept, pair, sms, 256);
    }
};

// Steps of a draft phase that one launch takes on, at most `most` (1: none but its own).  A launch costs the head's way through HBM
// and the chain behind it once, and a part per tile of 128 rows: the MMAs, or the epilogue where the contraction is short (us per
// tile, 4000 / 12000 / 32000 / 49152 x 256 1.0 / 1.8 / 4.0 / 5.3, x 768 1.1 / 2.1 / 5.8 / 8.8); a step after the last sequence has stopped
// costs a launch that returns (3 us, 5 with more than 128 rows), and rows of such steps that shared a launch were projected for
// nothing.  So: the number that is the cheapest on average, the longest look-ahead being anything from 1 to sl_max, of those that are
// no dearer than single steps even if every sequence stops at once (a seventh dearer at most on narrow heads: 200 sequences of 32000 x
// 256, all stop after the first / third step of 3, 27 / 54 us step by step, 31 / 31 in one launch).  us per call of the whole iteration with 1 / 2 / 4 / 8 / 16 steps to
// a launch, all stop after the first of 16, 32000 x 768: 64 sequences 91 / 69 / 63 / 65 / 87, 256 sequences 139 / 114 / 116 / - / -; after the
// third, 64 sequences 123 / 89 / 67 / 69 / 91.  1 sequence, 4 steps of 10: 104 -> 78 us.  64 sequences, look-aheads up to 10 of 10: 303 ->
// 200 us; 256 sequences of 49152 x 768, up to 16 of 16: 1710 -> 1555 us.
// Not so many rows that a row has fewer than ten CTAs: with three of its twelve words empty the shared bound bounds nothing (32000 x
// 256, 1536 / 2048 rows, 12 / 9 CTAs to a row: 59 / 119 us).
inline int draft_steps_per_launch(int V, int d, int B, int sl_max, int most, int sms) {
    const double epilogue = 0.6 + 1.05e-4 * V, mma = 256.0 * V * d / 1.1e9, per_tile = std::max(epilogue, mma);   // us
    const double allowed = epilogue > mma ? 1.15 : 1.0;
    const double once = 6.0 + std::max(7.0, 2.0 * V * d / 6.5e6);
    const double idle = B <= 64 ? 3.0 : B <= 128 ? 4.0 : 5.0;
    auto tiles = [&](int k) { return (k * B + 127) / 128; };
    auto cost = [&](int k) { return once + per_tile * tiles(k); };
    int best = 1;
    double least = 0.0;
    for (int k = 1; k <= most; ++k) {
        const int launches = (sl_max + k - 1) / k;
        if (k > 1 && (sms / tiles(k) < kDbBoundSlots - 2 || cost(k) + (launches - 1) * idle > allowed * (cost(1) + (sl_max - 1) * idle)))
            continue;
        double mean = 0.0;
        for (int l = 0; l < launches; ++l) {
            const double lives = 1.0 - (double)l * k / sl_max;
            mean += lives * cost(k) + (1.0 - lives) * idle;
        }
        if (k == 1 || mean < least) best = k, least = mean;
    }
    const int launches = (sl_max + best - 1) / best;
    return (sl_max + launches - 1) / launches;
}

}  // namespace disco
