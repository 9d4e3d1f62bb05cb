// lmhead_split.h -- how the LM head's rows and vocabulary are spread over CTAs.
// Plain C++, shared by lmhead.cu and its host test.
#pragma once

#include <algorithm>
#include <climits>
#include <cstdint>

#ifdef __CUDACC__
#define LMSPLIT_HD __host__ __device__
#else
#define LMSPLIT_HD
#endif

namespace rps {

constexpr int kTileM = 128;                 // hidden rows per tile (TMEM lanes)
constexpr int kTileN = 256;                 // tokens per tile (accumulator columns)
constexpr int kMaxSplits = 256;
constexpr int kQuarter = kTileN / 4;        // the smallest part of a tile a split may end at

// CTA pairs a device holds at once, from the occupancy query. A query that fails
// means no pairs: single CTAs need no cluster.
inline int lm_pairs(bool query_ok, int counted) { return query_ok && counted > 0 ? counted : 0; }

struct LmSplit {
    bool pair;    // CTA pairs, or single CTAs
    int units;    // pairs or CTAs per split
    int granule;  // tokens the splits are cut at
    int n_gran;   // granules of the vocabulary
    int splits;
    int longest;  // granules of the longest split
};

// `ctas` single CTAs or pairs at once, at most `cap` splits (the workspace's room).
inline LmSplit lm_cut(bool pair, int n_row_tiles, int granule, int64_t vocab, int64_t cap, int ctas) {
    LmSplit s;
    s.pair = pair;
    s.units = pair ? (n_row_tiles + 1) / 2 : n_row_tiles;
    s.granule = granule;
    s.n_gran = static_cast<int>((vocab + granule - 1) / granule);
    s.splits = std::max(1, std::min(ctas / s.units, static_cast<int>(cap)));
    s.longest = (s.n_gran + s.splits - 1) / s.splits;
    // As few as keep the longest range as short: more only make merging work (V
    // 40,115, 33 rows, d 3,904: 152 splits 69 us, 126 splits 63).
    s.splits = (s.n_gran + s.longest - 1) / s.longest;
    return s;
}

// Single CTAs' splits end at whole tiles or at quarters. Quarters even out the
// ranges: the longest of V 126,464 over 152 CTAs is four tiles against 3.25 (32 rows,
// d 4,096 181 -> 172 us). But a range then starts and ends inside a tile, whose
// copies are narrower and, packed, span two blocks. One row tile, bound by reading
// the unembedding, takes quarters; more take them where they shorten the longest
// range by an eighth (quarters against tiles, nine vocabularies of 8,000 to 151,936, d
// 1,024 to 4,096: 12 % faster at 0.625 of the length, 3 % at 0.81, slower from 0.94 on, by
// up to 15 %: 1,308 rows of V 100,000, d 4,096 825 us, tiles 750).
//
// CTA pairs. A pair shares each unembedding tile, half in each CTA: 32 KB per
// 64-wide slice and CTA instead of 48, from L2 and into shared memory, and a tile
// takes about 0.9 of a single CTA's time. But there are half as many, so that they
// fit the ranges less well; an odd row tile makes a pair with an empty half; and a
// launch of clusters takes longer (0.9 us in a graph, 4 us called directly). So pairs
// take an even number of row tiles whose longest range is at most 1.2 times the
// single CTAs', or an odd one from seven on (1.12, 1.09 below 16 tiles), and longer
// than 32 slices.
// Best single against pairs, statistics only, us: d 4,096, 512 rows of V 126,464 341 /
// 316, of V 8,000 31.8 / 31.1 (d 1,024: 17.4 / 21.0); 384 rows of V 126,464 297 / 332;
// 1,152 rows of V 126,464 (1.06) 815 / 794, of V 20,000 (1.1) 4 % slower, of V 8,000 (1.25)
// 54 / 65; 1,408 rows of V 126,464 (1.09), d 2,048 480 / 449; 896 rows of V 90,000 to 134,348
// (1.12) 3 % faster in pairs.
// (The packed unembedding's blocks are tensor coordinates in a pair, 32 bits.)
inline LmSplit lm_split(int n_row_tiles, int64_t vocab, int kblocks, int64_t cap, int sm_count, int pairs) {
    const LmSplit tiles = lm_cut(false, n_row_tiles, kTileN, vocab, cap, sm_count);
    const LmSplit quarters = lm_cut(false, n_row_tiles, kQuarter, vocab, cap, sm_count);
    const int64_t tiles_long = static_cast<int64_t>(tiles.longest) * kTileN;
    const int64_t quarters_long = static_cast<int64_t>(quarters.longest) * kQuarter;
    const bool cut = n_row_tiles == 1 || 8 * quarters_long <= 7 * tiles_long;
    const bool odd = n_row_tiles % 2 != 0;
    const int64_t n_blocks = (vocab + kTileN - 1) / kTileN * kblocks;
    if (pairs >= 1 && n_blocks <= INT32_MAX && (!odd || n_row_tiles >= 7)) {
        const LmSplit p = lm_cut(true, n_row_tiles, kTileN / 2, vocab, cap, pairs);
        const int64_t pair_long = static_cast<int64_t>(p.longest) * p.granule;
        const int64_t single_long = cut ? quarters_long : tiles_long;
        const int limit = !odd ? 120 : pair_long >= 16 * kTileN ? 112 : 109;
        if (100 * pair_long <= limit * single_long && pair_long * kblocks > 32 * kTileN) return p;
    }
    return cut ? quarters : tiles;
}

// First token of a split's range (of the split after it: its end). Whole granules,
// so the last range's end may lie past INT32_MAX.
LMSPLIT_HD inline int64_t lm_range(int split, int n_gran, int splits, int granule) {
    return static_cast<int64_t>(split) * n_gran / splits * granule;
}

}  // namespace rps
