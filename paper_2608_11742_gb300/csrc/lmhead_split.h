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
// Tokens the splits are cut at, by CTA group: one CTA, or a pair. Cut at whole
// tiles, the longest range of V 126,464 over 152 CTAs was four tiles against 3.25
// on average, of V 44,273 two against 1.14: 32 rows, d 4,096 181 -> 172 us; 80 rows of
// V 44,273, d 1,216 47 -> 40.
constexpr int lm_granule(int cta_group) { return cta_group == 1 ? kTileN / 4 : kTileN / 2; }

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

// CTA pairs or single CTAs. A pair shares each unembedding tile, half in each
// CTA: 32 KB per 64-wide slice and CTA instead of 48, from L2 and into shared
// memory. An odd row tile makes a pair with an empty half, which costs as much
// as two tiles: at 3 and 5 row tiles that is more than the pairs save. One row
// tile alone is bound by reading the unembedding. V 126,464, d 4,096, statistics
// only, single against pairs: 200 rows 232 / 189 us, 300 rows 271 / 292, 512 rows
// 338 / 309, 640 rows 442 / 447, 896 rows 605 / 586, 1,152 rows 765 / 734.
// (The packed unembedding's blocks are tensor coordinates in a pair, 32 bits.)
// cap: the most splits the workspace has room for.
inline LmSplit lm_split(int n_row_tiles, int64_t vocab, int64_t packed_blocks, int64_t cap, int sm_count, int pairs) {
    LmSplit s;
    s.pair = (n_row_tiles % 2 == 0 || n_row_tiles >= 7) && pairs >= 1 && packed_blocks <= INT32_MAX;
    s.units = s.pair ? (n_row_tiles + 1) / 2 : n_row_tiles;
    s.granule = lm_granule(s.pair ? 2 : 1);
    s.n_gran = static_cast<int>((vocab + s.granule - 1) / s.granule);
    s.splits = std::max(1, std::min((s.pair ? pairs : sm_count) / s.units, static_cast<int>(cap)));
    s.longest = (s.n_gran + s.splits - 1) / s.splits;
    // As few as keep the longest range as short: more only make merging work (V
    // 40,115, 33 rows, d 3,904: 152 splits 69 us, 126 splits 63).
    s.splits = (s.n_gran + s.longest - 1) / s.longest;
    return s;
}

// First token of a split's range (of the split after it: its end). Whole granules,
// so the last range's end may lie past INT32_MAX.
LMSPLIT_HD inline int64_t lm_range(int split, int n_gran, int splits, int granule) {
    return static_cast<int64_t>(split) * n_gran / splits * granule;
}

}  // namespace rps
