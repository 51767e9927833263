// Plan of the decode tiles (umma_linear.cu) and the border between them and the CTA pairs (pair_linear.cu): plain host arithmetic,
// no CUDA, so that it can be checked over every size.
#pragma once
#include <cstdint>

namespace dps {
namespace tile_plan {

constexpr int kTileRows = 128;   // weight rows per CTA (UMMA M)
constexpr int kMaxSplit = 8;     // portable cluster size

// K split for a launch of `tiles` output tiles.  capacity[s] = CTAs that can be resident at once
// when launched as clusters of s (clusters must fit inside one GPC, so this is not a multiple of
// the SM count).  Measured on B200: a second wave costs more than it buys, so take the largest
// factor (<= 8, a portable cluster) whose CTAs are all resident at once, keeping at least min_kb K
// blocks per CTA: 4 in fast mode, 5 in full mode (4096 x 4096 at 32-64 tokens in full mode: 6 CTAs per
// tile are 3-5 % faster than 8 with 4 blocks each, alone and inside the decode graphs; in fast mode they
// are as fast alone and 4 % slower inside the graphs).
inline int choose_split(int64_t tiles, int total_kb, const int* capacity, int min_kb) {
    int best = 1;
    for (int s = 2; s <= kMaxSplit; ++s) {
        if (total_kb / s < min_kb) break;
        if (tiles * s <= capacity[s]) best = s;
    }
    return best;
}

// A launch in turns: `rounds` times over the chip, a `split`-th of K each time.
struct Turns {
    int64_t rounds;
    int split;
};
inline Turns turns(int64_t tiles, int split, int at_once) {   // at_once: tiles at work together where K is not split
    return {split > 1 ? 1 : (tiles + at_once - 1) / at_once, split};
}

// 33-64 tokens, long K: whether CTA pairs are the faster ones.  A turn of the tiles is 256 rows per SM (two CTAs), one of the pairs 128,
// so one of the tiles counts for two.  Where K is long the pairs' fixed costs, which exceed the tiles', are small and a pair streams
// faster: with equal turns it wins while one round does (a last, partial wave of tiles leaves SMs with one CTA, which is faster by itself;
// a last round of pairs is a whole one), beyond that with fewer.
// Pairs / tiles at K = 16384, 64 tokens, fast | full, by 256-row tiles: 18-22 0.95-0.98 | 0.99-1.00 (split 3 and 6), 23-26 1.04-1.05 |
// 1.06-1.07 (2 and 6 or 5), 27-33 0.92-0.94 | 0.96-0.99 (2 and 4), 34-45 1.11-1.37 | 1.11-1.28 (1 and 4 or 3), 46-74 0.86-0.91 | 0.88-0.96
// (1 and 2), 75-148 1.15-1.01 | 1.02-0.99 (two rounds, one wave), 149-222 0.90-0.92 | 0.87-0.90 (three, two), 223-296 1.02-0.99 |
// 1.00-0.97 (four, two), 297-370 0.94-0.96 | 0.93-0.96; with K = 22016, 28672 and 53248 the same pattern, the gains two to ten per cent larger.
inline bool pairs_for_long_k(Turns pairs, Turns tiles) {
    const int64_t mine = pairs.rounds * tiles.split, theirs = 2 * tiles.rounds * pairs.split;
    return pairs.rounds == 1 ? mine <= theirs : mine < theirs;
}

}  // namespace tile_plan
}  // namespace dps
