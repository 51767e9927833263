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

// Rows per tile where K is not split because there are more tiles of kTileRows rows than SMs.  Two CTAs fit an SM: as many tiles as
// slots allow without another wave, and 5 % less, load the SMs evenly, where 172 tiles on 148 SMs leave one tile on most and two on
// some.  Full mode, tiles of kTileRows rows against what this chooses, us: 10-16 tokens 22016 x 4096 (88 rows) 35.9 / 32.1, 27648 x
// 5120 (104) 48.2 / 45.1, 32768 x 6144 (120) 63.5 / 60.4, 57344 x 8192 (104) 156.5 / 142.5, 128256 x 4096 166 / 156.5; 32 tokens, whose
// activations cost an SM more per tile, only where the load is most uneven: 22016 x 4096 (88) 36.5 / 33.0, but 27648 x 5120 48.5 / 48.4,
// 57344 x 8192 158.5 / 156.5, 128256 x 4096 170 / 172.7.  Below 88 rows the K blocks' latencies show: 22016 x 4096 with 72 rows 44.
// Fast mode, half the bytes per K block and so latencies earlier, only for 10-16 tokens, up to two waves, 96 or 104 rows and matrices
// of 2^27 weights and more: 40000 x 4096 (96) 37.9 / 34.4, 20000 x 8192 (96) 36.5 / 35.0, 57344 x 8192 (104) 81.2 / 78.2, a layer with
// the last of them 152.9 / 149.3; but 32768 x 6144 (120) 34.6 / 34.8, 128256 x 4096 (120) 88.3 / 93.2, and 22016 x 4096 (96), 21.0 /
// 20.0 by itself, leaves its layer at 50.3 / 50.4.  At 32 tokens, with 96 rows: 40.3 / 37.9, 38.1 / 38.2 on the first two, 22016 x 4096
// 21.0 / 21.4.  64-token tiles, which carry twice the activations again, lose in both modes.
// From K = 1536 on: a shorter K is over before the even load shows, and more tiles are more fixed costs.  Full mode, 128 rows / lower, us: 24
// tokens 22016 x 512 6.1 / 6.7, x 1024 9.5 / 10.2, x 1536 14.7 / 14.1, 41472 x 256 7.4 / 8.9, x 1536 29.4 / 26.1; 12 tokens 57344 x 768 17.3 / 19.5,
// x 1024 21.7 / 23.7, x 1536 32.4 / 30.6, 128256 x 1024 46.0 / 47.8, x 1536 66.0 / 62.3.  (In between, 38016 x 1024 18.6 / 17.3 at 24 tokens.)
inline int low_rows(bool full, int64_t N, int64_t K, int tn, int64_t sms) {
    const int64_t slots = 2 * sms, tiles = (N + kTileRows - 1) / kTileRows;
    if (tiles <= sms || K < 1536 || (!full && N * K < ((int64_t)1 << 27))) return kTileRows;
    const int64_t waves = (tiles + slots - 1) / slots;
    int64_t rows = (N * 20 + waves * slots * 19 - 1) / (waves * slots * 19);   // N / (0.95 of the slots)
    rows = (rows + 7) / 8 * 8;
    const int64_t least = full ? 88 : 96, most = full ? (tn > 16 ? 88 : 120) : 104;
    if (rows < least) rows = least;
    if (rows > most || (!full && (tn > 16 || waves > 2))) return kTileRows;
    return (int)rows;
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
