// Tile plan of the CTA-pair linear (pair_linear.cu): plain host arithmetic, no CUDA, so that it can be checked over every size.
#pragma once
#include <cmath>
#include <cstdint>
#include <cstdlib>

namespace dps {
namespace pair_plan {

constexpr int kRows = 128;                 // weight rows of a row block in one CTA
constexpr int kUnitK = 128;                // columns of K in a plane unit
constexpr int kMaxUnits = 12, kMaxXSlots = 8;
constexpr int kASteps = 4;                 // K steps the A ring in tensor memory holds
constexpr int kAccCols = 512 - kASteps * (kUnitK / 2);
constexpr int kMaxSplit = 4;               // pairs of a cluster (eight CTAs, the portable limit)
constexpr int kEpiCols = 32;               // token columns per epilogue chunk
constexpr int kEpiBytes = 4 * kEpiCols * 64;
constexpr int kSmemBytes = 222 * 1024;     // ring + slots + epilogue chunks + alignment

// Token widths are multiples of 32: CUTLASS's atom for this instruction, SM100_MMA_F16BF16_2x1SM_TS (A in tensor memory, two
// CTAs), admits N = 32, 64 .. 256 and nothing between; only the form with A in shared memory goes in steps of 16.
constexpr int kTokenStep = 32;
constexpr int kMaxTokens = 256;            // of one MMA

// Wide tiles, two MMAs of half the tokens each per step of A: what is rebuilt and stored to tensor memory, and fetched of the planes,
// serves half as many tokens more.  Their accumulators leave the A ring two steps.
constexpr int kWideTokens[] = {320, 384};
constexpr int kWideASteps = 2;
constexpr int mma_tokens(int tokens) { return tokens > kMaxTokens ? tokens / 2 : tokens; }

constexpr int unit_bytes(bool full) { return kRows * kUnitK * (full ? 2 : 1); }

struct Rings {
    int units, x_slots;
};

struct Plan {
    int tokens = 256, tail_parts = 1, tail_tokens = 256, split = 1;
    double cost = 0;
};

// Time of one K step of a tile in ns, all pairs at work: measured with 74 and 148 tiles of one width (18944 and 37888 rows,
// 8192 columns; in full mode, up to 128 tokens, on planes that come out of L2) every 32 tokens, between them in proportion.  Measured
// before the ring was filled ahead of the roles and, for full mode from 192 tokens on, without the L2 requests of ahead_units: it ranks
// widths and splits, it does not predict a launch (four Llama-7B linears, 64 tokens, full mode: 72 us by it, 95 measured).
inline double step_ns(bool full, int tokens) {
    static const double fast_ns[13] = {370, 370, 415, 480, 535, 610, 685, 750, 850, 940, 1030, 1115, 1200};
    static const double full_ns[13] = {500, 500, 520, 600, 680, 800, 1000, 1040, 1100, 1175, 1250, 1330, 1415};
    const double* t = full ? full_ns : fast_ns;
    const int i = tokens >= 384 ? 11 : tokens / 32;
    return t[i] + (t[i + 1] - t[i]) * (tokens - 32 * i) / 32.0;
}

// A round of tiles over the pairs takes as long as one tile, so the number of token tiles is chosen to make the sum over the
// rounds small; the tiles of a last, partial round are cut into pieces of the tokens if that shortens it.  Few tiles: up to
// four pairs share each, a range of K each; capacity[s] = clusters of s pairs that are resident at once.
// DPS_PAIR_TOKENS=1..384 (rounded up to a width there is) and DPS_PAIR_SPLIT=1..4 override (tuning knobs).
inline Plan make_plan(bool full, int64_t M, int64_t N, int64_t K, const int* capacity) {
    static const int forced = [] { const char* e = getenv("DPS_PAIR_TOKENS"); return e ? (atoi(e) + kTokenStep - 1) / kTokenStep * kTokenStep : 0; }();
    static const int forced_split = [] { const char* e = getenv("DPS_PAIR_SPLIT"); return e ? atoi(e) : 0; }();
    const int64_t steps = (K + kUnitK - 1) / kUnitK, pairs = capacity[1];
    const int64_t row_tiles = (N + 2 * kRows - 1) / (2 * kRows), t0 = (M + 255) / 256;
    Plan best;
    auto consider = [&](int64_t tokens, int split) {
        const int64_t tiles = row_tiles * ((M + tokens - 1) / tokens);
        if (split > 1 && (tiles > capacity[split] || steps < 2 * split)) return;
        if (forced_split && split != forced_split && !(split == 1 && (tiles > capacity[forced_split] || steps < 2 * forced_split))) return;
        const int64_t rounds = tiles / pairs, tail = split > 1 ? 1 : tiles % pairs;
        Plan p;
        p.split = split;
        p.tokens = p.tail_tokens = (int)tokens;
        // between tiles: with one accumulator the MMAs wait until it has been read out
        const double drain = 2 * tokens <= kAccCols ? 100.0 : 3.0 * (double)mma_tokens((int)tokens);
        const double cost1 = step_ns(full, (int)tokens);
        p.cost = (double)rounds * ((double)steps * cost1 + drain) + 4.0 * (double)tokens;
        if (split > 1) {
            // the sum over the cluster: 1 us + 30 ns per token (measured with a loop over the parts; it is about 0.4 us less now)
            p.cost = (double)((steps + split - 1) / split) * cost1 + 1000.0 + 30.0 * (double)tokens;
        } else if (tail > 0) {
            double last = (double)steps * cost1;
            for (int parts = 2; rounds > 0 && parts <= 8 && parts * tail <= pairs && kTokenStep * parts <= tokens; ++parts) {
                const int tt = (int)(((tokens + parts - 1) / parts + kTokenStep - 1) / kTokenStep * kTokenStep);
                const double c = 1.2 * (double)steps * step_ns(full, tt) + drain;   // (the pieces stream the planes again)
                if (c < 0.9 * last) { last = c; p.tail_parts = parts; p.tail_tokens = tt; }
            }
            p.cost += last;
        }
        // (wide tiles instead of others only for 3 % and more: four Llama-7B linears, 2048 tokens, fast mode, 0.6 % by this, 647 -> 661 us measured)
        const bool first_wide = tokens > kMaxTokens && best.tokens <= kMaxTokens;
        if (best.cost == 0 || p.cost < (first_wide ? 0.97 : 1.0) * best.cost) best = p;
    };
    for (int64_t t = t0, end = t0 + (t0 < 12 ? t0 + 4 : 16); t <= end; ++t) {
        int64_t tokens = ((M + t - 1) / t + kTokenStep - 1) / kTokenStep * kTokenStep;
        if (forced >= kTokenStep && forced <= kMaxTokens) tokens = forced;
        for (int split = 1; split <= kMaxSplit; ++split) consider(tokens, split);
    }
    if (M > kMaxTokens && (forced == 0 || forced > kMaxTokens)) {
        if (forced > kMaxTokens) best = Plan();
        for (int tokens : kWideTokens)
            if (forced == 0 || (forced <= 320) == (tokens == 320)) consider(tokens, 1);
    }
    return best;
}

// 17 to 128 tokens: whether the pairs take a matrix, and, where it has a row tile per pair and more, how many of its rows, the rest being
// better off as a launch of its own (decode tiles or pairs, K shared out over clusters) than as a last round that leaves most pairs idle.
//
// All figures are us per launch in loops of a third of a second, i.e. under the 1000 W cap, which is where a server runs; T: row tiles of 256 (74
// pairs), (r): of them behind whole rounds; tiles / pairs / pairs and a launch for the rest (the cut).
//
// 33-64 tokens, full mode          K = 2048               4096                 8192                 14336
//   T  76  (2)             21.2 / 19.8 / 20.7   41.6 / 40.0 / 37.1   80.0 / 78.3 / 67.8
//   T  78  (4)                                                       81.2 / 78.9 / 69.0    146 /  139 /  118
//   T  90 (16)             23.0 / 21.8 / 24.9   45.2 / 43.6 / 43.4   87.0 / 84.4 / 78.8    156 /  146 /  134
//   T 100 (26)             24.6 / 22.9 / 27.6   47.5 / 45.3 / 46.8   92.0 / 88.2 / 85.1    165 /  152 /  143
//   T 109 (35)                                                       99.0 / 92.4 / 95.2    172 /  159 /  163
//   T 119 (45)                                                        104 / 95.3 / 99.0    180 /  167 /  168
//   T 125 (51)                                                        106 / 98.2 /  108    185 /  173 /  188
//   T 150  (2)             40.7 / 34.4 / 35.6   76.7 / 67.7 / 64.9    148 /  132 /  122
//   T 152  (4)                                                        150 /  134 /  123    265 /  232 /  212
//   T 164 (16)                                                        156 /  140 /  134    284 /  241 /  228
//   T 174 (26)                                                        160 /  141 /  140    282 /  244 /  245
//   T 183 (35)                                                        163 /  144 /  152    286 /  254 /  258
//   T 190 (42)             46.1 / 40.0 / 45.4   86.0 / 76.9 / 81.2    168 /  149 /  149
//   T 199 (51)                                                        170 /  152 /  163    301 /  276 /  283
//   T 226  (4)             51.7 / 47.8 / 50.3    100 / 94.7 / 93.1    193 /  186 /  178
//   With linears between them that the tiles serve, two changes of the family and a launch more cost some 3.5 us: a Llama-7B layer, T 86 and
//   K 4096 on the pairs, 102.7 / 103.6, so one round and a rest only from K = 5120 on.
// 33-64 tokens, fast mode; a wave of the tiles is 148 T, and they are the faster ones where their waves are as full as the pairs' rounds
//   T  76  (2)                                  22.2 / 23.6 / 23.2   44.0 / 46.8 / 42.0
//   T  84 (10)                                  24.2 / 25.5 / 25.7   46.5 / 49.4 / 45.4
//   T 152  (4)                                  43.8 / 40.0 / 40.0   84.9 / 80.1 / 74.2    143 /  135 /  125
//   T 159 (11)                                  45.8 / 42.0 / 42.7   86.7 / 83.2 / 79.0    147 /  138 /  129
//   T 168 (20)                                  47.0 / 43.2 / 45.0   88.6 / 85.0 / 83.1    150 /  146 /  136
//   T 178 (30)                                  49.0 / 45.7 / 47.2   92.1 / 87.9 / 87.8    156 /  151 /  144
//   T 188 (40)                                  50.3 / 46.8 / 50.0   95.0 / 90.9 / 93.5    160 /  156 /  157
//   T 198 (50)                                  51.4 / 49.0 / 53.8   97.5 / 94.0 /  101    159 /  160 /  168
//   T 208 (60)                                  53.6 / 50.8 / 55.2    104 / 98.2 /  103    174 /  169 /  175
//   T 221 (73)                                  56.0 / 52.4 / 57.0    108 /  103 /  106    180 /  178 /  183
//   T 226  (4)                                  56.4 / 56.9 / 56.7    108 /  108 /  107
//   T 296  (0)                                  68.4 / 67.1           133 /  136
// 17-32 tokens, full mode
//   T  76  (2)                                  34.1 / 38.2 / 34.2   66.6 / 74.7 / 61.5
//   T  90 (16)                                  38.0 / 40.9 / 38.1   73.7 / 80.0 / 71.0
//   T 100 (26)                                                       80.5 / 83.4 / 78.3
//   T 150  (2)                                  61.9 / 63.3 / 60.3    118 /  125 /  112
//   T 158 (10)             35.9 / 33.3 / 34.7   68.2 / 65.8 / 62.0    136 /  128 /  116    238 /  223 /  198
//   T 178 (30)                                                        143 /  135 /  131    254 /  229 /  220
//   T 190 (42)             40.8 / 37.1 / 40.2   78.2 / 71.4 / 73.9
//   T 193 (45)                                                        154 /  142 /  142    266 /  241 /  243
//   T 226  (4)             46.5 / 45.2 / 46.9   88.4 / 89.2 / 86.2    173 /  173 /  163
//   (In a layer of hidden size 6144, T 150 and K 6144, 190 / 185.)
// 33-64 tokens, a tile per pair at most, tiles / pairs: fast mode       full mode
//   T 40                    K = 3072 11.1 / 12.0, 8192 24.5 / 25.8    3072 16.7 / 16.7, 8192 37.9 / 39.4
//   T 46                             12.6 / 12.2       30.5 / 27.8         18.9 / 17.8       47.7 / 42.4
//   T 58                             14.3 / 13.2       33.1 / 31.1         22.6 / 20.5       54.2 / 47.7
//   T 73                             16.6 / 15.3       37.3 / 35.5         25.5 / 24.5       63.1 / 57.3
//   T 74                             16.9 / 15.7       39.1 / 36.3         26.6 / 24.8  5104 49.4 / 40.5
//   With other linears between them, which the tiles serve, each change of the family costs: with T 48 on the pairs a Llama-7B layer took 63.5 / 64.3
//   in fast mode and 102.2 / 101.5 in full mode, with T 60 one of hidden size 5120 86.5 / 84.8 and 142 / 137, with T 66 one of 3088 43.1 / 42.0 and
//   63.1 / 62.4.  So: from 0.8 of the pairs on.
// 96 tokens, pairs / cut (a last round there is cut into pieces of the tokens), K 4096, 8192: full mode T 76 41.7 / 39.1, 81.7 / 72.0; 84 44.7 /
//   45.4, 84.6 / 78.1; 158 73.3 / 75.0, 142 / 136; 226 99.8 / 99.2, 197 / 193; fast mode 76 25.8 / 25.7, 50.3 / 46.0; 84 27.8 / 29.8, 54.1 / 52.2;
//   158 45.8 / 48.1, 89.2 / 86.3.
struct RowShare {
    bool pairs = false;      // false: as if there were no such rule
    int64_t rows = 0;        // of y that whole rounds serve; 0: all of them, in one launch
};
// What the cut gains over one launch of pairs, us, fitted to the tables: a round's memory time by its K steps, less a launch's fixed costs and the
// rest's own time, which grows with the K steps as well.  The fits are off by a microsecond or two, so a gain of less is none.
constexpr double kLeastGain = 1.5;
inline double cut_gain(bool full, int64_t M, int64_t steps, int64_t rest) {
    const double s = (double)steps, r = (double)rest;
    if (!full) return 0.15 * s - 3.5 - r * 0.0033 * s;
    return M > 32 ? 0.244 * s - 4.5 - r * (0.10 + 0.0033 * s) : 0.35 * s - 7.0 - r * 0.006 * s;
}
// The rest's row tiles at most (of 74 pairs): beyond, its decode tiles are too many to share K out over clusters five ways (33-64 tokens, full mode)
// or four ways, and a round of the pairs is as good.
inline int64_t most_rest(bool full, int64_t M) { return full && M > 32 ? 26 : 37; }
// DPS_ROW_CUT=0: never, 1: wherever there is a whole round and a rest, up to 256 tokens (tuning knob).
inline int row_cut_knob() {
    static const int knob = [] { const char* e = getenv("DPS_ROW_CUT"); return e ? atoi(e) : -1; }();
    return knob;
}
// Whether share_rows can answer anything but no: small matrices and other numbers of tokens, whose calls are host time, do not ask.
inline bool may_share_rows(int64_t M, int64_t N, int64_t sms) { return M > 16 && M <= (row_cut_knob() == 1 ? kMaxTokens : 128) && N * 4 >= sms * 2 * kRows; }
inline RowShare share_rows(bool full, int64_t M, int64_t N, int64_t K, int64_t pairs) {
    const int knob = row_cut_knob();
    const int64_t tiles = (N + 2 * kRows - 1) / (2 * kRows), steps = (K + kUnitK - 1) / kUnitK;
    const int64_t rounds = tiles / pairs, rest = tiles % pairs, rows = rest > 0 ? rounds * pairs * 2 * kRows : 0;
    if (knob == 0 || M <= 16 || M > kMaxTokens) return {};
    if (tiles <= pairs) {
        if (M <= 32 || M > 64 || K >= 16384) return {};
        return {5 * tiles >= 4 * pairs && K >= 3072, 0};
    }
    if (knob == 1) return {true, rows};
    const bool cut = rest > 0 && rest <= most_rest(full, M) && cut_gain(full, M, steps, rest) > kLeastGain;
    if (M <= 64 && K >= 16384) return {};        // (a rule of its own: tile_plan.h)
    if (M > 128) return {};
    if (M > 64) return (rest > 0 && ((steps >= 64 && rest <= 10) || (full && steps >= 32 && rest <= 4))) ? RowShare{true, rows} : RowShare{};
    if (rounds == 1) {
        if (full && M > 32 && K >= 5120) return {true, cut ? rows : 0};
        // (fast mode: from 33 tokens on, and against the tiles, which are the faster ones here)
        return (full || M > 32) && cut && steps >= 64 && rest <= (full ? 26 : 10) ? RowShare{true, rows} : RowShare{};
    }
    // two rounds and more; `even`: the tiles' waves are as full as the pairs' rounds
    const bool even = rounds + (rest > 0) >= 2 * ((tiles + 2 * pairs - 1) / (2 * pairs));
    if (steps < (full && M > 32 ? 16 : 32)) return {};
    if (M <= 32 && (!full || (steps < 48 && (even || rest <= 4)))) return {};
    if (!full && even) return {};
    return {true, cut ? rows : 0};
}

// Shared memory: activations take 2000 cycles and more out of L2, so four K steps of them are kept in flight at least
// (2.5 steps: 1250 cycles per step of 256 tokens in full mode instead of 1024; three of a wide tile, whose steps are longer), more if four plane
// units still fit; the planes have the A ring as a second buffer, two units do.  An even number of units, so that a unit's phases are all seen
// by the same zip warps.
inline Rings size_rings(bool full, int tokens) {
    const int x_bytes = tokens * 128, room = kSmemBytes - 1024 - kEpiBytes;
    int xs = (room - 4 * unit_bytes(full)) / x_bytes;
    const int least = tokens > kMaxTokens ? 3 : 4;
    xs = xs < least ? least : xs > kMaxXSlots ? kMaxXSlots : xs;
    const int units = (room - xs * x_bytes) / unit_bytes(full);
    return {units > kMaxUnits ? kMaxUnits : units & ~1, xs};
}

// Plane units asked of L2 ahead of their loads.  A ring of two units (full mode, tiles of 192 tokens and more) has 64 KB per SM in
// flight at best, and memory's latency takes more: the three units behind it are asked for too.  Up to 512 tokens: up to 256 every pair streams
// planes of its own; with two token tiles two pairs read, and ask for, the same planes and it still gains, with more it gained nothing.  Four linears in a
// chain, full mode, without / with 3 / 4 / 6 units, us: Llama-7B 192 tokens 132.8 / 121.5 / 122.2 / 124.2, 256 141 / 133.9 / 134.2 /
// 135.8, 512 222 / 216.8 / 216.7 / 217.1; 8192-wide 256 tokens 481 / 434 / 443 / 456.  Rings of four units lose by it: 12288 x 4096 at
// 128 tokens 24.7 / - / 25.5 in full mode, 256 tokens in fast mode 26.8 / - / 27.3.
inline int ahead_units(bool full, int64_t M, const Rings& rings) { return full && rings.units == 2 && M <= 512 ? 3 : 0; }

// Token-tile width of grouped launches: an expert with a quarter, or two and a half standard deviations of an even routing,
// more rows than the average still fits the average's number of tiles.
inline int grouped_tokens(int64_t A, int32_t E) {
    const double avg = (double)A / E, spread = 2.5 * sqrt(avg);
    const double want = avg + (spread > 0.25 * avg ? spread : 0.25 * avg);
    const int tiles = (int)ceil(want / 256.0);
    const int tokens = (int)ceil(want / tiles / kTokenStep) * kTokenStep;
    return tokens < kTokenStep ? kTokenStep : tokens > kMaxTokens ? kMaxTokens : tokens;
}

// Grouped launches: CTA pairs or 128-row tiles, two CTAs per SM.  From 48 rows per expert on pairs, whose tiles are wide enough for an expert's rows.
// Below, with a token tile per expert, it is turns over the chip: the pairs go in rounds of a 256-row tile each; a wave of the other tiles, as many
// as CTA slots, takes as long as two rounds and counts for two turns.  (An expert whose rows end in the first half of a 256-row tile is half a tile
// more work for the pairs: 32 experts of 1152 rows are three rounds of 160 tiles, or one wave of 288.)  The pairs win where rounds are fewer than
// turns, and from eight rounds on, which make fixed costs small, whatever the turns, that are then an eighth fewer at most.
// Tiles / pairs, us per call in loops, i.e. under the power cap, by rows per expert:
//   experts x N x K  rounds turns | fast mode: 16         24          40          | full mode: 12 or 13  16          24          40
//    8 x 28672 x 4096    13    14 |    178 / 186    194 / 188   209 / 208   |     335 / 322   340 / 328   350 / 330   357 / 349
//   16 x 12288 x 2048    11    12 |   85.9 / 82.9  93.3 / 85.8   104 / 92.9 |     151 / 144   155 / 142   158 / 146   164 / 159
//   64 x 2048 x 1408      7     8 |   47.3 / 45.5  53.2 / 46.6  59.0 / 53.4 |    78.6 / 71.1 81.6 / 72.6 83.5 / 74.8 90.9 / 82.4
//    4 x 4096 x 8192      1     2 |   38.3 / 36.1  42.7 / 36.9  44.0 / 38.2 |    75.1 / 57.0 76.5 / 57.1 70.3 / 57.7 71.5 / 59.1
//    8 x 4096 x 14336     2     2 |   91.5 / 100   99.6 / 105    114 / 115  |     174 / 173   174 / 174   181 / 176   189 / 187
//    8 x 2816 x 8192      2     2 |   43.7 / 57.6  49.8 / 56.7  53.4 / 59.4 |    85.4 / 91.5 86.5 / 91.9 83.0 / 92.3 88.0 / 94.9
//    4 x 16384 x 4096     4     4 |   53.6 / 59.5  59.6 / 59.8  65.2 / 67.4 |     102 / 101   101 / 102   102 / 103   107 / 110
//   64 x 2816 x 2048     10    10 |   83.0 / 81.3  92.0 / 83.3  99.5 / 96.4 |     143 / 136   143 / 137   149 / 140   158 / 151
//   32 x 1152 x 2048      3     2 |                24.6 / 28.8  26.4 / 31.8 |    37.0 / 42.7             39.8 / 44.4 41.2 / 46.5
//    8 x 4736 x 4096      3     2 |                38.0 / 45.1  39.5 / 47.9 |    60.0 / 73.2             61.4 / 73.7 64.8 / 76.8
//   64 x 1152 x 2048      5     4 |                43.8 / 44.6  49.8 / 52.6 |    68.4 / 69.9             71.3 / 72.5 77.4 / 80.0
//   16 x 6976 x 1024      7     6 |                33.0 / 32.0  36.5 / 36.9 |    48.6 / 49.3             51.6 / 49.7 54.3 / 54.1
//   64 x 1664 x 2048      7     6 |                59.2 / 58.4  66.3 / 67.4 |    91.8 / 94.6             96.8 / 97.6  103 / 105
//   32 x 4736 x 1024      9     8 |                44.4 / 41.5  49.4 / 47.2 |    65.0 / 62.8             69.2 / 65.7 72.6 / 70.1
//   64 x 2880 x 2048     11    10 |                94.2 / 90.0   105 / 104  |     151 / 149               154 / 151   164 / 163
//   256 x 1152 x 1024    18    16 |                 103 / 91.0   124 / 111  |     130 / 123               141 / 134   157 / 156
// Fast mode with fewer than 20 rows: 12 rows on the first three 168 / 176, 83.8 / 84.7, 46.5 / 44.3; eight rows lose in both modes.
// More than kRoutedByTable experts: the routing kernel, which then has a warp walk all rows for each expert, is most of a call, and lives on the L1
// cache.  A launch of pairs leaves the SMs split for its 222 KB of shared memory, and the next call's routing reads through what is left: 512 experts of
// 384 x 1024 with 24 rows each, fast mode, calls back to back, 799 / 1372 (routing alone 800 / 1270, calls with waits between them 830 / 830); 1024 of 128 x 1024
// 3742 / 5260; 13 rows, full mode, 481 / 777 and 1600 / 2820.
constexpr int kRoutedByTable = 256;
inline bool grouped_on_pairs(bool full, int64_t A, int64_t N, int64_t K, int32_t E, int64_t pairs) {
    if (A >= 48 * (int64_t)E) return true;
    if (A < (full ? 12 : 20) * (int64_t)E || E > kRoutedByTable) return false;
    const int64_t tiles = E * ((N + 2 * kRows - 1) / (2 * kRows)), rounds = (tiles + pairs - 1) / pairs;
    const int64_t half_tiles = E * ((N + kRows - 1) / kRows), turns = 2 * ((half_tiles + 4 * pairs - 1) / (4 * pairs));
    if (rounds == 1) return 5 * tiles >= 4 * pairs && K >= 3072;      // (as dense launches: share_rows)
    return rounds < turns || rounds >= 8;
}

// The token-tile width of a grouped launch.  Below 48 rows per expert an uneven routing must not undo what grouped_on_pairs counted: an expert with
// more rows than a tile is another row of items, and one round of the pairs becomes two where the other kernel's wave has room.  A wider tile costs
// the ring's depth only (an item multiplies the columns it has): nothing in full mode up to 128 tokens in one round and 96 in more, 0-2 % in fast
// mode for 96.  128-row tiles / pairs by the average's width / as it is, us, 40 rows per expert, an even routing and one that gives an expert 30 %
// of the rows on top, fast | full mode:
//   4 x 4096 x 8192 (one round)     44.1 / 38.9 / 39.8, 46.0 / 53.3 / 38.7 | 71.9 / 60.7 / 61.8, 76.7 / 85.1 / 61.5
//   8 x 2304 x 8192 (one)           47.4 / 42.6 / 43.4, 49.5 / 56.0 / 56.7 | 76.4 / 67.1 / 67.2, 81.9 / 89.8 / 66.8     (128 in fast mode: 44.8, 45.2)
//   16 x 1024 x 4096 (one)          28.5 / 24.3 / 24.2, 30.3 / 33.2 / 24.2 | 43.7 / 36.8 / 37.1, 46.3 / 49.0 / 36.7
//   3 x 15496 x 4096 (three)        51.6 / 49.4 / 49.4, 55.5 / 55.4 / 55.4 | 87.3 / 83.2 / 82.1, 90.7 / 98.5 / 81.1
//   8 x 14336 x 4096 (seven)         114 /  115 /  115,  118 /  110 /  110 |  189 /  184 /  186,  200 /  204 /  185
inline int grouped_width(bool full, int64_t A, int64_t N, int32_t E, int64_t pairs) {
    const int tokens = grouped_tokens(A, E);
    if (A >= 48 * (int64_t)E) return tokens;
    const bool one_round = E * ((N + 2 * kRows - 1) / (2 * kRows)) <= pairs;
    const int least = one_round ? (full ? 128 : 96) : full ? 96 : kTokenStep;
    return tokens < least ? least : tokens;
}

}  // namespace pair_plan
}  // namespace dps
