// Dense linear layer for many tokens: tcgen05.mma over CTA PAIRS (cta_group::2), the rebuilt weights as the A operand in
// tensor memory, the activations as the B operand in the shared memory of both CTAs.
//
// Paper: "Scheduler: Dual-Precision Execution" -- full mode combines the FP8 tensor with the residual tensor into the
// original FP16 values during computation; fast mode uses the FP8 tensor alone.
//
// What bounds a prefill main loop on this part is what an SM can pull out of L2, about 50 bytes a clock, and in full mode
// its shared memory (128 bytes a clock).  A CTA by itself with a 128 x 256 tile needs 48 KB (full mode) per 64 columns of K
// and 512 tensor cycles; a CTA of a pair with a (2 x 128) x 256 tile needs 32 KB, because it fetches half of the tokens
// and the tensor cores of both SMs read both halves.
//
// Tile: 256 weight rows x `tokens` tokens (a multiple of kTokenStep, chosen per launch), K walked in steps of 128.  Persistent: a pair
// per two SMs walks the tiles.  Roles of a CTA (24 warps):
//   warp 0       plane producer: units of 128 rows x 128 columns of P (and R) into a ring; a unit is handed back as soon as
//                the zip warps have it in registers, so the ring holds nothing that waits for the tensor core
//   warp 2       activation producer: this CTA's half of the tile's tokens into slots, a K step at a time (64 columns at a
//                time the loop took 880 cycles per step); the bytes of both CTAs are counted on the first CTA's barrier,
//                where the MMAs that read both halves are issued
//   warp 3       (first CTA) waits for both halves of a step's activations and reports them to the MMA warp
//   warps 8-23   zip warps: plane bytes -> FP16 in registers -> tensor memory.  Eight take a step (a quarter of the rows and a
//                half of the columns each), eight the next one.  A step is a chain of latencies in a warp (1400 cycles for
//                64 columns: waits of 150 each even when nothing has to be waited for, loads and conversion 600), not
//                arithmetic: eight warps in all made 650 cycles per 64 columns
//   warp 1       (first CTA) issues the MMAs of the pair: one wait, eight MMAs and one commit per step, about 600 cycles;
//                with a barrier of its own for the activations and another commit for the A slots, in steps of 64 columns,
//                it took 650 per step however few tokens there were
//   warps 4-7    epilogue of this CTA's rows: each warp takes its 32 rows by itself (64 contiguous bytes of a token's y)
// Against single CTAs, the four Llama-7B linears together, fast / full mode: 256 tokens 140 / 183 -> 114 / 150 us, 512
// 209 / 269 -> 174 / 237, 2048 715 / 889 -> 644 / 739, 8192 2696 / 3500 -> 2598 / 3007 (there the power cap holds the clock
// near 1.4 GHz).
// The arrivals on the other CTA's barriers carry no cluster-scope release (with it a step took twice as long): what they
// order is tensor memory only, by the tcgen05 fences on both sides.  Nothing that a CTA or its copy engine wrote to shared
// memory is handed over by them: the activations of the second CTA complete on the first one's barrier.
#include <cuda_fp16.h>

#include <cstdio>
#include <cstdlib>
#include <type_traits>

#include "bits.cuh"
#include "dps_internal.h"
#include "pair_plan.h"
#include "sm100.cuh"
#include "tensor_map.h"

namespace dps {

namespace {

using namespace sm100;

using namespace pair_plan;

constexpr int kACols = kUnitK / 2;         // tensor memory of one K step of A
constexpr int kDone = 8;                   // ring of barriers that report completed K steps
constexpr int kThreads = 768;

struct PairParams {
    __half* y;
    int M, N, K;
    int tokens;        // per tile
    int tail_tokens;   // per piece of a tile of the last, partial round
    int tail_parts;    // pieces such a tile is cut into (1: not cut)
    int units, x_slots;
    int ahead;         // plane units asked of L2 in front of their loads
    int split;         // K split: pairs of a cluster that share a tile, each a range of its K steps (then one tile per cluster)
    // What every warp would have to divide for in front of the first load: pairs in the grid (with a split, clusters), row tiles,
    // (not grouped) token tiles and the tiles of whole rounds, and the K steps' quotient and remainder by the split (the first
    // ranges are a step longer).  With several token tiles, with pieces and in grouped launches an item still takes a division or two.
    int pairs, row_tiles, tok_tiles, t_main, steps_each, steps_over;
    int* status;
    int64_t ldy;       // elements from one token's row of y to the next
};

// D[tmem] (+)= A[tmem] * B[smem] over a CTA pair; issued by ONE thread of the pair's first CTA.  Addresses and descriptor
// hold for both CTAs: each brings its 128 rows of A and its half of B's rows.
__device__ __forceinline__ void umma_f16_ts_pair(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc,
                                                 uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
        ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}

__device__ __forceinline__ uint4 lds128(uint32_t addr) {
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr));
    return v;
}

// Tensor memory: accumulators first (two tiles' worth where they fit, so that the next tile's MMAs overlap the epilogue),
// then the A slots.
struct Work {
    int row_tile, m0;       // tile row index, first token (grouped: first sorted row)
    int tokens, ncols;      // MMA columns, columns that exist
    int plane_row0;         // grouped: first plane row of the expert in the [E * N][K] view
    bool piece;             // a piece of a tile of the last round
    bool e5m2, rounded;     // grouped: the expert's encoding
};

// Grouped (MoE) launches: token tiles built on the device by the routing pre-pass, (expert, first sorted row, rows, unused).
struct PairGroups {
    const int4* tiles;
    const int32_t* num_tiles;
    const int32_t* sorted_rows;   // sorted position -> caller's row id
    uint32_t e5m2[32];            // bit e set: expert e is E5M2 (truncated or rounded)
    uint32_t rounded[32];         // bit e set: expert e is a rounded nest (full mode only; fast mode reads P alike)
};

// 64 columns of one row (half a unit): plane bytes -> packed FP16 pairs.
template <int ENC, bool FULL>
__device__ __forceinline__ void rebuild(uint32_t prow, int half, uint32_t sw, uint32_t (&h)[32]) {
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const uint32_t off = ((uint32_t)(4 * half + c) ^ sw) * 16u;
        const uint4 pv = lds128(prow + off);
        const uint4 rv = FULL ? lds128(prow + kRows * kUnitK + off) : make_uint4(0, 0, 0, 0);
        uint32_t h8[8];
        if (FULL) join16<ENC, FULL>(pv, rv, h8);
        else fast16<ENC>(pv, h8);   // E4M3: 2^8 times the weights, undone in the epilogue
#pragma unroll
        for (int q = 0; q < 8; ++q) h[c * 8 + q] = h8[q];
    }
}

// GROUPED: a work item is a row tile of one expert x one of its token tiles; ENC is not used, the encoding is the expert's.
// WIDE: tiles of 320 or 384 tokens in two halves, an accumulator and MMAs each: what is fetched, rebuilt and stored of the weights serves half
// as many tokens more.  74 row tiles of 8192 columns, short of the power cap, 256 -> 384 tokens, us: fast 56.8 -> 79.5, full 70.7 -> 93.0, 7 and
// 12 % less per token.  Under the cap, where the MMAs' energy is most of it: a Llama-7B layer, full mode, tiles of 256 -> these, 1536 tokens 630 -> 566,
// 4096 1525 -> 1466, 8192 2950 -> 2866 (two runs a side, 3 % apart).  (A template argument: with the halves counted at run time in the issuer's
// loop 512 tokens took 2 % longer.)
template <int ENC, bool FULL, bool GROUPED, bool WIDE>
__global__ void __launch_bounds__(kThreads, 1)
umma_pair_kernel(const __grid_constant__ CUtensorMap map_p, const __grid_constant__ CUtensorMap map_r,
                 const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_xt, const PairParams prm,
                 const PairGroups gp) {
    constexpr int kUnit = unit_bytes(FULL);
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t bar_p_full[kMaxUnits], bar_p_empty[kMaxUnits];
    __shared__ __align__(8) uint64_t bar_x_full[kMaxXSlots];    // the first CTA's count the bytes of both
    __shared__ __align__(8) uint64_t bar_a_full[kASteps];       // the first CTA's: A and activations of both are ready
    __shared__ __align__(8) uint64_t bar_done[kDone];           // the MMAs of a K step are complete
    __shared__ __align__(8) uint64_t bar_d_full[2];
    __shared__ __align__(8) uint64_t bar_d_empty[2];            // the first CTA's count for both
    __shared__ uint32_t tmem_base_slot;

    grid_launch_dependents();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int split = prm.split;
    const uint32_t first = cluster_ctarank() & ~1u;             // cluster rank of the pair's first CTA
    const int rank = (int)(cluster_ctarank() & 1u), ks = (int)(first >> 1);
    const int pair = (int)cluster_id(), pairs = prm.pairs;      // (split > 1: the cluster)
    const int units = prm.units, x_slots = prm.x_slots;
    constexpr int kHalves = WIDE ? 2 : 1, kRing = WIDE ? kWideASteps : kASteps;
    const int x_atom = prm.tokens / (2 * kHalves) * 128, x_bytes = prm.tokens * 128;   // 64 columns of K of a half; a slot, 128 of all
    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t x_base = smem_base + (uint32_t)(units * kUnit);
    const uint32_t epi_base = x_base + (uint32_t)(x_slots * x_bytes);
    const int row_tiles = prm.row_tiles;
    if (GROUPED) grid_dependency_wait();                        // the tile list comes from the routing pre-pass
    const int tok_tiles = GROUPED ? *gp.num_tiles : prm.tok_tiles;
    const int total = row_tiles * tok_tiles, t_main = GROUPED ? total : prm.t_main;
    const int step0 = ks * prm.steps_each + min(ks, prm.steps_over);      // this pair's K steps of a tile
    const int steps_k = prm.steps_each + (ks < prm.steps_over ? 1 : 0);

    // Work item `i` of this pair: whole tiles, then at most one piece of a tile of the last round.
    auto work = [&](int i, Work& w) -> bool {
        int lin = pair + i * pairs, part = 0;
        w.piece = false;
        if (GROUPED) {
            if (lin >= total) return false;
            const int4 g = gp.tiles[lin / row_tiles];
            w.row_tile = lin % row_tiles;
            w.m0 = g.y;
            w.ncols = g.z;
            w.tokens = (g.z + kTokenStep - 1) / kTokenStep * kTokenStep;
            w.plane_row0 = g.x * prm.N;
            w.e5m2 = (gp.e5m2[g.x >> 5] >> (g.x & 31)) & 1u;
            w.rounded = FULL && ((gp.rounded[g.x >> 5] >> (g.x & 31)) & 1u);
            return true;
        }
        w.plane_row0 = 0;
        if (lin >= t_main) {
            if (lin - pair != t_main || prm.tail_parts <= 1) return false;
            lin = t_main + pair / prm.tail_parts;
            part = pair % prm.tail_parts;
            if (lin >= total) return false;
            w.piece = true;
        }
        int tok_tile = 0;
        w.row_tile = lin;
        if (tok_tiles > 1) {
            // groups of 8 row tiles x all token tiles: the planes and activation tiles in use stay in L2
            constexpr int kRowGroup = 8;
            const int per_group = kRowGroup * tok_tiles;
            const int group = lin / per_group, within = lin % per_group;
            const int rows_here = min(kRowGroup, row_tiles - group * kRowGroup);
            w.row_tile = group * kRowGroup + within % rows_here;
            tok_tile = within / rows_here;
        }
        w.tokens = w.piece ? prm.tail_tokens : prm.tokens;
        const int end = min(prm.M, (tok_tile + 1) * prm.tokens);
        w.m0 = tok_tile * prm.tokens + part * prm.tail_tokens;
        w.ncols = min(w.tokens, end - w.m0);
        return w.ncols > 0;      // a piece past the last token is the end: nothing follows a piece
    };

    auto load_unit = [&](int s, int step, int row) {            // by one thread
        const uint32_t full = smem_u32(&bar_p_full[s]), dst = smem_base + (uint32_t)(s * kUnit);
        mbar_arrive_expect_tx(full, (uint32_t)kUnit);
        tma_load_2d(dst, &map_p, full, step * kUnitK, row);
        if (FULL) tma_load_2d(dst + kRows * kUnitK, &map_r, full, step * kUnitK, row);
    };
    auto ask = [&](int step, int row) {                         // the same unit into L2 only
        tma_prefetch_l2_2d(&map_p, step * kUnitK, row);
        if (FULL) tma_prefetch_l2_2d(&map_r, step * kUnitK, row);
    };
    const int ahead = FULL ? prm.ahead : 0;
    Work w;
    int loaded = 0;               // units loaded ahead of the roles (by warp 0)
    if (warp == 0) {
        if (lane == 0) {
            for (int s = 0; s < units; ++s) {
                mbar_init(smem_u32(&bar_p_full[s]), 1);
                mbar_init(smem_u32(&bar_p_empty[s]), 8);            // the zip warps that take the step
            }
            fence_barrier_init();
            fence_async_proxy();
        }
        __syncwarp();
        // the others need the barriers only: they do not wait for the requests below (130 cycles each, twelve in fast mode)
        named_barrier_arrive(1, kThreads);
        cluster_arrive();
        // The planes are model state, and their barriers this CTA's own: the ring fills while tensor memory is allocated and the pair
        // meets.  Four linears in a chain, fast / full mode, loads by the role after the meeting (and quotients computed on the device)
        // -> loads here with the block waiting for this warp -> as it is, us: Llama-7B 72 tokens 72.3 / 102.8 -> 71.3 / 100.4 -> 70.7 /
        // 100.4, 512 168.6 / 213.9 -> 167.0 / 207.2 -> 164.5 / 201.2; 2048-wide layers, 256 tokens, 50.6 / 60.5 -> 50.0 / 56.0 -> 47.3 /
        // 53.5; 1264-wide, 1189 tokens, planes out of L2, 61.7 / 71.2 -> 63.3 / 72.3 -> 59.6 / 67.2.  (The step between holds the L2
        // requests in full mode and the sum over a K split as well.)
        if (work(0, w)) {
            loaded = min(units, steps_k);
            if (elect_one()) {
                const int row = w.plane_row0 + (2 * w.row_tile + rank) * kRows;
                for (int s = 0; s < loaded; ++s) load_unit(s, step0 + s, row);
                for (int s = loaded; s < min(loaded + ahead, steps_k); ++s) ask(step0 + s, row);
            }
            __syncwarp();
        }
    } else if (warp == 2) {
        if (lane == 0) {
            for (int s = 0; s < x_slots; ++s) mbar_init(smem_u32(&bar_x_full[s]), 1);
            for (int a = 0; a < kRing; ++a) mbar_init(smem_u32(&bar_a_full[a]), 2 * 8 + 1);   // both CTAs' eight zip warps, warp 3
            for (int a = 0; a < kDone; ++a) mbar_init(smem_u32(&bar_done[a]), 1);
            for (int a = 0; a < 2; ++a) {
                mbar_init(smem_u32(&bar_d_full[a]), 1);
                mbar_init(smem_u32(&bar_d_empty[a]), 8);            // the epilogue warps of both CTAs
            }
            fence_barrier_init();
            prefetch_tensormap(&map_x);
        }
        __syncwarp();             // the barriers below are .aligned: the whole warp arrives at once
    }
    if (warp == 1) tmem_alloc_pair(smem_u32(&tmem_base_slot), 512);
    if (warp != 0) {
        tc_fence_before_sync();
        named_barrier_sync(1, kThreads);
        cluster_arrive();
    }
    cluster_wait();               // the other CTA's barriers exist
    tc_fence_after_sync();
    const uint32_t tmem_base = tmem_base_slot;
    const uint32_t tmem_a = tmem_base + 512u - kRing * kACols;
    // accumulators: one or two tiles' worth
    const int accs = 2 * prm.tokens <= kAccCols ? 2 : 1;

    // K steps are counted over all tiles of the pair (t).  A waiter for step t cannot take an older phase of
    // bar_done[t % kDone] for it: it has seen a step later than t - kDone before.
    auto wait_done = [&](uint32_t t) { return mbar_wait(smem_u32(&bar_done[t % kDone]), (t / kDone) & 1u); };

    bool ok = true;
    if (warp == 0) {
        // ---------------- plane producer (model state: does not wait for the preceding kernel): what follows the ring above ----------------
        int s = 0;
        uint32_t ph = 1;          // a fresh barrier passes a wait for the phase before its first
        uint32_t issued = 0;
        bool more = work(0, w);
        for (int i = 0; ok && more; ++i) {
            const int row = w.plane_row0 + (2 * w.row_tile + rank) * kRows;
            more = work(i + 1, w);
            const int next_row = w.plane_row0 + (2 * w.row_tile + rank) * kRows;
            for (int u = 0; u < steps_k && ok; ++u, ++issued, s = (s + 1 == units) ? 0 : s + 1, ph ^= (s == 0)) {
                if (issued < (uint32_t)loaded) continue;
                ok = mbar_wait(smem_u32(&bar_p_empty[s]), ph);
                ok = __all_sync(0xFFFFFFFFu, ok);
                if (!ok) break;
                if (elect_one()) {
                    load_unit(s, step0 + u, row);
                    if (ahead > 0) {
                        const int v = u + ahead - steps_k;       // that many steps into the next tile
                        if (v < 0) ask(step0 + u + ahead, row);
                        else if (more && v < steps_k) ask(step0 + v, next_row);
                    }
                }
                __syncwarp();
            }
        }
        drain_copies(bar_p_full, issued, (uint32_t)units);
    } else if (warp == 2) {
        // ---------------- activation producer: this CTA's half of the tokens ----------------
        grid_dependency_wait();
        int s = 0;
        uint32_t t = 0;
        for (int i = 0; ok && work(i, w); ++i) {
            const int halves = WIDE && !w.piece ? 2 : 1, half = w.tokens / (2 * halves);   // this CTA's share of an MMA's tokens
            const int m0 = w.m0 + rank * half;
            // (grouped: boxes of a quarter of the tile's tokens when they do)
            const bool small = GROUPED ? 4 * half <= prm.tokens : w.piece;
            const CUtensorMap* map = small ? &map_xt : &map_x;
            const int box = GROUPED ? (small ? prm.tokens / 4 : prm.tokens / 2) : half;
            for (int j = 0; j < steps_k && ok; ++j, ++t, s = (s + 1 == x_slots) ? 0 : s + 1) {
                if (t >= (uint32_t)x_slots) ok = wait_done(t - (uint32_t)x_slots);
                ok = __all_sync(0xFFFFFFFFu, ok);
                if (!ok) break;
                if (elect_one()) {
                    const uint32_t full = map_to_cta(smem_u32(&bar_x_full[s]), first), dst = x_base + (uint32_t)(s * x_bytes);
                    // (the second CTA's bytes may land before this: the phase still waits for the one arrival)
                    if (rank == 0) mbar_arrive_expect_tx(smem_u32(&bar_x_full[s]), (uint32_t)(2 * 2 * box * 128 * halves));
                    for (int h = 0; h < halves; ++h) {
                        const uint32_t to = dst + (uint32_t)(2 * h * x_atom);
                        tma_load_2d_pair(to, map, full, (step0 + j) * kUnitK, m0 + 2 * h * half);
                        tma_load_2d_pair(to + (uint32_t)x_atom, map, full, (step0 + j) * kUnitK + 64, m0 + 2 * h * half);
                    }
                }
                __syncwarp();
            }
        }
        // (t: steps issued; the first CTA's barriers count both CTAs' bytes, the second CTA leaves with it)
        if (rank == 0) drain_copies(bar_x_full, t, (uint32_t)x_slots);
    } else if (warp == 3) {
        // ---------------- reports the activations of a K step, both halves: the pair's first CTA ----------------
        int s = 0;
        uint32_t ph = 0, t = 0;
        for (int i = 0; rank == 0 && ok && work(i, w); ++i) {
            for (int j = 0; j < steps_k && ok; ++j, ++t, s = (s + 1 == x_slots) ? 0 : s + 1, ph ^= (s == 0)) {
                if (t >= kRing) ok = wait_done(t - kRing);    // else the arrival might count for that step
                if (ok) ok = mbar_wait(smem_u32(&bar_x_full[s]), ph);
                ok = __all_sync(0xFFFFFFFFu, ok);
                if (ok && lane == 0) mbar_arrive(smem_u32(&bar_a_full[t % kRing]));
            }
        }
    } else if (warp == 1) {
        // ---------------- MMA issuer: the pair's first CTA ----------------
        int xs = 0;
        uint32_t t = 0;
        for (int i = 0; rank == 0 && ok && work(i, w); ++i) {
            const int halves = WIDE && !w.piece ? 2 : 1, n = w.tokens / halves;
            const uint32_t idesc = umma_idesc_f16(2 * kRows, n);
            const int acc = accs == 2 ? i & 1 : 0, use = accs == 2 ? i >> 1 : i;
            const uint32_t tmem_d = tmem_base + (uint32_t)(acc * prm.tokens);
            // the tile before must have been read out of the accumulator by both CTAs
            auto wait_empty = [&](int a) {
                if (use > 0) {
                    ok = __all_sync(0xFFFFFFFFu, mbar_wait(smem_u32(&bar_d_empty[a]), (uint32_t)(use - 1) & 1u));
                    tc_fence_after_sync();
                }
                return ok;
            };
            if (!wait_empty(acc)) break;
            for (int j = 0; j < steps_k && ok; ++j, ++t) {
                const uint32_t a = t % kRing;
                const bool second = (step0 + j) * kUnitK + 64 < prm.K;        // (behind the end of K both operands are zero)
                const uint64_t bdesc_first = umma_desc_k_sw128(x_base + (uint32_t)(xs * x_bytes));
                ok = __all_sync(0xFFFFFFFFu, mbar_wait(smem_u32(&bar_a_full[a]), (t / kRing) & 1u));
                if (!ok) break;
                tc_fence_after_sync();
#pragma unroll
                for (int h = 0; h < kHalves; ++h) {
                    if (h == 1 && (halves == 1 || (j == 0 && !wait_empty(1)))) break;
                    const uint64_t bdesc0 = bdesc_first + (uint64_t)((2 * h * x_atom) >> 4);
                    const uint64_t bdesc1 = bdesc0 + (uint64_t)(x_atom >> 4);
                    const uint32_t d = tmem_d + (uint32_t)(h * n);
                    if (elect_one()) {
#pragma unroll
                        for (int q = 0; q < 4; ++q)                 // 16 columns of K = 32 bytes of the 128-byte swizzle atom
                            umma_f16_ts_pair(d, tmem_a + a * kACols + q * 8, bdesc0 + (uint64_t)(q * 2), idesc, (j > 0 || q > 0) ? 1u : 0u);
                        if (second) {
#pragma unroll
                            for (int q = 0; q < 4; ++q)
                                umma_f16_ts_pair(d, tmem_a + a * kACols + 32 + q * 8, bdesc1 + (uint64_t)(q * 2), idesc, 1u);
                        }
                        if (h == halves - 1) umma_commit_pair(smem_u32(&bar_done[t % kDone]), first);
                        if (j == steps_k - 1) umma_commit_pair(smem_u32(&bar_d_full[acc + h]), first);
                    }
                    __syncwarp();
                }
                xs = xs + 1 == x_slots ? 0 : xs + 1;
            }
        }
    } else if (warp >= 8) {
        // ---------------- zip warps: planes -> FP16 -> tensor memory ----------------
        const int set = (warp - 8) >> 3, half = ((warp - 8) >> 2) & 1;   // K steps of this parity; columns 64 half ... of a step
        const int row = (warp & 3) * 32 + lane;
        const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
        const uint32_t sw = (uint32_t)(row & 7);                // TMA swizzle: 16-byte chunk index ^= row % 8
        // t: the step; s, ph: its unit (an even number of units: a unit's readers are always the same)
        uint32_t s = (uint32_t)set, ph = 0, t = (uint32_t)set, done = 0;
        for (int i = 0; ok && work(i, w); ++i) {
            done += (uint32_t)steps_k;                          // steps up to the end of this tile
            for (; t < done; t += 2) {
                ok = __all_sync(0xFFFFFFFFu, mbar_wait(smem_u32(&bar_p_full[s]), ph));
                if (!ok) break;
                const uint32_t prow = smem_base + s * kUnit + (uint32_t)(row * kUnitK);
                uint32_t h[32];
                if constexpr (!GROUPED) {
                    rebuild<ENC, FULL>(prow, half, sw, h);
                } else if (FULL && w.rounded) {
                    if (w.e5m2) rebuild<kEncE5M2R, FULL>(prow, half, sw, h);
                    else rebuild<kEncE4M3R, FULL>(prow, half, sw, h);
                } else {
                    if (w.e5m2) rebuild<kEncE5M2, FULL>(prow, half, sw, h);
                    else rebuild<kEncE4M3, FULL>(prow, half, sw, h);
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&bar_p_empty[s]));
                s += 2;
                if (s >= (uint32_t)units) s -= (uint32_t)units, ph ^= 1u;
                const uint32_t a = t % kRing;
                if (t >= kRing) ok = __all_sync(0xFFFFFFFFu, wait_done(t - kRing));  // the MMAs that read the slot before
                if (!ok) break;
                tc_fence_after_sync();
                tmem_st_32x32b_x32(tmem_a + lane_base + a * kACols + (uint32_t)(half * 32), h);
                tmem_wait_st();
                tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster(map_to_cta(smem_u32(&bar_a_full[a]), first));
            }
        }
    } else if (warp >= 4 && split == 1) {
        // ---------------- epilogue: D[row][token] -> FP16 -> y[token][row], every warp its 32 rows ----------------
        const int q = warp & 3;
        const uint32_t lane_base = (uint32_t)(q * 32) << 16;
        const uint32_t buf = epi_base + (uint32_t)(q * kEpiCols * 64);
        for (int i = 0; work(i, w); ++i) {
            const float out_scale = (!FULL && (GROUPED ? !w.e5m2 : base_enc(ENC) == kEncE4M3)) ? 0.00390625f : 1.0f;
            // grouped: the callers' row ids of the chunk's tokens, one per lane, a chunk ahead of their use
            int32_t ids = GROUPED && lane < w.ncols ? gp.sorted_rows[w.m0 + lane] : 0;
            const int acc = accs == 2 ? i & 1 : 0, use = accs == 2 ? i >> 1 : i;
            const int halves = WIDE && !w.piece ? 2 : 1, per = w.tokens / halves;
            const uint32_t tmem_d = tmem_base + lane_base + (uint32_t)(acc * prm.tokens);
            const int n = (2 * w.row_tile + rank) * kRows + q * 32 + (lane & 3) * 8;
            __half* yrow = prm.y + (GROUPED ? (int64_t)n : (int64_t)(w.m0 + (lane >> 2)) * prm.ldy + n);
            // (a grouped launch of 8 x 1024 x 4096, fast mode, 48 / 128 rows per expert: 20.7 / 25.7 us with a chunk end and a 64-bit pitch for every kind of
            // tile, 20.3 / 25.4 with both only where they are needed)
            for (int h = 0, c0 = 0; h < kHalves; ++h) {
                if (h == halves) break;
                ok = mbar_wait(smem_u32(&bar_d_full[acc + h]), (uint32_t)use & 1u);
                ok = __all_sync(0xFFFFFFFFu, ok);
                if (!ok) break;
                tc_fence_after_sync();
                const int end = WIDE ? min(w.ncols, (h + 1) * per) : w.ncols;
                auto read_out = [&] {                        // the accumulator is free again
                    tc_fence_before_sync();
                    __syncwarp();
                    if (lane == 0) mbar_arrive_cluster(map_to_cta(smem_u32(&bar_d_empty[acc + h]), first));
                };
                if (WIDE && c0 >= end) read_out();           // no token reaches this half
                for (; c0 < end; c0 += kEpiCols) {
                    uint32_t v[32];
                    tmem_ld_32x32b_x32(tmem_d + (uint32_t)c0, v);
                    int32_t next_ids = 0;
                    if (GROUPED && c0 + kEpiCols + lane < w.ncols) next_ids = gp.sorted_rows[w.m0 + c0 + kEpiCols + lane];
                    tmem_wait_ld();
                    if (c0 + kEpiCols >= end) read_out();    // last chunk read
#pragma unroll
                    for (int j = 0; j < 32; ++j) {
                        const __half hv = __float2half_rn(__uint_as_float(v[j]) * out_scale);
                        asm volatile("st.shared.u16 [%0], %1;" ::"r"(buf + (uint32_t)(j * 64 + lane * 2)),
                                     "h"(__half_as_ushort(hv))
                                     : "memory");
                    }
                    __syncwarp();
#pragma unroll
                    for (int t = 0; t < 4; ++t) {            // 8 tokens x 64 bytes per instruction; N is a multiple of 8
                        const uint4 val = lds128(buf + (uint32_t)(t * 512 + lane * 16));
                        const int64_t m = GROUPED ? __shfl_sync(0xFFFFFFFFu, ids, 8 * t + (lane >> 2)) : c0 + 8 * t;
                        if (n < prm.N && c0 + 8 * t + (lane >> 2) < w.ncols)
                            *reinterpret_cast<uint4*>(yrow + m * (GROUPED ? (int64_t)prm.N : prm.ldy)) = val;
                    }
                    ids = next_ids;
                    __syncwarp();                            // the buffer is free for the next chunk
                }
            }
            if (!ok) break;
        }
    }
    if (!ok) atomicExch(prm.status, (int)DPS_ERR_CUDA);
    if (!WIDE && split > 1) {
        // A range of K each: the FP32 partial tile goes to shared memory, [token][row], over the rings -- the tile's MMAs are complete,
        // nothing is in flight any more.  Five warps share a quarter's columns (the epilogue's and its four zip warps).
        const bool tile = work(0, w);
        if (warp >= 4 && tile) {
            const int q = warp & 3;
            ok = __all_sync(0xFFFFFFFFu, ok && mbar_wait(smem_u32(&bar_d_full[0]), 0u));
            if (!ok) atomicExch(prm.status, (int)DPS_ERR_CUDA);
            tc_fence_after_sync();
            const float out_scale = (!FULL && base_enc(ENC) == kEncE4M3) ? 0.00390625f : 1.0f;
            for (int c0 = ((warp - 4) >> 2) * kEpiCols; ok && c0 < w.ncols; c0 += 5 * kEpiCols) {
                uint32_t v[32];
                tmem_ld_32x32b_x32(tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)c0, v);
                tmem_wait_ld();
#pragma unroll
                for (int j = 0; j < 32; ++j)
                    if (c0 + j < w.ncols)
                        asm volatile("st.shared.f32 [%0], %1;" ::"r"(smem_base + (uint32_t)(((c0 + j) * kRows + q * 32 + lane) * 4)),
                                     "f"(__uint_as_float(v[j]) * out_scale)
                                     : "memory");
            }
        }
        // Summed in the order of the K ranges: pair ks takes every split-th token, each CTA its own rows (the same in all pairs),
        // consecutive threads consecutive 8-row pieces.  All loads of a piece are issued before the first sum: one trip
        // through the cluster each instead of `split`.  4096 x 4096, fast / full mode, with four warps for the partial tiles and a
        // loop over the parts: 64 tokens 10.9 / 12.6 us, 256 15.0 / 17.3; now 10.4 / 12.2 and 14.5 / 16.7.
        __syncthreads();
        cluster_sync_all();
        auto sum = [&](auto parts) {
            constexpr int kParts = decltype(parts)::value;
            const int n0 = (2 * w.row_tile + rank) * kRows;
            const int mine = (w.ncols - ks + kParts - 1) / kParts;
            for (int idx = (int)threadIdx.x; idx < mine * (kRows / 8); idx += kThreads) {
                const int c = ks + kParts * (idx / (kRows / 8)), n = n0 + (idx % (kRows / 8)) * 8;
                if (n >= prm.N) continue;                // N is a multiple of 8
                const uint32_t local = smem_base + (uint32_t)((c * kRows + (idx % (kRows / 8)) * 8) * 4);
                float4 a[kParts], b[kParts];
#pragma unroll
                for (int p = 0; p < kParts; ++p) {
                    const uint32_t from = map_to_cta(local, (uint32_t)(2 * p + rank));
                    a[p] = ld_cluster_v4_f32(from);
                    b[p] = ld_cluster_v4_f32(from + 16u);
                }
                float t[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
                for (int p = 0; p < kParts; ++p) {
                    t[0] += a[p].x; t[1] += a[p].y; t[2] += a[p].z; t[3] += a[p].w;
                    t[4] += b[p].x; t[5] += b[p].y; t[6] += b[p].z; t[7] += b[p].w;
                }
                uint32_t out[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const __half2 h = __floats2half2_rn(t[2 * k], t[2 * k + 1]);
                    out[k] = *reinterpret_cast<const uint32_t*>(&h);
                }
                *reinterpret_cast<uint4*>(prm.y + (int64_t)(w.m0 + c) * prm.ldy + n) = make_uint4(out[0], out[1], out[2], out[3]);
            }
        };
        if (tile) {
            if (split == 2) sum(std::integral_constant<int, 2>{});
            else if (split == 3) sum(std::integral_constant<int, 3>{});
            else sum(std::integral_constant<int, 4>{});
        }
    }
    tc_fence_before_sync();
    __syncthreads();
    cluster_sync_all();           // nobody frees tensor memory or leaves while the pair still works
    if (warp == 1) {
        tc_fence_after_sync();
        tmem_dealloc_pair(tmem_base, 512);
    }
}

// ---- host side ---------------------------------------------------------------------------------

// `query`, where not null: nothing is launched, its answers are filled in.  prepare_only: all but the launch.
template <int ENC, bool FULL>
cudaError_t launch_enc(const void* x, const uint8_t* p, const uint8_t* r, void* y, int64_t ldy, int64_t M, int64_t N, int64_t K, int* status,
                       cudaStream_t stream, const PairQuery* query, bool prepare_only) {
    auto kernel = umma_pair_kernel<ENC, FULL, false, false>, wide_kernel = umma_pair_kernel<ENC, FULL, false, true>;
    // Clusters of s pairs that are resident at once, per device (they must fit inside a GPC): filled by the first call on a
    // device, read only after that set-up has returned.
    static int capacity_of[kMaxDevices][kMaxSplit + 1] = {};
    static PerDeviceOnce setup;     // per instantiation and per device
    int dev = 0;
    {
        const cudaError_t e = setup.run([&] {
            int d = 0;
            cudaGetDevice(&d);
            cudaError_t a = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
            if (a == cudaSuccess) a = cudaFuncSetAttribute(wide_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
            if (a != cudaSuccess) return a;
            for (int s = 1; s <= kMaxSplit; ++s) {
                cudaLaunchConfig_t q = {};
                q.gridDim = dim3((unsigned)(2 * s), 1, 1);
                q.blockDim = dim3(kThreads, 1, 1);
                q.dynamicSmemBytes = kSmemBytes;
                cudaLaunchAttribute qa[1];
                qa[0].id = cudaLaunchAttributeClusterDimension;
                qa[0].val.clusterDim.x = (unsigned)(2 * s);
                qa[0].val.clusterDim.y = 1;
                qa[0].val.clusterDim.z = 1;
                q.attrs = qa;
                q.numAttrs = 1;
                int clusters = 0;
                if (cudaOccupancyMaxActiveClusters(&clusters, kernel, &q) != cudaSuccess) clusters = 0;
                capacity_of[d][s] = clusters;
            }
            (void)cudaGetLastError();
            if (capacity_of[d][1] <= 0) capacity_of[d][1] = sm_count() / 2;
            return cudaSuccess;
        }, &dev);
        if (e != cudaSuccess) return e;
    }
    const int pairs = capacity_of[dev][1];
    if (query != nullptr && query->share != nullptr) *query->share = share_rows(FULL, M, N, K, pairs);
    if (query != nullptr && query->turns == nullptr) return cudaSuccess;
    const Plan plan = make_plan(FULL, M, N, K, capacity_of[dev]);
    const int64_t row_tiles = (N + 2 * kRows - 1) / (2 * kRows), tok_tiles = (M + plan.tokens - 1) / plan.tokens;
    const int64_t tiles = row_tiles * tok_tiles, grid_pairs = plan.split > 1 ? tiles : tiles < pairs ? tiles : pairs;
    if (query != nullptr) {
        *query->turns = tile_plan::turns(tiles, plan.split, pairs);
        return cudaSuccess;
    }
    CUtensorMap mp, mr, mx, mxt;
    if (!make_map_2d(&mp, p, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, (uint64_t)N, (uint64_t)K, kRows, kUnitK,
                     CU_TENSOR_MAP_SWIZZLE_128B))
        return cudaErrorInvalidValue;
    mr = mp;
    if (FULL && !make_map_2d(&mr, r, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, (uint64_t)N, (uint64_t)K, kRows, kUnitK,
                             CU_TENSOR_MAP_SWIZZLE_128B))
        return cudaErrorInvalidValue;
    if (!make_map_2d(&mx, x, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, (uint64_t)M, (uint64_t)K, (uint32_t)mma_tokens(plan.tokens) / 2, 64,
                     CU_TENSOR_MAP_SWIZZLE_128B))
        return cudaErrorInvalidValue;
    mxt = mx;
    if (plan.tail_parts > 1 && !make_map_2d(&mxt, x, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, (uint64_t)M, (uint64_t)K,
                                            (uint32_t)plan.tail_tokens / 2, 64, CU_TENSOR_MAP_SWIZZLE_128B))
        return cudaErrorInvalidValue;
    if (prepare_only) return cudaSuccess;
    PairParams prm = {};
    prm.y = static_cast<__half*>(y);
    prm.M = (int)M;
    prm.N = (int)N;
    prm.K = (int)K;
    prm.ldy = ldy;
    prm.tokens = plan.tokens;
    prm.tail_tokens = plan.tail_tokens;
    prm.tail_parts = plan.tail_parts;
    prm.split = plan.split;
    prm.status = status;
    const Rings rings = size_rings(FULL, plan.tokens);
    prm.units = rings.units;
    prm.x_slots = rings.x_slots;
    prm.ahead = ahead_units(FULL, M, rings);
    const int64_t steps = (K + kUnitK - 1) / kUnitK;
    prm.pairs = (int)grid_pairs;
    prm.row_tiles = (int)row_tiles;
    prm.tok_tiles = (int)tok_tiles;
    prm.t_main = (int)(plan.tail_parts > 1 ? tiles - tiles % grid_pairs : tiles);
    prm.steps_each = (int)(steps / plan.split);
    prm.steps_over = (int)(steps % plan.split);
    if (getenv("DPS_DEBUG"))
        fprintf(stderr, "[dps] pair full=%d M=%lld N=%lld K=%lld tokens=%d tiles=%lld tail=%dx%d split=%d (%d %d %d %d) units=%d x_slots=%d\n", (int)FULL,
                (long long)M, (long long)N, (long long)K, plan.tokens, (long long)tiles, plan.tail_parts, plan.tail_tokens,
                plan.split, capacity_of[dev][1], capacity_of[dev][2], capacity_of[dev][3], capacity_of[dev][4], prm.units, prm.x_slots);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(2 * plan.split * grid_pairs), 1, 1);
    cfg.blockDim = dim3(kThreads, 1, 1);
    cfg.dynamicSmemBytes = kSmemBytes;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)(2 * plan.split);
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    cudaError_t e = cudaLaunchKernelEx(&cfg, plan.tokens > kMaxTokens ? wide_kernel : kernel, mp, mr, mx, mxt, prm, PairGroups{});
    count_launch();
    return e;
}

template <bool FULL>
cudaError_t launch_grouped(const uint32_t* masks, const void* x_sorted, const uint8_t* p, const uint8_t* r, void* y, int64_t A,
                           int64_t N, int64_t K, int32_t E, int tn, const void* tiles, const int32_t* num_tiles,
                           const int32_t* sorted_rows, int max_tiles, int* status, cudaStream_t stream) {
    auto kernel = umma_pair_kernel<0, FULL, true, false>;
    static PerDeviceOnce setup;     // per instantiation and per device
    {
        const cudaError_t e = setup.run(
            [&] { return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes); });
        if (e != cudaSuccess) return e;
    }
    CUtensorMap mp, mr, mx, mxt;
    if (!make_map_2d(&mp, p, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, (uint64_t)E * (uint64_t)N, (uint64_t)K, kRows, kUnitK,
                     CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B))
        return cudaErrorInvalidValue;
    mr = mp;
    if (FULL && !make_map_2d(&mr, r, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, (uint64_t)E * (uint64_t)N, (uint64_t)K, kRows, kUnitK,
                             CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B))
        return cudaErrorInvalidValue;
    if (!make_map_2d(&mx, x_sorted, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, (uint64_t)A, (uint64_t)K, (uint32_t)tn / 2, 64,
                     CU_TENSOR_MAP_SWIZZLE_128B))
        return cudaErrorInvalidValue;
    if (!make_map_2d(&mxt, x_sorted, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, (uint64_t)A, (uint64_t)K, (uint32_t)tn / 4, 64,
                     CU_TENSOR_MAP_SWIZZLE_128B))
        return cudaErrorInvalidValue;
    PairParams prm = {};
    prm.y = static_cast<__half*>(y);
    prm.M = (int)A;
    prm.N = (int)N;
    prm.K = (int)K;
    prm.ldy = N;
    prm.tokens = prm.tail_tokens = tn;
    prm.tail_parts = 1;
    prm.split = 1;
    prm.status = status;
    const Rings rings = size_rings(FULL, tn);
    prm.units = rings.units;
    prm.x_slots = rings.x_slots;
    PairGroups gp;
    gp.tiles = static_cast<const int4*>(tiles);
    gp.num_tiles = num_tiles;
    gp.sorted_rows = sorted_rows;
    for (int i = 0; i < 32; ++i) {   // the caller's array holds the E5M2 bits, then the rounded-nest bits
        gp.e5m2[i] = masks[i];
        gp.rounded[i] = FULL ? masks[32 + i] : 0u;
    }
    const int64_t row_tiles = (N + 2 * kRows - 1) / (2 * kRows), upper = row_tiles * max_tiles;
    const int64_t pairs = upper < sm_count() / 2 ? upper : sm_count() / 2;
    prm.pairs = (int)pairs;
    prm.row_tiles = (int)row_tiles;
    prm.steps_each = (int)((K + kUnitK - 1) / kUnitK);
    if (getenv("DPS_DEBUG"))
        fprintf(stderr, "[dps] pair grouped full=%d A=%lld N=%lld K=%lld E=%d tokens=%d tiles<=%lld units=%d x_slots=%d\n", (int)FULL,
                (long long)A, (long long)N, (long long)K, (int)E, tn, (long long)upper, prm.units, prm.x_slots);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(2 * pairs), 1, 1);
    cfg.blockDim = dim3(kThreads, 1, 1);
    cfg.dynamicSmemBytes = kSmemBytes;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = 2;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, mp, mr, mx, mxt, prm, gp);
    count_launch();
    return e;
}

}  // namespace

cudaError_t launch_pair_grouped(int mode, const uint32_t* masks, const void* x_sorted, const uint8_t* p, const uint8_t* r, void* y,
                                int64_t A, int64_t N, int64_t K, int32_t E, int tn, const void* tiles, const int32_t* num_tiles,
                                const int32_t* sorted_rows, int max_tiles, int* status, cudaStream_t stream) {
    return mode == DPS_MODE_FULL ? launch_grouped<true>(masks, x_sorted, p, r, y, A, N, K, E, tn, tiles, num_tiles, sorted_rows,
                                                        max_tiles, status, stream)
                                 : launch_grouped<false>(masks, x_sorted, p, r, y, A, N, K, E, tn, tiles, num_tiles, sorted_rows,
                                                         max_tiles, status, stream);
}

namespace {
cudaError_t launch_or_plan(int mode, int enc, const void* x, const uint8_t* p, const uint8_t* r, void* y, int64_t ldy, int64_t M, int64_t N,
                           int64_t K, int* status, cudaStream_t stream, const PairQuery* query, bool prepare_only) {
    const bool full = mode == DPS_MODE_FULL;
    if (!full) enc = base_enc(enc);   // fast mode reads the persistent byte of a rounded nest like any other
    auto go = [&](auto launch) { return launch(x, p, r, y, ldy, M, N, K, status, stream, query, prepare_only); };
    if (enc == kEncE4M3R) return go(launch_enc<kEncE4M3R, true>);
    if (enc == kEncE5M2R) return go(launch_enc<kEncE5M2R, true>);
    if (enc == kEncE4M3) return full ? go(launch_enc<kEncE4M3, true>) : go(launch_enc<kEncE4M3, false>);
    return full ? go(launch_enc<kEncE5M2, true>) : go(launch_enc<kEncE5M2, false>);
}
}  // namespace

cudaError_t launch_pair_linear(int mode, int enc, const void* x, const uint8_t* p, const uint8_t* r, void* y, int64_t ldy, int64_t M,
                               int64_t N, int64_t K, int* status, cudaStream_t stream, bool prepare_only) {
    return launch_or_plan(mode, enc, x, p, r, y, ldy, M, N, K, status, stream, nullptr, prepare_only);
}

cudaError_t ask_pair_plan(int mode, int enc, int64_t M, int64_t N, int64_t K, const PairQuery& query) {
    return launch_or_plan(mode, enc, nullptr, nullptr, nullptr, nullptr, N, M, N, K, nullptr, nullptr, &query, false);
}

}  // namespace dps
