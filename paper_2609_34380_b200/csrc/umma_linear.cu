// Tensor-core path of the dense linear layer: tcgen05.mma with the reconstructed weights as the
// A operand in tensor memory and the activations as the B operand in shared memory.
//
// Paper: "Scheduler: Dual-Precision Execution" -- full mode combines the FP8 tensor with the
// residual tensor into the original FP16 values *during computation*; fast mode uses the FP8
// tensor alone.  Here that combination happens on the way from shared memory to tensor memory.
//
// Tile: 128 weight rows (UMMA M; 88 to 120 of them hold weights in the lower tiles, see low_rows in tile_plan.h) x TN tokens (UMMA N),
// K walked in blocks of 128 or 64.  The problem
// is "swapped": D[row][token] = sum_k W[row][k] * x[token][k], so that even a handful of decode
// tokens fills the 128-lane datapath with weight rows and every weight byte is fetched once.
//
// Roles (10 warps):
//   warp 0     TMA producer: P tile (a tile's rows x 128 or 64 bytes), R tile (full mode), x tile (TN rows
//              of 64-element swizzle atoms) into a ring of shared-memory stages, completion
//              counted on mbarriers.  Dense tiles keep x in slots of their own, a second stream with its
//              own barriers (see x_slots below).
//   warp 1     allocates tensor memory; one elected lane issues tcgen05.mma (A from TMEM, B from
//              smem) and commits stage-release barriers.
//   warps 2-9  two groups of four "zip" warps; a warp owns 32 TMEM lanes = 32 weight rows.  Per K
//              block a thread reads its row's plane bytes (swizzled, conflict-free), rebuilds the
//              FP16 words in registers (byte permutes; hardware FP8 conversion for E4M3 fast mode)
//              and writes them to the A ring in TMEM with tcgen05.st.  The groups alternate K
//              blocks.  After the K loop the zip warps drain the accumulator (tcgen05.ld), round to
//              FP16 and store y through a shared-memory tile with 16-byte stores.
// Shared memory never holds FP16 weights, so its bandwidth is spent on 1-2 bytes per weight
// instead of 5-6, and the tensor core reads only the small activation tile from it.
//
// One tile per CTA, two CTAs per SM, 16 to 64 tokens wide; K is split over a cluster with a DSMEM mailbox.
// Wider tiles belong to the CTA pairs of pair_linear.cu.
#include <cuda_fp16.h>

#include <cstdio>
#include <cstdlib>

#include "bits.cuh"
#include "dps_internal.h"
#include "sm100.cuh"
#include "tensor_map.h"

namespace dps {

namespace {

using namespace sm100;
using namespace tile_plan;

// K elements per pipeline stage: 128 (128-byte plane rows, the widest swizzled TMA box) where it still leaves a ring of
// at least three or four stages, i.e. in fast mode; 64 in full mode (two planes per stage) with 64 tokens.  A ring of
// two stages cannot cover the 1600-2150 cycles a stage load takes; halving the stage doubles the ring depth.
// Full-mode tiles of up to 64 tokens read 64 columns per K block (two planes: the stage is as large as a
// fast-mode one), except the 32-token decode tiles: their stages are handed back as soon as the zip warps have
// read them, so two stages of 128-byte rows do, and 128-byte rows stream better than 64-byte ones (measured at
// 32 tokens, full mode, Llama-7B QKV / gate-up / o / down: 22.3 / 36.3 / 11.0 / 19.7 us against 22.8 / 38.9 /
// 11.5 / 20.2).
#ifndef DPS_FULL_BK128_MAX_TN
#define DPS_FULL_BK128_MAX_TN 32
#endif
#ifndef DPS_FULL_BK128_MIN_TN
#define DPS_FULL_BK128_MIN_TN 16   // 16-token tiles alike: 21.3 / 36.1 / 18.8 us against 23.0 / 38.4 / 20.0 (no o: too small)
#endif
__host__ __device__ constexpr int block_k(bool full, int tn) {
    return (full && !(tn >= DPS_FULL_BK128_MIN_TN && tn <= DPS_FULL_BK128_MAX_TN)) ? 64 : 128;
}
constexpr int kMaxAStages = 4;   // barrier array size for the A ring in tensor memory
// Groups of 4 zip warps; group g takes K blocks g, g + 2, ...
constexpr int kZipGroups = 2;
constexpr int kThreads = 64 + kZipGroups * 128;
constexpr int kMaxStages = 12;

__host__ __device__ constexpr int plane_stage_bytes(bool full, int tn) { return kTileRows * block_k(full, tn); }
__host__ __device__ constexpr int stage_bytes(bool full, int tn) {
    return plane_stage_bytes(full, tn) * (full ? 2 : 1) + tn * block_k(full, tn) * 2;
}
// Columns to allocate: accumulator + A ring, three or four A slots inside 256 columns (two CTAs per SM).
// A ring with an even stage ring: slots alternate between the zip groups (slot = block % slots).
__host__ __device__ constexpr int a_slots_max(bool full, int tn) { return block_k(full, tn) == 64 ? 4 : 3; }
__host__ __device__ constexpr int tmem_cols(bool full, int tn) {
    const int need = tn + a_slots_max(full, tn) * (block_k(full, tn) / 2);
    int c = 32;
    while (c < need) c <<= 1;
    return c;
}

// Activation slots kept apart from the plane ring.  Decode tiles (dense launches, 32 tokens): the plane
// stage and the activation tile of a K block have different consumers -- the zip warps take the planes into
// registers and hand the stage back at once, the MMAs read the activations several K blocks later -- and a
// tile fetched by the copy engine was measured to arrive 2000-2400 cycles after its request even out of L2.
// So the tiles get slots of their own, requested as soon as the MMAs that read a slot last are complete,
// five K blocks ahead in fast mode (three were 2-4 % slower on most Llama-7B shapes, six and eight leave
// too few plane stages in fast mode).  0 = the activation tile travels inside the stage.
// (16- and 64-token tiles: below.)
// Plane loading ahead of the dependency in decode tiles (see kPre in the kernel).  Measured inside the decode
// graphs at 32 tokens (fast / full, fraction of the copy bandwidth): nothing 0.55 / 0.60, the first ring pass
// 0.58 / 0.67, refills too 0.59 / 0.71, with the L2 prefetch of the second pass the same.
#ifndef DPS_PRE_DEP
#define DPS_PRE_DEP 3
#endif
#ifndef DPS_XSLOTS
#define DPS_XSLOTS 5        // fast mode
#endif
#ifndef DPS_XSLOTS_FULL
#define DPS_XSLOTS_FULL 3   // full mode: a stage is two planes of 16 KB, and three 8 KB slots leave room for two
#endif
constexpr int kMaxXSlots = 8;   // barrier array size
// 64-token tiles: the split-K mailbox takes 36 KB there, which leaves three plane stages and three slots in
// full mode and two of each in fast mode (one more slot each no longer fits two CTAs on an SM).  Measured
// at 64 tokens on the Llama-7B shapes against tiles that carry the activations in the stages: 0-14 % faster.
// 16-token tiles: slots in full mode only (fast mode with slots: gate-up 1-3 % faster, down 4 % slower).
#ifndef DPS_XSLOTS_FAST16
#define DPS_XSLOTS_FAST16 0
#endif
#ifndef DPS_XSLOTS_FULL64
#define DPS_XSLOTS_FULL64 3
#endif
#ifndef DPS_XSLOTS_FAST64
#define DPS_XSLOTS_FAST64 2
#endif
__host__ __device__ constexpr int x_slots(bool full, bool grouped, int tn) {
    if (grouped) return 0;
    if (tn == 64) return full ? DPS_XSLOTS_FULL64 : DPS_XSLOTS_FAST64;
    if (tn == 16) return full ? DPS_XSLOTS_FULL : DPS_XSLOTS_FAST16;
    return full ? DPS_XSLOTS_FULL : DPS_XSLOTS;
}
// Slots of a launch whose K is not split (no mailbox in shared memory): what the freed space holds best.
// 64-token tiles, fast mode: three slots and three stages instead of two and four (gate-up at 64 tokens:
// 22.3 us against 25.1); full mode: five slots beside the same number of stages.
__host__ __device__ constexpr int x_slots_alone(bool full, int tn) {
    if (x_slots(full, false, tn) == 0) return 0;
    if (tn == 64) return full ? 5 : 3;
    return 5;
}
__host__ __device__ constexpr int x_tile_bytes(bool full, int tn) { return tn * block_k(full, tn) * 2; }

// Optional timeline trace (compile with -DDPS_TRACE): lane 0 of each role of CTA (0,0,0) stamps
// the SM clock at pipeline events of every K block.  Read back with dps_debug_trace().
#ifdef DPS_TRACE
constexpr int kTraceBlocks = 64, kTraceEvents = 16;
__device__ long long g_trace[kTraceBlocks * kTraceEvents];
__device__ unsigned long long g_cta_times[2 * 2048 * 12];
#define DPS_CTA_STAMP(ev)                                                                          \
    do {                                                                                           \
        const int cta_ = blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z);           \
        if (threadIdx.x == 64 && cta_ < 2048) g_cta_times[(prm.trace_slot * 2048 + cta_) * 12 + (ev)] = global_timer_ns(); \
    } while (0)
#define DPS_CTA_STAMP_T(ev, tid)                                                                   \
    do {                                                                                           \
        const int cta_ = blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z);           \
        if (threadIdx.x == (tid) && cta_ < 2048)                                                   \
            g_cta_times[(prm.trace_slot * 2048 + cta_) * 12 + (ev)] = global_timer_ns();           \
    } while (0)
#ifdef DPS_TRACE_BLOCKS
#define DPS_STAMP(ev, i)                                                                          \
    do {                                                                                          \
        if (blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0 && (threadIdx.x & 31) == 0 &&   \
            (i) < kTraceBlocks)                                                                   \
            g_trace[(i) * kTraceEvents + (ev)] = clock64();                                       \
    } while (0)
#else
#define DPS_STAMP(ev, i) do { } while (0)
#endif
#else
#define DPS_STAMP(ev, i) do { } while (0)
#define DPS_CTA_STAMP(ev) do { } while (0)
#define DPS_CTA_STAMP_T(ev, tid) do { } while (0)
#endif

// Grouped (MoE) launches: blockIdx.y indexes a list of token tiles built on the device by the
// routing pre-pass; each entry is (expert, first sorted row, rows in the tile, unused).
struct GroupedParams {
    const int4* tiles;
    const int32_t* num_tiles;
    const int32_t* sorted_rows;   // sorted position -> caller's row id
    uint32_t e5m2[32];            // bit e set: expert e is E5M2 (truncated or rounded)
    uint32_t rounded[32];         // bit e set: expert e is a rounded nest (full mode only; fast mode reads P alike)
};

struct UmmaParams {
    __half* y;
    int M, N, K;
    int64_t ldy;     // elements from one token's row of y to the next
    int rows;        // LOW: weight rows of a tile (a multiple of 8)
    int num_stages;
    int split;       // K split = cluster size along z; partial tiles are summed through DSMEM
    int red_offset;  // byte offset (from the aligned base of dynamic smem) of the split-K mailbox
    int x_offset;    // byte offset of the activation slots (tiles whose activations do not ride in the stages)
    int x_slots;     // activation slots (tiles that keep the activations apart from the plane ring)
    int* status;
#ifdef DPS_TRACE
    int trace_slot;  // which half of the CTA time table this launch writes
#endif
};

// Two floats -> packed FP16 pair (first in the low half), round to nearest even.
__device__ __forceinline__ uint32_t pack_half2(float lo, float hi) {
    const __half2 h = __floats2half2_rn(lo, hi);
    return *reinterpret_cast<const uint32_t*>(&h);
}

// What a zip warp needs to know about its CTA's pipeline.
struct ZipCtx {
    int group, warp, lane, row, num_kb, num_stages, stage_bytes, plane_bytes;
    uint32_t smem_base, tmem_a, lane_base, sw;
    uint64_t *bar_full, *bar_empty, *bar_a_full, *bar_a_empty;
};

// Zip loop of one warp: for each of its K blocks, wait for the planes to land and for the A slot
// to be free, rebuild 128 FP16 weights of this thread's row from the plane bytes and store them
// into tensor memory.  Returns false if a wait timed out.
//
// EARLY: the stage holds planes only, so it is handed back as soon as this warp has it in registers.
template <int ENC, bool FULL, int TN, bool EARLY = false>
__device__ __forceinline__ bool zip_blocks(const ZipCtx& z) {
    constexpr int kBlockK = block_k(FULL, TN);
    constexpr int kACols = kBlockK / 2;
    bool ok = true;
    // Ring positions are advanced incrementally (no division in the loop).  Every stage and every A
    // slot always belongs to the same zip group, so that each waiter sees every phase of the barriers
    // it waits on: stage s belongs to group s % 2 (any ring depth; with an even ring that is simply
    // alternate K blocks), and group g owns the A slots g, g + 2, ... below the slot count, which
    // it uses in turn.
    constexpr int kTotalSlots = a_slots_max(FULL, TN);
    const int my_slots = (kTotalSlots - z.group + 1) / 2;   // 1 or 2
    int s = 0;
    uint32_t s_parity = 0;             // phase parity of stage s
    int cnt = 0;                       // K blocks this group has rebuilt so far
    for (int i = 0; i < z.num_kb && ok; ++i, s = (s + 1 == z.num_stages) ? 0 : s + 1, s_parity ^= (s == 0)) {
        if ((s & 1) != z.group) continue;
        const int turn = my_slots == 2 ? (cnt & 1) : 0;
        const int a = z.group + 2 * turn;
        const uint32_t a_parity = (uint32_t)(my_slots == 2 ? (cnt >> 1) : cnt) & 1u;
        ++cnt;
        if (z.warp == 2 + 4 * z.group) DPS_STAMP(4, i);
        ok = mbar_wait(smem_u32(&z.bar_full[s]), s_parity);
        ok = __all_sync(0xFFFFFFFFu, ok);
        if (!ok) break;
        if (z.warp == 2 + 4 * z.group) DPS_STAMP(5, i);
        // Read and rebuild the weights FIRST, into registers: that needs the stage, not the A slot,
        // so it overlaps the MMAs that are still reading the slot's previous contents.
        const uint32_t prow = z.smem_base + (uint32_t)s * z.stage_bytes +
                              (uint32_t)z.row * kBlockK;
        uint32_t h[kACols];
#pragma unroll
        for (int c = 0; c < kBlockK / 16; ++c) {
            const uint32_t off = ((uint32_t)c ^ z.sw) * 16u;   // sw already reduced for the swizzle width
            uint4 pv, rv = make_uint4(0, 0, 0, 0);
            asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];"
                         : "=r"(pv.x), "=r"(pv.y), "=r"(pv.z), "=r"(pv.w)
                         : "r"(prow + off));
            if (FULL)
                asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];"
                             : "=r"(rv.x), "=r"(rv.y), "=r"(rv.z), "=r"(rv.w)
                             : "r"(prow + z.plane_bytes + off));
            uint32_t h8[8];
            if (FULL) join16<ENC, FULL>(pv, rv, h8);
            else fast16<ENC>(pv, h8);   // E4M3: 2^8 times the weights, undone in the epilogue
#pragma unroll
            for (int j = 0; j < 8; ++j) h[c * 8 + j] = h8[j];
        }
        if (EARLY) {
            __syncwarp();
            if (z.lane == 0) mbar_arrive(smem_u32(&z.bar_empty[s]));
        }
        ok = mbar_wait(smem_u32(&z.bar_a_empty[a]), a_parity ^ 1u);   // now the slot must be free
        ok = __all_sync(0xFFFFFFFFu, ok);
        if (!ok) break;
        if (z.warp == 2 + 4 * z.group) DPS_STAMP(6, i);
        tc_fence_after_sync();
#pragma unroll
        for (int t = 0; t < kACols / 32; ++t) {
            uint32_t part[32];
#pragma unroll
            for (int j = 0; j < 32; ++j) part[j] = h[t * 32 + j];
            tmem_st_32x32b_x32(z.tmem_a + z.lane_base + (uint32_t)(a * kACols + t * 32), part);
        }
        if (z.warp == 2 + 4 * z.group) DPS_STAMP(7, i);
        tmem_wait_st();
        tc_fence_before_sync();
        __syncwarp();
        if (z.lane == 0) {
            mbar_arrive(smem_u32(&z.bar_a_full[a]));
            if (!EARLY) mbar_arrive(smem_u32(&z.bar_empty[s]));
        }
        if (z.warp == 2 + 4 * z.group) DPS_STAMP(8, i);
    }
    return ok;
}

// ENC == 0 (grouped launches only): the encoding is a per-expert run-time value.
// LOW: tiles of less than kTileRows rows (see low_rows), K not split; a template argument because the others take a run-time
// height for 0.3 % of their time.
template <int ENC, bool FULL, int TN, bool GROUPED, bool LOW>
__global__ void __launch_bounds__(kThreads, 2)
umma_linear_kernel(const __grid_constant__ CUtensorMap map_p, const __grid_constant__ CUtensorMap map_r,
                   const __grid_constant__ CUtensorMap map_x, const UmmaParams prm, const GroupedParams gp) {
    constexpr int kBlockK = block_k(FULL, TN);
    constexpr int kXAtoms = kBlockK / 64;    // the x tile is stored as 64-element (128-byte) swizzle atoms
    constexpr int kACols = kBlockK / 2;      // TMEM columns of one A slot (two FP16 per column)
    constexpr bool kXS = x_slots(FULL, GROUPED, TN) > 0;   // the activations have slots of their own ...
    const int xs_n = prm.x_slots;                               // ... this many (chosen per launch: what fits)
    constexpr int kXBytes = x_tile_bytes(FULL, TN);
    const int rows = LOW ? prm.rows : kTileRows, quarters = (rows + 31) / 32;   // quarters of the lanes that hold rows
    const int plane_bytes = rows * kBlockK, x_offset = plane_bytes * (FULL ? 2 : 1);
    const int stage = x_offset + (kXS ? 0 : kXBytes);
    constexpr uint32_t kCols = tmem_cols(FULL, TN);
    static_assert(kCols <= 256, "two CTAs share the tensor memory of an SM");

    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t bar_full[kMaxStages];
    __shared__ __align__(8) uint64_t bar_empty[kMaxStages];
    __shared__ __align__(8) uint64_t bar_a_full[kMaxAStages];
    __shared__ __align__(8) uint64_t bar_a_empty[kMaxAStages];
    __shared__ __align__(8) uint64_t bar_d_full;
    __shared__ __align__(8) uint64_t bar_x_full[kMaxXSlots];
    __shared__ __align__(8) uint64_t bar_x_empty[kMaxXSlots];
    __shared__ __align__(8) uint64_t bar_dep;
    __shared__ uint32_t tmem_base_slot;
    __shared__ int s_rows[GROUPED ? TN : 1];   // grouped launches: row ids of the tile's tokens

    grid_launch_dependents();  // the next kernel's prologue may overlap this kernel's tail
    DPS_CTA_STAMP(0);
#ifdef DPS_TRACE
    {
        unsigned smid_;
        asm volatile("mov.u32 %0, %%smid;" : "=r"(smid_));
        const int cta_ = blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z);
        if (threadIdx.x == 64 && cta_ < 2048) g_cta_times[(prm.trace_slot * 2048 + cta_) * 12 + 5] = smid_;
    }
#endif
    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int num_stages = prm.num_stages;
    // Tile order (dense launches with several token tiles): CTAs are handed out x-fastest, so walk
    // groups of 8 row tiles x all token tiles.  The CTAs running at any moment then share 8 row
    // tiles of planes and a few dozen activation tiles, which stay in L2, instead of sweeping
    // the whole weight matrix once per token tile (measured: 1.04 GB of DRAM reads for a
    // 100 MB full-mode QKV layer at 2048 tokens before this, because P + R no longer fit in L2).
    int row_tile = blockIdx.x, tok_tile = blockIdx.y;
    if (!GROUPED && gridDim.y > 1) {
        constexpr int kRowGroup = 8;
        const int lin = blockIdx.x + gridDim.x * blockIdx.y;
        const int per_group = kRowGroup * gridDim.y;
        const int group = lin / per_group, within = lin % per_group;
        const int rows_here = min(kRowGroup, (int)gridDim.x - group * kRowGroup);
        row_tile = group * kRowGroup + within % rows_here;
        tok_tile = within / rows_here;
    }
    const int n0 = row_tile * rows;
    int m0 = tok_tile * TN;          // first token (dense) / first sorted row (grouped) of the tile
    int tile_tokens = TN;            // valid token columns of the tile (grouped)
    int plane_row0 = n0;             // first plane row of the tile in the [E * N][K] view
    bool e5m2 = (ENC == kEncE5M2);
    bool rounded = false;         // grouped launches: this tile's expert is a rounded nest (full mode)
    if (GROUPED) {
        grid_dependency_wait();      // the tile list comes from the routing pre-pass
        if ((int)blockIdx.y >= *gp.num_tiles) return;
        const int4 t = gp.tiles[blockIdx.y];
        m0 = t.y;
        tile_tokens = t.z;
        plane_row0 = t.x * prm.N + n0;
        e5m2 = (gp.e5m2[t.x >> 5] >> (t.x & 31)) & 1u;
        rounded = FULL && ((gp.rounded[t.x >> 5] >> (t.x & 31)) & 1u);
    }
    // UMMA N of this tile.  A grouped tile multiplies only the token columns it has (rounded up to
    // 16): at 64-96 tokens per expert a fast-mode MoE layer sits at the ridge between HBM and the
    // tensor pipe, and padded columns are tensor time.  The activation box still brings TN rows.
    const int mma_n = GROUPED ? min(TN, (tile_tokens + 15) & ~15) : TN;
    const uint32_t idesc = umma_idesc_f16(kTileRows, mma_n);
    const int total_kb = (prm.K + kBlockK - 1) / kBlockK;
    const int split = LOW ? 1 : prm.split;
    const int rank = (split > 1) ? (int)cluster_ctarank() : 0;   // == blockIdx.z
    // K blocks are dealt round-robin to the CTAs of the cluster: at any moment the cluster reads
    // `split` adjacent 64-byte pieces of each weight row, which DRAM serves as one longer burst.
    const int num_kb = (total_kb - rank + split - 1) / split;

    if (threadIdx.x == 0) {
        for (int s = 0; s < num_stages; ++s) {
            mbar_init(smem_u32(&bar_full[s]), 1);
            // the zip warps of a reader group, one for each quarter, + 1 tcgen05.commit; a stage that holds planes
            // only (the activations have slots) is read by the zip warps alone
            mbar_init(smem_u32(&bar_empty[s]), kXS ? quarters : quarters + 1);
        }
        for (int a = 0; a < kMaxAStages; ++a) {
            mbar_init(smem_u32(&bar_a_full[a]), quarters);
            mbar_init(smem_u32(&bar_a_empty[a]), 1);
        }
        mbar_init(smem_u32(&bar_d_full), 1);
        for (int a = 0; a < kMaxXSlots; ++a) {
            mbar_init(smem_u32(&bar_x_full[a]), 1);
            mbar_init(smem_u32(&bar_x_empty[a]), 1);   // the tcgen05.commit behind the MMAs that read the slot
        }
        mbar_init(smem_u32(&bar_dep), 1);
        fence_barrier_init();
        prefetch_tensormap(&map_p);
        if (FULL) prefetch_tensormap(&map_r);
        prefetch_tensormap(&map_x);
    }
    if (warp == 1) tmem_alloc(smem_u32(&tmem_base_slot), kCols);
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    DPS_CTA_STAMP(1);
    const uint32_t tmem_base = tmem_base_slot;
    const uint32_t tmem_d = tmem_base;           // TN accumulator columns
    const uint32_t tmem_a = tmem_base + TN; // A ring: slots of kACols columns of packed FP16 pairs

    // Split-K sums: every CTA owns the tokens c with c % split == rank and has a mailbox
    // mail[source rank][slot = c / split][row] in its own shared memory, outside the stage ring; peers
    // store their partial sums straight into it, one cluster barrier later the owner adds them in
    // rank order.
    float* red = reinterpret_cast<float*>(smem_raw + (smem_base - smem_u32(smem_raw)));
    const uint32_t mail_addr = smem_base + (uint32_t)prm.red_offset;
    const int slots = (TN + split - 1) / split;

    bool ok = true;
    if (warp == 0) {
        // ---------------- TMA producer (whole warp converged, one elected lane issues) ----------------
        // First pass over the ring.  The planes are model state: (dense launches) their loads are
        // issued BEFORE the dependency wait, so that the ring fills while the preceding kernel
        // drains; only the activations -- that kernel's output in a decoder -- wait for it.  A
        // stage's barrier expects the bytes of both, so it completes when the later one lands.
        const int first = num_kb < num_stages ? num_kb : num_stages;
        auto load_planes = [&](int i, int s) {
            const uint32_t full = smem_u32(&bar_full[s]);
            const uint32_t dst = smem_base + (uint32_t)(s * stage);
            const int k = (rank + i * split) * kBlockK;
            mbar_arrive_expect_tx(full, (uint32_t)stage);
            tma_load_2d(dst, &map_p, full, k, plane_row0);
            if (FULL) tma_load_2d(dst + plane_bytes, &map_r, full, k, plane_row0);
        };
        auto load_x = [&](int i, int s) {       // activation tile of K block i, riding in stage s
            const uint32_t full = smem_u32(&bar_full[s]);
            const uint32_t dst = smem_base + (uint32_t)(s * stage);
            const int k = (rank + i * split) * kBlockK;
#pragma unroll
            for (int t = 0; t < kXAtoms; ++t)
                tma_load_2d(dst + x_offset + (uint32_t)(t * TN * 128), &map_x, full, k + t * 64, m0);
        };
        auto load_x_slot = [&](int j, int slot) {   // activation tile of K block j into its own slot
            const uint32_t full = smem_u32(&bar_x_full[slot]);
            const uint32_t dst = smem_base + (uint32_t)prm.x_offset + (uint32_t)(slot * kXBytes);
            const int k = (rank + j * split) * kBlockK;
            mbar_arrive_expect_tx(full, (uint32_t)kXBytes);
#pragma unroll
            for (int t = 0; t < kXAtoms; ++t)
                tma_load_2d(dst + (uint32_t)(t * TN * 128), &map_x, full, k + t * 64, m0);
        };
        // How much of that a tile with activation slots does ahead of the dependency (tuning knob): 0 nothing,
        // 1 the first ring pass, 2 also refills of stages the zip warps hand back, 3 also the L2 prefetch.
        constexpr int kPre = kXS ? DPS_PRE_DEP : 3;
        if (!GROUPED && elect_one()) {
            for (int i = 0; kPre >= 1 && i < first; ++i) load_planes(i, i);
            // ... and the plane tiles of the second pass are pulled into L2 meanwhile.
            // (A rolling L2 prefetch further ahead during the main loop was measured slower.)
            const int ahead = kPre >= 3 ? (num_kb < 2 * num_stages ? num_kb : 2 * num_stages) : 0;
            for (int i = first; i < ahead; ++i) {
                const int k = (rank + i * split) * kBlockK;
                tma_prefetch_l2_2d(&map_p, k, plane_row0);
                if (FULL) tma_prefetch_l2_2d(&map_r, k, plane_row0);
            }
        }
        __syncwarp();
        DPS_CTA_STAMP_T(8, 0);
        // grouped launches waited before reading the tile list; with activation slots the MMA warp waits and
        // reports on bar_dep, so that this warp can go on requesting planes meanwhile
        if (!GROUPED && !kXS) grid_dependency_wait();
        if (!kXS) DPS_CTA_STAMP_T(9, 0);
        if (!kXS && elect_one()) {
            for (int i = 0; i < first; ++i) {
                if (GROUPED) load_planes(i, i);
                load_x(i, i);
            }
        }
        __syncwarp();
        // Steady state without activation slots: wait for stage s to be free, refill it (planes and
        // activations of K block i).
        int s = first == num_stages ? 0 : first;
        uint32_t ph = first == num_stages ? 1u : 0u;
        int issued = first;
        for (int i = first; !kXS && i < num_kb && ok; ++i, s = (s + 1 == num_stages) ? 0 : s + 1, ph ^= (s == 0)) {
            ok = mbar_wait(smem_u32(&bar_empty[s]), ph ^ 1u);
            ok = __all_sync(0xFFFFFFFFu, ok);
            if (!ok) break;
            DPS_STAMP(0, i);
            if (elect_one()) {
                load_planes(i, s);
                load_x(i, s);
            }
            __syncwarp();
            ++issued;
        }
        if (!kXS) drain_copies(bar_full, (uint32_t)issued, (uint32_t)num_stages);
        // Steady state with activation slots: two streams with different consumers.  A plane stage is free as
        // soon as its zip group holds it in registers; an activation slot is free when the MMAs that read it
        // are complete, several K blocks later.  One loop serves both by PROBING (test_wait never suspends)
        // whichever barrier comes next in each stream, so that neither stream waits for the other's consumer;
        // the clock is read once in a while to keep the wait bounded.
        if (kXS) {
            int ip = kPre >= 1 ? first : 0, ix = 0;                     // next K block of each stream
            int sp = ip == num_stages ? 0 : ip, sx = 0;                 // its stage / slot
            // parity of the "free" phase awaited there (a fresh barrier passes a wait for the phase before its first)
            uint32_t php = ip == num_stages ? 0u : 1u, phx = 0u;
            bool dep = false;                                           // the preceding kernel's output may be read
            uint32_t idle = 0;
            unsigned long long t0 = 0;
            while ((ip < num_kb || ix < num_kb) && ok) {
                bool progress = false;
                if (ip < num_kb && (kPre >= 2 || dep) &&
                    __any_sync(0xFFFFFFFFu, mbar_test_wait(smem_u32(&bar_empty[sp]), php))) {
                    DPS_STAMP(0, ip);
                    if (elect_one()) load_planes(ip, sp);
                    __syncwarp();
                    ++ip;
                    sp = (sp + 1 == num_stages) ? 0 : sp + 1;
                    php ^= (sp == 0);
                    progress = true;
                }
                if (!dep && __any_sync(0xFFFFFFFFu, mbar_test_wait(smem_u32(&bar_dep), 0u))) {
                    grid_dependency_wait();     // returns at once; orders this warp's loads behind the dependency
                    DPS_CTA_STAMP_T(9, 0);
                    dep = true;
                }
                if (dep && ix < num_kb &&
                    (ix < xs_n || __any_sync(0xFFFFFFFFu, mbar_test_wait(smem_u32(&bar_x_empty[sx]), phx)))) {
                    if (elect_one()) load_x_slot(ix, sx);
                    __syncwarp();
                    ++ix;
                    sx = (sx + 1 == xs_n) ? 0 : sx + 1;
                    if (sx == 0 && ix > xs_n) phx ^= 1u;
                    progress = true;
                }
                if (progress) {
                    idle = 0;
                } else if ((++idle & 1023u) == 0) {
                    const unsigned long long now = global_timer_ns();
                    if (idle == 1024u) t0 = now;
                    else if (now - t0 > kWaitLimitNs) ok = false;
                }
            }
            drain_copies(bar_full, (uint32_t)ip, (uint32_t)num_stages);
            drain_copies(bar_x_full, (uint32_t)ix, (uint32_t)xs_n);
        }
    } else if (warp == 1) {
        // ---------------- MMA issuer (whole warp converged, one elected lane issues) ----------------
        constexpr int kTotalSlots = a_slots_max(FULL, TN);
        if (kXS) {
            // idle until the first activations arrive anyway: waits for the preceding kernel on the producer's behalf
            grid_dependency_wait();
            if (lane == 0) mbar_arrive(smem_u32(&bar_dep));
            __syncwarp();
        }
        {
            // Stage s belongs to zip group s % 2, which rotates through its own A slots (see zip_blocks); the
            // activation tile rides in the stage or sits in a slot of its own (K block i: slot i % slots).  The zip warps waited for the stage's
            // TMA loads before they arrived on a_full, so a tile inside the stage is complete once a_full is;
            // a tile in a slot has a barrier of its own.
            int s = 0, xslot = 0;
            uint32_t xparity = 0, cnt0 = 0, cnt1 = 0;   // K blocks taken from each zip group so far
            for (int i = 0; i < num_kb && ok; ++i, s = (s + 1 == num_stages) ? 0 : s + 1) {
                constexpr int g0_slots = (kTotalSlots + 1) / 2, g1_slots = kTotalSlots / 2;   // 1 or 2 each
                int a;
                uint32_t a_parity;
                if ((s & 1) == 0) {
                    a = g0_slots == 2 ? 2 * (int)(cnt0 & 1u) : 0;
                    a_parity = (g0_slots == 2 ? cnt0 >> 1 : cnt0) & 1u;
                    ++cnt0;
                } else {
                    a = g1_slots == 2 ? 1 + 2 * (int)(cnt1 & 1u) : 1;
                    a_parity = (g1_slots == 2 ? cnt1 >> 1 : cnt1) & 1u;
                    ++cnt1;
                }
                const uint32_t xbase = kXS ? smem_base + (uint32_t)prm.x_offset + (uint32_t)(xslot * kXBytes)
                                           : smem_base + (uint32_t)(s * stage) + x_offset;
                DPS_STAMP(1, i);
                ok = mbar_wait(smem_u32(&bar_a_full[a]), a_parity);
                if (i == 0) DPS_CTA_STAMP_T(11, 32);
                DPS_STAMP(9, i);
                if (kXS && ok) ok = mbar_wait(smem_u32(&bar_x_full[xslot]), xparity);
                ok = __all_sync(0xFFFFFFFFu, ok);
                if (!ok) break;
                DPS_STAMP(2, i);
                if (i == 0) DPS_CTA_STAMP_T(10, 32);
                tc_fence_after_sync();
                if (elect_one()) {
#pragma unroll
                    for (int j = 0; j < kBlockK / 16; ++j) {
                        // 16 K elements = 32 bytes inside the 128-byte swizzle atom (j / 4)
                        const uint64_t bdesc = umma_desc_k_sw128(xbase + (uint32_t)((j >> 2) * TN * 128)) +
                                               (uint64_t)((j & 3) * 2);
                        umma_f16_ts(tmem_d, tmem_a + (uint32_t)(a * kACols + j * 8), bdesc, idesc,
                                    (i > 0 || j > 0) ? 1u : 0u);
                    }
                    DPS_STAMP(10, i);
                    if (kXS) umma_commit(smem_u32(&bar_x_empty[xslot]));   // the slot may be refilled ...
                    else umma_commit(smem_u32(&bar_empty[s]));             // ... or the stage that holds the tile
                    umma_commit(smem_u32(&bar_a_empty[a]));
                    if (i == num_kb - 1) umma_commit(smem_u32(&bar_d_full));
                }
                __syncwarp();
                DPS_STAMP(3, i);
                if (kXS) {
                    xslot = (xslot + 1 == xs_n) ? 0 : xslot + 1;
                    xparity ^= (xslot == 0);
                }
            }
        }
    } else {
        // ---------------- zip warps: planes -> FP16 -> tensor memory; then epilogue ----------------
        const int group = (warp - 2) >> 2;
        const int q = warp & 3;                  // TMEM lane quarter this warp may touch
        const int row = q * 32 + lane;           // weight row inside the tile
        const int zip_row = min(row, rows - 1);  // (lanes without a row repeat the last one: nobody reads theirs)
        const uint32_t lane_base = (uint32_t)(q * 32) << 16;
        ZipCtx zc;
        zc.group = group; zc.warp = warp; zc.lane = lane; zc.row = zip_row;
        zc.num_kb = num_kb; zc.num_stages = num_stages; zc.stage_bytes = stage; zc.plane_bytes = plane_bytes;
        zc.smem_base = smem_base; zc.tmem_a = tmem_a; zc.lane_base = lane_base;
        // TMA swizzle of the plane tiles: 128-byte rows: 16-byte chunk index ^= row % 8;
        // 64-byte rows: chunk index ^= (row / 2) % 4
        zc.sw = kBlockK == 128 ? (uint32_t)(zip_row & 7) : (uint32_t)((zip_row >> 1) & 3);
        zc.bar_full = bar_full; zc.bar_empty = bar_empty; zc.bar_a_full = bar_a_full; zc.bar_a_empty = bar_a_empty;
        // grouped launches: the callers' row ids of the tile's tokens, fetched before the zip loop (which
        // hides the latency) rather than in front of every store of the epilogue
        if (GROUPED && (int)threadIdx.x - 64 < tile_tokens) s_rows[threadIdx.x - 64] = gp.sorted_rows[m0 + (int)threadIdx.x - 64];
        if constexpr (GROUPED) {
            // encoding known only at run time (one per expert): uniform branch per CTA
            if (FULL && rounded)
                ok = e5m2 ? zip_blocks<kEncE5M2R, FULL, TN>(zc) : zip_blocks<kEncE4M3R, FULL, TN>(zc);
            else
                ok = e5m2 ? zip_blocks<kEncE5M2, FULL, TN>(zc) : zip_blocks<kEncE4M3, FULL, TN>(zc);
        } else {
            if (q < quarters) ok = zip_blocks<ENC, FULL, TN, kXS>(zc);
        }
        // E4M3 fast mode multiplied with 2^8 times the weights (hardware FP8 conversion)
        const float out_scale = (!FULL && !e5m2) ? 0.00390625f : 1.0f;
        if (split == 1) {
            // ---- epilogue without a K split: D -> FP16 -> shared memory -> y, by all zip warps ----
            // The accumulator is drained into a [token][row] FP16 tile that overlays the idle stage
            // ring (every load has been consumed once the last MMA is complete), and then written
            // out with 16-byte stores: one warp instruction covers 512 contiguous bytes of a row
            // of y.  Storing straight from the accumulator registers (2 bytes per thread per
            // token, 64 bytes per warp instruction) took 5 us per 256 x 96 tile, with nothing
            // else running on the SM.
            constexpr int kColsPerGroup = TN < 32 ? TN : TN / 2;   // the groups share the columns
            const int ncols = GROUPED ? tile_tokens : min(TN, prm.M - m0);     // token columns that exist
            if (ok) ok = mbar_wait(smem_u32(&bar_d_full), 0u);
            ok = __all_sync(0xFFFFFFFFu, ok);
            DPS_CTA_STAMP(2);
            const bool drains = TN >= 32 || group == 0;
            if (ok && drains) {
                tc_fence_after_sync();
                const int cbeg = TN >= 32 ? group * kColsPerGroup : 0;
#pragma unroll
                for (int cc = 0; cc < kColsPerGroup; cc += 16) {
                    const int c0 = cbeg + cc;
                    if (c0 >= ncols) break;                       // warp-uniform
                    uint32_t v[16];
                    tmem_ld_32x32b_x16(tmem_d + lane_base + (uint32_t)c0, v);
                    tmem_wait_ld();
#pragma unroll
                    for (int j = 0; j < 16; ++j) {
                        const __half h = __float2half_rn(__uint_as_float(v[j]) * out_scale);
                        const uint32_t addr = smem_base + (uint32_t)(((c0 + j) * kTileRows + row) * 2);
                        asm volatile("st.shared.u16 [%0], %1;" ::"r"(addr), "h"(__half_as_ushort(h)) : "memory");
                    }
                }
            }
            named_barrier_sync(1, kZipGroups * 128);              // the zip warps only
            DPS_CTA_STAMP(3);
            if (ok) {
                constexpr int kChunks = kTileRows / 8;             // 16-byte pieces of one token's rows
                const int zt = (int)threadIdx.x - 64;             // index among the zip threads
                for (int item = zt; item < ncols * kChunks; item += kZipGroups * 128) {
                    const int c = item / kChunks, q = item % kChunks;
                    const int n = n0 + q * 8;
                    if (q * 8 >= rows || n >= prm.N) continue;    // both are multiples of 8: a piece is in or out
                    const int m = GROUPED ? s_rows[c] : m0 + c;
                    uint4 val;
                    asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];"
                                 : "=r"(val.x), "=r"(val.y), "=r"(val.z), "=r"(val.w)
                                 : "r"(smem_base + (uint32_t)((c * kTileRows + q * 8) * 2)));
                    *reinterpret_cast<uint4*>(prm.y + m * prm.ldy + n) = val;
                }
            }
        } else if (group == 0 || TN >= 32) {
            // ---- epilogue with a K split: partial sums -> mailbox / red; the zip groups share the columns ----
            constexpr int kColsPerGroup = TN >= 32 ? TN / 2 : TN;
            const int cbeg = TN >= 32 ? group * kColsPerGroup : 0;
            if (ok) ok = mbar_wait(smem_u32(&bar_d_full), 0u);
            ok = __all_sync(0xFFFFFFFFu, ok);
            DPS_CTA_STAMP(2);
            // The partial tile first goes into this CTA's own shared memory as red[token][row], over the idle
            // ring (every load has been consumed), then out to the owners' mailboxes four rows at a time --
            // sixteen scalar remote stores per thread straight out of the accumulator registers took 0.75 us
            // of every launch.
            if (ok) {
                tc_fence_after_sync();
#pragma unroll
                for (int cc = 0; cc < kColsPerGroup; cc += 16) {
                    const int c0 = cbeg + cc;
                    uint32_t v[16];
                    tmem_ld_32x32b_x16(tmem_d + lane_base + (uint32_t)c0, v);
                    tmem_wait_ld();
#pragma unroll
                    for (int j = 0; j < 16; ++j)
                        red[(c0 + j) * kTileRows + row] = __uint_as_float(v[j]) * out_scale;
                }
            }
            constexpr int kPushers = TN >= 32 ? kZipGroups * 128 : 128;   // the threads in this branch
            asm volatile("bar.sync 2, %0;" ::"n"(kPushers) : "memory");
            if (ok) {
                const int zt = (int)threadIdx.x - 64;
                for (int e = zt; e < TN * (kTileRows / 4); e += kPushers) {
                    const int c = e / (kTileRows / 4), r4 = (e % (kTileRows / 4)) * 4;
                    const int owner = c % split, slot = c / split;
                    const float4 val = *reinterpret_cast<const float4*>(&red[c * kTileRows + r4]);
                    const uint32_t local = mail_addr + (uint32_t)(((rank * slots + slot) * kTileRows + r4) * 4);
                    st_cluster_v4_f32(map_to_cta(local, (uint32_t)owner), val);
                }
            }
        }
    }
    if (!ok) atomicExch(prm.status, (int)DPS_ERR_CUDA);
    if (split > 1) DPS_CTA_STAMP(3);

    if (split > 1) {
        __syncthreads();
        cluster_sync_all();  // release/acquire: every peer's stores into this CTA's mailbox are visible
        DPS_CTA_STAMP(4);
        const float* mail = reinterpret_cast<const float*>(smem_raw + (smem_base - smem_u32(smem_raw)) + prm.red_offset);
        // one item = 8 consecutive rows of one owned token: 16 bytes of y
        for (int e = threadIdx.x; e < slots * (kTileRows / 8); e += kThreads) {
            const int slot = e / (kTileRows / 8), r = (e % (kTileRows / 8)) * 8;
            const int c = slot * split + rank;
            const int m = m0 + c, n = n0 + r;
            if (c >= TN || m >= prm.M || n >= prm.N) continue;   // N is a multiple of 8
            float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
            for (int j = 0; j < split; ++j) {
                const float4* src = reinterpret_cast<const float4*>(mail + (j * slots + slot) * kTileRows + r);
                const float4 a = src[0], b = src[1];
                acc[0] += a.x; acc[1] += a.y; acc[2] += a.z; acc[3] += a.w;
                acc[4] += b.x; acc[5] += b.y; acc[6] += b.z; acc[7] += b.w;
            }
            uint4 out;
            out.x = pack_half2(acc[0], acc[1]);
            out.y = pack_half2(acc[2], acc[3]);
            out.z = pack_half2(acc[4], acc[5]);
            out.w = pack_half2(acc[6], acc[7]);
            *reinterpret_cast<uint4*>(prm.y + m * prm.ldy + n) = out;
        }
    }
    DPS_CTA_STAMP(6);
    tc_fence_before_sync();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after_sync();
        tmem_dealloc(tmem_base, kCols);
    }
    DPS_CTA_STAMP(7);
}

// ---- host side ---------------------------------------------------------------------------------

// Tuning / debugging knob: DPS_FORCE_SPLIT=<1..8> pins the K split.
int forced_split() {
    static const int v = [] {
        const char* e = getenv("DPS_FORCE_SPLIT");
        return e ? atoi(e) : 0;
    }();
    return v;
}

// DPS_TILE_ROWS=64..120 pins the height.
int rows_of_tiles(bool full, int64_t N, int64_t K, int tn) {
    static const int forced = [] { const char* e = getenv("DPS_TILE_ROWS"); return e ? atoi(e) / 8 * 8 : 0; }();
    return forced >= 64 && forced < kTileRows ? forced : low_rows(full, N, K, tn, sm_count());
}

// `plan`, where not null: nothing is launched, *plan receives the turns the launch would take.  prepare_only: all but the launch.
template <int ENC, bool FULL, int TN, bool LOW = false>
cudaError_t launch_tn(const void* x, const uint8_t* p, const uint8_t* r, void* y, int64_t ldy, int64_t M, int64_t N, int64_t K,
                      int* status, cudaStream_t stream, bool prepare_only, int rows = kTileRows, Turns* plan = nullptr) {
    constexpr int kXSlots = x_slots(FULL, false, TN);            // with a split-K mailbox in shared memory
    constexpr int kXSlotsAlone = x_slots_alone(FULL, TN);           // without one (K not split)
    constexpr int kXTile = x_tile_bytes(FULL, TN);
    constexpr int kCtasPerSm = 2;
    constexpr int kSmemTotal = 111 * 1024;
    constexpr int kMailMax = (TN + kMaxSplit) * kTileRows * 4;  // mailbox, worst case
    // Ring depth for a given mailbox size: whatever fits (stage s is rebuilt by zip group s % 2, so
    // odd depths work; they just give the first group one stage more).
    auto stage_of = [](int tile_rows) { return tile_rows * block_k(FULL, TN) * (FULL ? 2 : 1) + (kXSlots ? 0 : kXTile); };
    auto ring_depth = [&](int mail_bytes, int tile_rows) {
        const int x_ring = (mail_bytes > 0 ? kXSlots : kXSlotsAlone) * kXTile;
        const int d = (kSmemTotal - mail_bytes - x_ring) / stage_of(tile_rows);
        return d > 8 ? 8 : d < 2 ? 2 : d;
    };
    const size_t smem_query = (size_t)ring_depth(kMailMax, kTileRows) * stage_of(kTileRows) + kXSlots * kXTile + kMailMax + 1024;
    auto kernel = umma_linear_kernel<ENC, FULL, TN, false, LOW>;
    // CTAs that can be resident at once for each cluster size: per instantiation and per device, filled by
    // the first call on that device and read only after that set-up has returned.
    static int capacity_of[kMaxDevices][kMaxSplit + 1] = {};
    static PerDeviceOnce setup;
    int dev = 0;
    {
        const cudaError_t e0 = setup.run([&] {
            int d = 0;
            cudaGetDevice(&d);
            int* capacity = capacity_of[d];
            cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 224 * 1024);
            if (e != cudaSuccess) return e;
            // Ask for the largest shared-memory carve-out, otherwise the driver may size it for ONE CTA
            // of this kernel and a second CTA never becomes resident on the SM.
            e = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout,
                                     cudaSharedmemCarveoutMaxShared);
            if (e != cudaSuccess) return e;
            if constexpr (LOW) return cudaSuccess;       // never split over K: nobody asks
            for (int s = 1; s <= kMaxSplit; ++s) {
                cudaLaunchConfig_t q = {};
                q.gridDim = dim3(1, 1, (unsigned)s);
                q.blockDim = dim3(kThreads, 1, 1);
                q.dynamicSmemBytes = smem_query;
                cudaLaunchAttribute qa[1];
                qa[0].id = cudaLaunchAttributeClusterDimension;
                qa[0].val.clusterDim.x = 1;
                qa[0].val.clusterDim.y = 1;
                qa[0].val.clusterDim.z = (unsigned)s;
                q.attrs = qa;
                q.numAttrs = 1;
                int clusters = 0;
                if (cudaOccupancyMaxActiveClusters(&clusters, kernel, &q) != cudaSuccess) clusters = 0;
                capacity[s] = clusters * s;
            }
            (void)cudaGetLastError();
            // The query can be more conservative about CTAs per SM than the hardware turns out to be
            // (it reported one where two were measured resident); keep its GPC packing ratios and
            // rescale to the CTAs per SM this kernel is sized for.
            const int slots = sm_count() * kCtasPerSm;
            if (capacity[1] <= 0) capacity[1] = slots;
            const int base = capacity[1];
            for (int s = 1; s <= kMaxSplit; ++s) capacity[s] = (int)((int64_t)capacity[s] * slots / base);
            // With two CTAs per SM a cluster of even size s needs only s / 2 SMs of a GPC, so it packs
            // like a cluster of s / 2 at one CTA per SM (32 row tiles split 8 ways, 256 CTAs, were
            // measured 5-11 % faster than split 6 ways, which the plain rescaling would have chosen).
            for (int s = kMaxSplit; s >= 2; s -= 2)
                if (capacity[s / 2] > capacity[s]) capacity[s] = capacity[s / 2];
            return cudaSuccess;
        }, &dev);
        if (e0 != cudaSuccess) return e0;
    }
    const int* capacity = capacity_of[dev];
    constexpr int kBlockK = block_k(FULL, TN);
    const int64_t tok_tiles = (M + TN - 1) / TN;
    const int total_kb = (int)((K + kBlockK - 1) / kBlockK);
    int split = LOW ? 1 : forced_split();
    if (split <= 0) split = choose_split((N + rows - 1) / rows * tok_tiles, total_kb, capacity, FULL ? 5 : 4);
    if (split > total_kb) split = total_kb;
    if (split > kMaxSplit) split = kMaxSplit;
    if (plan != nullptr) {
        *plan = turns((N + rows - 1) / rows * tok_tiles, split, capacity[1]);
        return cudaSuccess;
    }
    CUtensorMap mp, mr, mx;
    constexpr CUtensorMapSwizzle kPlaneSwizzle = kBlockK == 128 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B;
    constexpr CUtensorMapL2promotion kPromotion = CU_TENSOR_MAP_L2_PROMOTION_L2_256B;
    if (!make_map_2d(&mp, p, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, (uint64_t)N, (uint64_t)K, (uint32_t)rows, kBlockK,
                     kPlaneSwizzle, kPromotion))
        return cudaErrorInvalidValue;
    if (FULL) {
        if (!make_map_2d(&mr, r, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, (uint64_t)N, (uint64_t)K, (uint32_t)rows, kBlockK,
                         kPlaneSwizzle, kPromotion))
            return cudaErrorInvalidValue;
    } else {
        mr = mp;
    }
    if (!make_map_2d(&mx, x, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, (uint64_t)M, (uint64_t)K, TN, 64,
                     CU_TENSOR_MAP_SWIZZLE_128B))
        return cudaErrorInvalidValue;
    if (prepare_only) return cudaSuccess;
    const int64_t row_tiles = (N + rows - 1) / rows;
    // the mailbox exists only when K is split, and then has its exact size
    const int slots = split > 1 ? (TN + split - 1) / split : 0;
    const int mail_bytes = (split > 1 && kMailMax > 0) ? split * slots * kTileRows * 4 : 0;
    const int stages = ring_depth(mail_bytes, rows), stage = stage_of(rows);
    const int xs_n = mail_bytes > 0 ? kXSlots : kXSlotsAlone;
    const int x_ring = xs_n * kXTile;
    const size_t smem = (size_t)stages * stage + x_ring + mail_bytes + 1024;
    if (getenv("DPS_DEBUG"))
        fprintf(stderr, "[dps] umma TN=%d full=%d N=%lld K=%lld M=%lld rows=%d stages=%d split=%d capacity=%d,%d,%d,%d,%d,%d,%d,%d\n",
                TN, (int)FULL, (long long)N, (long long)K, (long long)M, rows, stages, split, capacity[1], capacity[2],
                capacity[3], capacity[4], capacity[5], capacity[6], capacity[7], capacity[8]);
    UmmaParams prm = {};
    prm.y = static_cast<__half*>(y);
    prm.M = (int)M;
    prm.N = (int)N;
    prm.K = (int)K;
    prm.ldy = ldy;
    prm.status = status;
    prm.num_stages = stages;
    prm.split = split;
    prm.rows = rows;
    prm.x_offset = stages * stage;
    prm.x_slots = xs_n;
    prm.red_offset = stages * stage + x_ring;
    prm.status = status;
#ifdef DPS_TRACE
    static int trace_launches = 0;
    prm.trace_slot = (trace_launches++) & 1;
#endif

    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)row_tiles, (unsigned)tok_tiles, (unsigned)split);
    cfg.blockDim = dim3(kThreads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 1;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = (unsigned)split;
    // Programmatic dependent launch: this kernel may start while the previous one drains; it
    // waits (griddepcontrol.wait) before its first global read.
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    GroupedParams gp = {};
    cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, mp, mr, mx, prm, gp);
    count_launch();
    return e;
}

template <int ENC, bool FULL>
cudaError_t launch_enc(const void* x, const uint8_t* p, const uint8_t* r, void* y, int64_t ldy, int64_t M, int64_t N, int64_t K,
                       int* status, cudaStream_t stream, bool prepare_only) {
    if (M <= 32 && forced_split() <= 1) {
        const int rows = rows_of_tiles(FULL, N, K, M <= 16 ? 16 : 32);
        if (rows < kTileRows && M <= 16) return launch_tn<ENC, FULL, 16, true>(x, p, r, y, ldy, M, N, K, status, stream, prepare_only, rows);
        if (rows < kTileRows) return launch_tn<ENC, FULL, 32, true>(x, p, r, y, ldy, M, N, K, status, stream, prepare_only, rows);
    }
    if (M <= 16) return launch_tn<ENC, FULL, 16>(x, p, r, y, ldy, M, N, K, status, stream, prepare_only);
    if (M <= 32) return launch_tn<ENC, FULL, 32>(x, p, r, y, ldy, M, N, K, status, stream, prepare_only);
    // 33 tokens and more (beyond 64 only where the dispatcher prefers two 64-token tiles per 128 rows to CTA pairs)
    return launch_tn<ENC, FULL, 64>(x, p, r, y, ldy, M, N, K, status, stream, prepare_only);
}

}  // namespace

// Byte-matrix tensor map for the other translation units (row-major [rows][cols] bytes, boxes of
// box_rows x 128 bytes, 128-byte swizzle).
bool make_byte_map_sw128(CUtensorMap* map, const void* base, uint64_t rows, uint64_t cols, uint32_t box_rows) {
    return make_map_2d(map, base, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, rows, cols, box_rows, 128, CU_TENSOR_MAP_SWIZZLE_128B);
}

#ifdef DPS_TRACE
extern "C" __attribute__((visibility("default"))) int dps_debug_trace(long long* out, int max_words) {
    const int n = max_words < kTraceBlocks * kTraceEvents ? max_words : kTraceBlocks * kTraceEvents;
    return (int)cudaMemcpyFromSymbol(out, g_trace, sizeof(long long) * n);
}
extern "C" __attribute__((visibility("default"))) int dps_debug_cta_times(unsigned long long* out) {
    return (int)cudaMemcpyFromSymbol(out, g_cta_times, sizeof(unsigned long long) * 2 * 2048 * 12);
}
#endif

namespace {

template <bool FULL, int TN>
cudaError_t launch_grouped_tn(const uint32_t* e5m2_mask, const void* x_sorted, const uint8_t* p, const uint8_t* r,
                              void* y, int64_t A, int64_t N, int64_t K, int32_t E, const void* tiles,
                              const int32_t* num_tiles, const int32_t* sorted_rows, int max_tiles, int* status,
                              cudaStream_t stream) {
    constexpr int kStage = stage_bytes(FULL, TN);
    constexpr int kSmemTotal = 111 * 1024;   // two CTAs per SM
    int stages = kSmemTotal / kStage;
    if (stages > 8) stages = 8;
    if (stages < 2) stages = 2;
    const size_t smem = (size_t)stages * kStage + 1024;
    auto kernel = umma_linear_kernel<0, FULL, TN, true, false>;
    static PerDeviceOnce setup;     // per instantiation and per device
    {
        const cudaError_t e = setup.run([&] {
            cudaError_t a = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 224 * 1024);
            if (a != cudaSuccess) return a;
            return cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout,
                                        cudaSharedmemCarveoutMaxShared);
        });
        if (e != cudaSuccess) return e;
    }
    CUtensorMap mp, mr, mx;
    constexpr int kBlockK = block_k(FULL, TN);
    constexpr CUtensorMapSwizzle kPlaneSwizzle = kBlockK == 128 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B;
    if (!make_map_2d(&mp, p, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, (uint64_t)E * (uint64_t)N, (uint64_t)K, kTileRows,
                     kBlockK, kPlaneSwizzle, CU_TENSOR_MAP_L2_PROMOTION_L2_256B))
        return cudaErrorInvalidValue;
    if (FULL) {
        if (!make_map_2d(&mr, r, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, (uint64_t)E * (uint64_t)N, (uint64_t)K, kTileRows,
                         kBlockK, kPlaneSwizzle, CU_TENSOR_MAP_L2_PROMOTION_L2_256B))
            return cudaErrorInvalidValue;
    } else {
        mr = mp;
    }
    if (!make_map_2d(&mx, x_sorted, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, (uint64_t)A, (uint64_t)K, TN, 64,
                     CU_TENSOR_MAP_SWIZZLE_128B))
        return cudaErrorInvalidValue;
    UmmaParams prm = {};
    prm.y = static_cast<__half*>(y);
    prm.M = (int)A;
    prm.N = (int)N;
    prm.K = (int)K;
    prm.ldy = N;
    prm.num_stages = stages;
    prm.split = 1;
    prm.red_offset = 0;
    prm.status = status;
    GroupedParams gp;
    gp.tiles = static_cast<const int4*>(tiles);
    gp.num_tiles = num_tiles;
    gp.sorted_rows = sorted_rows;
    for (int i = 0; i < 32; ++i) {   // the caller's array holds the E5M2 bits, then the rounded-nest bits
        gp.e5m2[i] = e5m2_mask[i];
        gp.rounded[i] = FULL ? e5m2_mask[32 + i] : 0u;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((N + kTileRows - 1) / kTileRows), (unsigned)max_tiles, 1);
    cfg.blockDim = dim3(kThreads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, mp, mr, mx, prm, gp);
    count_launch();
    return e;
}

}  // namespace

// Token-tile width of grouped launches (below 48 rows per expert): wide enough that an expert with 1.5 times the average
// number of rows (1.33 at 48) still fits one tile, its planes are then streamed once.
int grouped_tile_tokens(int64_t A, int32_t E) {
    const int64_t avg = (A + E - 1) / E;
    const int64_t target = avg + (avg + 1) / 2;
    return target <= 16 ? 16 : target <= 32 ? 32 : 64;
}

cudaError_t launch_umma_grouped(int mode, const uint32_t* e5m2_mask, const void* x_sorted, const uint8_t* p,
                                const uint8_t* r, void* y, int64_t A, int64_t N, int64_t K, int32_t E, int tn,
                                const void* tiles, const int32_t* num_tiles, const int32_t* sorted_rows,
                                int max_tiles, int* status, cudaStream_t stream) {
#define DPS_GROUPED_CASE(TNV)                                                                                         \
    if (tn == TNV)                                                                                                    \
        return mode == DPS_MODE_FULL                                                                                  \
                   ? launch_grouped_tn<true, TNV>(e5m2_mask, x_sorted, p, r, y, A, N, K, E, tiles, num_tiles,         \
                                                  sorted_rows, max_tiles, status, stream)                             \
                   : launch_grouped_tn<false, TNV>(e5m2_mask, x_sorted, p, r, y, A, N, K, E, tiles, num_tiles,        \
                                                   sorted_rows, max_tiles, status, stream);
    DPS_GROUPED_CASE(16)
    DPS_GROUPED_CASE(32)
    DPS_GROUPED_CASE(64)
#undef DPS_GROUPED_CASE
    return cudaErrorInvalidValue;
}

cudaError_t launch_umma_linear(int mode, int enc, const void* x, const uint8_t* p, const uint8_t* r, void* y, int64_t ldy,
                               int64_t M, int64_t N, int64_t K, int* status, cudaStream_t stream, bool prepare_only) {
    const bool full = mode == DPS_MODE_FULL;
    if (!full) enc = base_enc(enc);   // fast mode reads the persistent byte of a rounded nest like any other
    if (enc == kEncE4M3R) return launch_enc<kEncE4M3R, true>(x, p, r, y, ldy, M, N, K, status, stream, prepare_only);
    if (enc == kEncE5M2R) return launch_enc<kEncE5M2R, true>(x, p, r, y, ldy, M, N, K, status, stream, prepare_only);
    if (enc == kEncE4M3)
        return full ? launch_enc<kEncE4M3, true>(x, p, r, y, ldy, M, N, K, status, stream, prepare_only)
                    : launch_enc<kEncE4M3, false>(x, p, r, y, ldy, M, N, K, status, stream, prepare_only);
    return full ? launch_enc<kEncE5M2, true>(x, p, r, y, ldy, M, N, K, status, stream, prepare_only)
                : launch_enc<kEncE5M2, false>(x, p, r, y, ldy, M, N, K, status, stream, prepare_only);
}

cudaError_t tile_turns_64(int mode, int enc, int64_t M, int64_t N, int64_t K, Turns* plan) {
    auto ask = [&](auto launch) { return launch(nullptr, nullptr, nullptr, nullptr, N, M, N, K, nullptr, nullptr, false, kTileRows, plan); };
    const bool full = mode == DPS_MODE_FULL;
    if (!full) enc = base_enc(enc);
    if (enc == kEncE4M3R) return ask(launch_tn<kEncE4M3R, true, 64>);
    if (enc == kEncE5M2R) return ask(launch_tn<kEncE5M2R, true, 64>);
    if (enc == kEncE4M3) return full ? ask(launch_tn<kEncE4M3, true, 64>) : ask(launch_tn<kEncE4M3, false, 64>);
    return full ? ask(launch_tn<kEncE5M2, true, 64>) : ask(launch_tn<kEncE5M2, false, 64>);
}

}  // namespace dps
