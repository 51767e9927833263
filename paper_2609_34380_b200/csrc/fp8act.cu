// Fast mode with FP8 activations: the persistent plane is consumed by the FP8 tensor cores AS IT IS.
//
// Paper: "Mapper: Semi-Unified Memory Abstraction", "Persistent Region" paragraph -- FP8 execution
// can halve memory accesses "or double peak tensor-core throughput with hardware support".  The
// persistent byte of the nested format is a valid FP8 number (E5M2: the fast-mode weight itself;
// E4M3: 2^8 times it), so with activations quantised to E4M3 the layer is a plain FP8 x FP8
// contraction: no rebuilding of weights, both operands straight from shared memory
// (tcgen05.mma kind::f8f6f4, SS form), FP32 accumulation in tensor memory.
//
// Activation quantisation (the paper gives no recipe; per-token dynamic scaling is the reading
// taken): scale[m] = max_k |x[m][k]| / 448 (1 for an all-zero token), q = E4M3(x / scale), round to
// nearest even, saturating; y[m][n] = scale[m] * sum_k q[m][k] * W_fast[n][k].
//
// Kernel: tiles of 256 weight rows x up to 256 tokens, K in blocks of 128 bytes, one persistent CTA PAIR
// (cta_group::2) per two SMs.  In each CTA: warp 0 TMA producer (its 128 rows of P, its half of the
// tokens, 128-byte swizzle), warp 1 MMA issuer (in the first CTA, for both; two accumulators in tensor
// memory), warps 2-5 epilogue of its 128 rows (TMEM -> scale -> FP16 -> shared-memory buffer ->
// 16-byte stores), overlapped with the next tile's MMAs.
#include <cuda.h>
#include <cuda_fp16.h>
#include <cuda_fp8.h>

#include <cstdlib>

#include "dps_internal.h"
#include "sm100.cuh"

namespace dps {

bool make_byte_map_sw128(CUtensorMap* map, const void* base, uint64_t rows, uint64_t cols, uint32_t box_rows);

namespace {

using namespace sm100;

// ---- activation quantisation ------------------------------------------------------------------
constexpr int kQuantThreads = 256;

// One CTA per token: maximum magnitude, scale, then the E4M3 codes.  Rows of up to 8192 elements stay
// in registers between the two passes (four 16-byte pieces per thread); longer rows are read again.
constexpr int kQuantKeep = 4;

__device__ __forceinline__ uint2 quantize8(const uint4& v, float sc) {
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
    uint32_t out[2] = {0u, 0u};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&w[j]));
        const float2 d = make_float2(__fdiv_rn(f.x, sc), __fdiv_rn(f.y, sc));
        const uint32_t pair = (uint32_t)__nv_cvt_float2_to_fp8x2(d, __NV_SATFINITE, __NV_E4M3);   // .x in the low byte
        out[j >> 1] |= pair << ((j & 1) * 16);
    }
    return make_uint2(out[0], out[1]);
}

// (x without __restrict__: its writer may still run when a CTA starts)
__global__ void __launch_bounds__(kQuantThreads)
quantize_activations_kernel(const uint4* x, uint2* q, float* scale, int64_t k8, int* status) {
    __shared__ float s_max[kQuantThreads / 32];
    __shared__ float s_scale;
    grid_launch_dependents();
    grid_dependency_wait();   // the activations are the preceding kernel's output
    const int64_t m = blockIdx.x;
    const uint4* row = x + m * k8;
    const bool keep = k8 <= (int64_t)kQuantKeep * kQuantThreads;
    uint4 held[kQuantKeep];
    float amax = 0.f;
    bool bad = false;
    auto scan = [&](const uint4& v) {
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&w[j]));
            const float a = fabsf(f.x), b = fabsf(f.y);
            bad |= !(a <= 65504.f) || !(b <= 65504.f);   // Inf or NaN
            amax = fmaxf(amax, fmaxf(a, b));
        }
    };
    if (keep) {
#pragma unroll
        for (int u = 0; u < kQuantKeep; ++u) {
            const int64_t i = (int64_t)u * kQuantThreads + threadIdx.x;
            held[u] = make_uint4(0u, 0u, 0u, 0u);
            if (i < k8) held[u] = row[i];
            scan(held[u]);
        }
    } else {
        for (int64_t i = threadIdx.x; i < k8; i += kQuantThreads) scan(row[i]);
    }
    for (int o = 16; o > 0; o >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xFFFFFFFFu, amax, o));
    if (__syncthreads_or(bad) && threadIdx.x == 0) atomicExch(status, (int)DPS_ERR_DATA);
    if ((threadIdx.x & 31) == 0) s_max[threadIdx.x >> 5] = amax;
    __syncthreads();
    if (threadIdx.x == 0) {
        float a = 0.f;
        for (int w = 0; w < kQuantThreads / 32; ++w) a = fmaxf(a, s_max[w]);
        const float sc = a > 0.f ? __fdiv_rn(a, 448.0f) : 1.0f;
        s_scale = sc;
        scale[m] = sc;
    }
    __syncthreads();
    const float sc = s_scale;
    uint2* qrow = q + m * k8;
    if (keep) {
#pragma unroll
        for (int u = 0; u < kQuantKeep; ++u) {
            const int64_t i = (int64_t)u * kQuantThreads + threadIdx.x;
            if (i < k8) qrow[i] = quantize8(held[u], sc);
        }
    } else {
        for (int64_t i = threadIdx.x; i < k8; i += kQuantThreads) qrow[i] = quantize8(row[i], sc);
    }
}

// ---- FP8 x FP8 linear ---------------------------------------------------------------------------
constexpr int kRows = 128;      // weight rows per CTA; a pair's tile has 256 (UMMA M)
constexpr int kBlockBytes = 128;                                  // K per stage (one swizzle atom of bytes)
constexpr int kThreads = 192;
constexpr int kMaxTokens = 256;                                   // tokens per tile (UMMA N): any multiple of 16 up to this
constexpr int kStageBytes = (kRows + kMaxTokens / 2) * kBlockBytes;   // 32 KB: this CTA's rows, its half of the tokens
constexpr int kStages = 6;
constexpr uint32_t kTmemCols = 2 * kMaxTokens;                    // two accumulators

// Instruction descriptor for kind::f8f6f4: FP32 accumulator, K-major operands; formats 0 = E4M3, 1 = E5M2.
__host__ __device__ constexpr uint32_t idesc_f8(int m, int n, int a_format, int b_format) {
    return (1u << 4) | ((uint32_t)a_format << 7) | ((uint32_t)b_format << 10) | ((uint32_t)(n >> 3) << 17) |
           ((uint32_t)(m >> 4) << 24);
}

// D[tmem] (+)= A[smem] * B[smem] over a CTA pair, FP8 operands; issued by ONE thread of the pair's first CTA.
// Descriptors and addresses hold for both CTAs: each brings its 128 rows of A and its half of B's rows.
__device__ __forceinline__ void umma_f8_ss_pair(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                                uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f8f6f4 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}

struct Fp8Params {
    __half* y;
    const float* scale;
    int M, N, K;
    int tokens;    // per tile
    int e5m2;      // the persistent plane is E5M2 (else E4M3, whose bytes read as FP8 are 2^8 times the weights)
    int* status;
};

constexpr int kEpiCols = 32;                                      // token columns per epilogue chunk
constexpr int kEpiBytes = kEpiCols * kRows * 2 + 4 * kMaxTokens * 4;   // behind the ring: four warps' chunks (2 KB each) and scales

// Persistent: one CTA pair per two SMs walks the tiles (groups of 8 row tiles x all token tiles).  What bounds the
// main loop is not the tensor pipe but what an SM can pull out of L2, about 50 bytes a clock: a CTA by itself with
// a 128 x 256 tile needs 48 KB per 512 tensor cycles, a pair with a 256 x 256 tile 32 KB per CTA, since each CTA
// fetches half of the tokens and the tensor cores of both read both halves.  Four Llama-7B linears at 512 / 2048 /
// 8192 tokens: 147 / 413 / 1562 us with single CTAs, 123 / 361 / 1428 us with pairs (2.35 PFLOP/s; from about 2000
// tokens on the 1000 W power cap holds the clock down).
// Two accumulators of 256 columns fill tensor memory, so the MMA warp starts the next tile while the four
// epilogue warps of each CTA drain the previous one.  The epilogue goes through a small buffer, 32 token columns
// at a time: the stage ring never idles.
__global__ void __launch_bounds__(kThreads, 1)
fp8act_linear_kernel(const __grid_constant__ CUtensorMap map_p, const __grid_constant__ CUtensorMap map_x,
                     const Fp8Params prm) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t bar_full[kStages];     // the first CTA's count for both
    __shared__ __align__(8) uint64_t bar_empty[kStages];
    __shared__ __align__(8) uint64_t bar_d_full[2];
    __shared__ __align__(8) uint64_t bar_d_empty[2];        // the first CTA's count for both
    __shared__ uint32_t tmem_base_slot;

    grid_launch_dependents();
    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t epi_base = smem_base + (uint32_t)(kStages * kStageBytes);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rank = (int)cluster_ctarank();
    const int pair = (int)blockIdx.x >> 1, pairs = (int)gridDim.x >> 1;
    const int tokens = prm.tokens;
    const int row_tiles = (prm.N + 2 * kRows - 1) / (2 * kRows), tok_tiles = (prm.M + tokens - 1) / tokens;
    const int total = row_tiles * tok_tiles;
    const int num_kb = (prm.K + kBlockBytes - 1) / kBlockBytes;
    auto tile_origin = [&](int lin, int& n0, int& m0) {     // this CTA's first row, the pair's first token
        int row_tile = lin, tok_tile = 0;
        if (tok_tiles > 1) {
            constexpr int kRowGroup = 8;
            const int per_group = kRowGroup * tok_tiles;
            const int group = lin / per_group, within = lin % per_group;
            const int rows_here = min(kRowGroup, row_tiles - group * kRowGroup);
            row_tile = group * kRowGroup + within % rows_here;
            tok_tile = within / rows_here;
        }
        n0 = (2 * row_tile + rank) * kRows;
        m0 = tok_tile * tokens;
    };

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(smem_u32(&bar_full[s]), 1);
            mbar_init(smem_u32(&bar_empty[s]), 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(smem_u32(&bar_d_full[a]), 1);
            mbar_init(smem_u32(&bar_d_empty[a]), 8);   // one arrival per epilogue warp of the pair
        }
        fence_barrier_init();
        prefetch_tensormap(&map_p);
        prefetch_tensormap(&map_x);
    }
    if (warp == 1) tmem_alloc_pair(smem_u32(&tmem_base_slot), kTmemCols);
    tc_fence_before_sync();
    __syncthreads();
    cluster_sync_all();           // the other CTA's barriers exist
    tc_fence_after_sync();
    const uint32_t tmem_base = tmem_base_slot;

    bool ok = true;
    if (warp == 0) {
        // ---------------- TMA producer: this CTA's rows and its half of the tokens ----------------
        grid_dependency_wait();   // the activation codes come from the quantisation kernel
        int s = 0;
        uint32_t ph = 0, issued = 0;
        const uint32_t half_tokens = (uint32_t)tokens / 2;
        const uint32_t pair_bytes = 2u * (kRows + half_tokens) * kBlockBytes;
        for (int lin = pair; lin < total && ok; lin += pairs) {
            int n0, m0;
            tile_origin(lin, n0, m0);
            m0 += rank * (int)half_tokens;
            for (int i = 0; i < num_kb && ok; ++i, s = (s + 1 == kStages) ? 0 : s + 1, ph ^= (s == 0)) {
                ok = mbar_wait(smem_u32(&bar_empty[s]), ph ^ 1u);
                ok = __all_sync(0xFFFFFFFFu, ok);
                if (!ok) break;
                if (elect_one()) {
                    const uint32_t full = map_to_cta(smem_u32(&bar_full[s]), 0u);
                    const uint32_t dst = smem_base + (uint32_t)s * kStageBytes;
                    // (the second CTA's bytes may land before this: the phase still waits for the one arrival)
                    if (rank == 0) mbar_arrive_expect_tx(smem_u32(&bar_full[s]), pair_bytes);
                    tma_load_2d_pair(dst, &map_p, full, i * kBlockBytes, n0);
                    tma_load_2d_pair(dst + kRows * kBlockBytes, &map_x, full, i * kBlockBytes, m0);
                }
                __syncwarp();
                ++issued;
            }
        }
        // (the first CTA's barriers count both CTAs' bytes, the second CTA leaves with it)
        if (rank == 0) drain_copies(bar_full, issued, kStages);
    } else if (warp == 1) {
        // ---------------- MMA issuer: the pair's first CTA ----------------
        const uint32_t idesc = idesc_f8(2 * kRows, tokens, prm.e5m2 ? 1 : 0, 0);
        int s = 0, it = 0;
        uint32_t ph = 0;
        for (int lin = pair; rank == 0 && lin < total && ok; lin += pairs, ++it) {
            const int acc = it & 1;
            if (it >= 2) {   // the tile before last used this accumulator: both epilogues must have read it out
                ok = mbar_wait(smem_u32(&bar_d_empty[acc]), (uint32_t)((it >> 1) - 1) & 1u);
                ok = __all_sync(0xFFFFFFFFu, ok);
                if (!ok) break;
                tc_fence_after_sync();
            }
            const uint32_t tmem_d = tmem_base + (uint32_t)(acc * kMaxTokens);
            for (int i = 0; i < num_kb && ok; ++i, s = (s + 1 == kStages) ? 0 : s + 1, ph ^= (s == 0)) {
                ok = mbar_wait(smem_u32(&bar_full[s]), ph);
                ok = __all_sync(0xFFFFFFFFu, ok);
                if (!ok) break;
                tc_fence_after_sync();
                if (elect_one()) {
                    const uint32_t abase = smem_base + (uint32_t)s * kStageBytes;
                    const uint64_t adesc = umma_desc_k_sw128(abase), bdesc = umma_desc_k_sw128(abase + kRows * kBlockBytes);
#pragma unroll
                    for (int j = 0; j < kBlockBytes / 32; ++j)   // 32 K elements = 32 bytes per instruction
                        umma_f8_ss_pair(tmem_d, adesc + (uint64_t)(j * 2), bdesc + (uint64_t)(j * 2), idesc,
                                        (i > 0 || j > 0) ? 1u : 0u);
                    umma_commit_pair(smem_u32(&bar_empty[s]));
                    if (i == num_kb - 1) umma_commit_pair(smem_u32(&bar_d_full[acc]));
                }
                __syncwarp();
            }
        }
    } else {
        // ---------------- epilogue: D[row][token] * scale[token] -> FP16 -> y[token][n0 + row] ----------------
        // Every warp by itself, without barriers among the four: its 32 rows are 64 contiguous bytes of a token's y,
        // whole sectors.  32 token columns go through 2 KB of shared memory of its own, [token][row].  (With barriers
        // among the four warps and the scales fetched per thread and column, a tile of 256 tokens took 6 us more than its
        // MMAs at 4096 columns: QKV at 2048 tokens 101 against 89 us.)
        const int q = warp & 3;                          // TMEM lane quarter this warp may touch
        const uint32_t lane_base = (uint32_t)(q * 32) << 16;
        const float wscale = prm.e5m2 ? 1.0f : 0.00390625f;   // E4M3 bytes read as FP8 are 2^8 times the weights
        const uint32_t buf = epi_base + (uint32_t)(q * kEpiCols * 64);
        float* scales = reinterpret_cast<float*>(smem_raw + (epi_base - smem_u32(smem_raw)) + 4 * kEpiCols * 64) + q * kMaxTokens;
        grid_dependency_wait();   // the scales come from the quantisation kernel, as the codes do
        int it = 0;
        for (int lin = pair; lin < total; lin += pairs, ++it) {
            int n0, m0;
            tile_origin(lin, n0, m0);
            const int acc = it & 1;
            const uint32_t tmem_d = tmem_base + (uint32_t)(acc * kMaxTokens) + lane_base;
            const int ncols = min(tokens, prm.M - m0);
            ok = mbar_wait(smem_u32(&bar_d_full[acc]), (uint32_t)(it >> 1) & 1u);
            ok = __all_sync(0xFFFFFFFFu, ok);
            if (!ok) break;
            tc_fence_after_sync();
            for (int c = lane; c < ncols; c += 32) scales[c] = prm.scale[m0 + c] * wscale;
            __syncwarp();
            const int row0 = n0 + q * 32;                // this warp's first row
            __half* yrow = prm.y + (int64_t)(m0 + (lane >> 2)) * prm.N + row0 + (lane & 3) * 8;
            const bool row_in = row0 + (lane & 3) * 8 < prm.N;   // N is a multiple of 8
            for (int c0 = 0; c0 < ncols; c0 += kEpiCols) {
                uint32_t v[32];
                tmem_ld_32x32b_x32(tmem_d + (uint32_t)c0, v);
                tmem_wait_ld();
                if (c0 + kEpiCols >= ncols) {            // last chunk read: the accumulator is free again
                    tc_fence_before_sync();
                    __syncwarp();
                    if (lane == 0) mbar_arrive_cluster(map_to_cta(smem_u32(&bar_d_empty[acc]), 0u));
                }
#pragma unroll
                for (int j = 0; j < 32; ++j) {
                    const __half hv = __float2half_rn(__uint_as_float(v[j]) * scales[c0 + j]);   // columns past ncols are not stored
                    asm volatile("st.shared.u16 [%0], %1;" ::"r"(buf + (uint32_t)(j * 64 + lane * 2)), "h"(__half_as_ushort(hv))
                                 : "memory");
                }
                __syncwarp();
#pragma unroll
                for (int i = 0; i < 4; ++i) {            // 8 tokens x 64 bytes per instruction
                    const int c = c0 + 8 * i + (lane >> 2);
                    uint4 val;
                    asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];"
                                 : "=r"(val.x), "=r"(val.y), "=r"(val.z), "=r"(val.w)
                                 : "r"(buf + (uint32_t)(i * 512 + lane * 16)));
                    if (row_in && c < ncols) *reinterpret_cast<uint4*>(yrow + (int64_t)(c0 + 8 * i) * prm.N) = val;
                }
                __syncwarp();                            // the buffer is free for the next chunk
            }
        }
    }
    if (!ok) atomicExch(prm.status, (int)DPS_ERR_CUDA);
    tc_fence_before_sync();
    __syncthreads();
    cluster_sync_all();           // nobody frees tensor memory or leaves while the pair still works
    if (warp == 1) {
        tc_fence_after_sync();
        tmem_dealloc_pair(tmem_base, kTmemCols);
    }
}

// Tokens per tile.  A round of tiles over the pairs takes as long as its slowest member, so the number of token tiles
// is chosen to make the sum over the rounds small.  Measured per K block on Llama-7B QKV, 512 tokens: 0.24 / 0.30 / 0.41 /
// 0.48 us with tiles of 64 / 128 / 192 / 256 tokens, i.e. proportional to 128 + tokens (a CTA's share of what comes out
// of L2 is 128 rows and half of the tokens, its tensor time grows with the tokens).
// DPS_FP8_TOKENS=16..256 overrides (tuning knob).
int pick_tokens(int64_t M, int64_t N, int pairs) {
    static const int forced = [] {
        const char* e = getenv("DPS_FP8_TOKENS");
        return e ? atoi(e) / 16 * 16 : 0;
    }();
    if (forced >= 16 && forced <= kMaxTokens) return forced;
    const int64_t row_tiles = (N + 2 * kRows - 1) / (2 * kRows);
    int64_t best = 16, best_cost = INT64_MAX;
    for (int64_t t = (M + kMaxTokens - 1) / kMaxTokens, end = t + (t < 10 ? t + 6 : 16); t <= end; ++t) {
        const int64_t tokens = ((M + t - 1) / t + 15) / 16 * 16;
        const int64_t tiles = row_tiles * ((M + tokens - 1) / tokens), rounds = (tiles + pairs - 1) / pairs;
        const int64_t cost = rounds * (128 + tokens);
        if (cost < best_cost) { best_cost = cost; best = tokens; }
    }
    return (int)best;
}

}  // namespace

cudaError_t launch_quantize_activations(const void* x, uint8_t* q, float* scale, int64_t M, int64_t K, int* status,
                                        cudaStream_t stream) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)M, 1, 1);
    cfg.blockDim = dim3(kQuantThreads, 1, 1);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaError_t e = cudaLaunchKernelEx(&cfg, quantize_activations_kernel, static_cast<const uint4*>(x),
                                       reinterpret_cast<uint2*>(q), scale, (int64_t)(K / 8), status);
    count_launch();
    return e;
}

cudaError_t launch_linear_fp8act(int enc, const uint8_t* q, const float* scale, const uint8_t* p, void* y, int64_t M,
                                 int64_t N, int64_t K, int* status, cudaStream_t stream) {
    static PerDeviceOnce setup;     // per device
    const size_t smem = (size_t)kStages * kStageBytes + kEpiBytes + 1024;
    {
        const cudaError_t e = setup.run(
            [&] { return cudaFuncSetAttribute(fp8act_linear_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem); });
        if (e != cudaSuccess) return e;
    }
    const int pairs = sm_count() / 2;
    const int tokens = pick_tokens(M, N, pairs);
    CUtensorMap mp, mx;
    if (!make_byte_map_sw128(&mp, p, (uint64_t)N, (uint64_t)K, kRows) ||
        !make_byte_map_sw128(&mx, q, (uint64_t)M, (uint64_t)K, (uint32_t)tokens / 2))
        return cudaErrorInvalidValue;
    Fp8Params prm;
    prm.y = static_cast<__half*>(y);
    prm.scale = scale;
    prm.M = (int)M;
    prm.N = (int)N;
    prm.K = (int)K;
    prm.tokens = tokens;
    prm.e5m2 = enc == DPS_ENC_E5M2;
    prm.status = status;
    const int64_t tiles = ((N + 2 * kRows - 1) / (2 * kRows)) * ((M + tokens - 1) / tokens);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(2 * (tiles < pairs ? tiles : pairs)), 1, 1);   // one pair per two SMs walks the tiles
    cfg.blockDim = dim3(kThreads, 1, 1);
    cfg.dynamicSmemBytes = smem;
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
    cudaError_t e = cudaLaunchKernelEx(&cfg, fp8act_linear_kernel, mp, mx, prm);
    count_launch();
    return e;
}

}  // namespace dps
