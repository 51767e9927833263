// Grouped (MoE) linear layer: device-side routing pre-pass, activation gather, grouped kernel.
// Paper: "Scheduler: Dual-Precision Execution", paragraph "Dual-mode serving (DPS) with
// asymmetric switching" -- GroupedGEMM kernels with nested reconstruction serve MoE models.
//
// Steps, all enqueued on the caller's stream without synchronising:
//   (up to 1024 rows: 1 and 2 in one launch, see moe_rank_gather_kernel)
//   1. route   (one CTA): validate rows, count rows per expert (integer atomics), group row ids by
//               expert in ascending row order (stable), and cut every group into token tiles.
//   2. gather  : x_sorted[i][:] = x[token(sorted_rows[i])][:], so that each expert's activations
//               are one contiguous matrix a TMA tile load can address.
//   3. grouped tensor-core kernel over (weight-row tile, token tile): every expert's planes are
//               streamed once per token tile; results are scattered to the caller's row order.
//
// Workspace layout (E4 = E rounded up to 4, A4 = A rounded up to 4, all parts 16-byte aligned):
//   int32 counts[E4] | int32 offsets[E4 + 4] | int32 sorted_rows[A4] | int32 num_tiles[4]
//   | int4 tiles[A4 / 16 + E + 4] | fp16 x_sorted[A][K]
#include <mutex>

#include "dps_internal.h"
#include "gemv.cuh"
#include "sm100.cuh"

namespace dps {

namespace {

constexpr int kRouteThreads = 1024;
constexpr int kMaxExperts = 1024;

inline int64_t round4(int64_t v) { return (v + 3) / 4 * 4; }

struct Workspace {
    int32_t* counts;
    int32_t* offsets;
    int32_t* sorted_rows;
    int32_t* num_tiles;
    int4* tiles;
    __half* x_sorted;
    int64_t max_tiles;
    size_t bytes;
};

Workspace carve(void* base, int64_t A, int32_t E, int64_t K) {
    Workspace w;
    const int64_t e4 = round4(E), a4 = round4(A);
    int32_t* p = static_cast<int32_t*>(base);
    w.counts = p;
    w.offsets = w.counts + e4;
    w.sorted_rows = w.offsets + e4 + 4;
    w.num_tiles = w.sorted_rows + a4;
    w.max_tiles = a4 / 16 + E + 4;
    w.tiles = reinterpret_cast<int4*>(w.num_tiles + 4);
    w.x_sorted = reinterpret_cast<__half*>(w.tiles + w.max_tiles);
    const size_t head = (size_t)(e4 + e4 + 4 + a4 + 4) * 4 + (size_t)w.max_tiles * 16;
    w.bytes = (head + (size_t)A * (size_t)K * 2 + 255) / 256 * 256;
    return w;
}

__device__ __forceinline__ bool row_valid(const int32_t* token_of_row, const int32_t* expert_of_row, int a,
                                          int T, int E) {
    const int e = expert_of_row[a];
    const int t = token_of_row ? token_of_row[a] : a;
    return e >= 0 && e < E && t >= 0 && t < T;
}

constexpr int kTableExperts = pair_plan::kRoutedByTable;   // of the routing kernel's table

// By the whole block: rows per expert (s_cnt, E entries, zero on entry), then by its first warp the first position and the
// first tile of every expert, the tile list and the totals.  s_off (where not null): the first positions.
template <int THREADS>
__device__ __forceinline__ void list_tiles(const int32_t* token_of_row, const int32_t* expert_of_row, int A, int T, int E,
                                           int tile_tokens, int* s_cnt, int* s_off, int32_t* counts, int32_t* offsets,
                                           int32_t* num_tiles, int4* tiles, int* status) {
    const int tid = threadIdx.x, lane = tid & 31;
    int bad = 0;
    for (int a = tid; a < A; a += THREADS) {
        if (row_valid(token_of_row, expert_of_row, a, T, E)) atomicAdd(&s_cnt[expert_of_row[a]], 1);
        else bad = 1;
    }
    if (__syncthreads_or(bad) && tid == 0) atomicExch(status, (int)DPS_ERR_DATA);
    if (tid < 32) {
        int rows = 0, nt = 0;
        for (int base = 0; base < E; base += 32) {
            const int e = base + lane;
            const int c = e < E ? s_cnt[e] : 0, k = (c + tile_tokens - 1) / tile_tokens;
            int ci = c, ki = k;
            for (int o = 1; o < 32; o <<= 1) {
                const int cu = __shfl_up_sync(0xFFFFFFFFu, ci, o), ku = __shfl_up_sync(0xFFFFFFFFu, ki, o);
                if (lane >= o) {
                    ci += cu;
                    ki += ku;
                }
            }
            if (e < E) {
                const int off = rows + ci - c;
                if (s_off != nullptr) s_off[e] = off;
                offsets[e] = off;
                counts[e] = c;
                int t = nt + ki - k;
                for (int first = 0; first < c; first += tile_tokens)
                    tiles[t++] = make_int4(e, off + first, c - first < tile_tokens ? c - first : tile_tokens, 0);
            }
            rows += __shfl_sync(0xFFFFFFFFu, ci, 31);
            nt += __shfl_sync(0xFFFFFFFFu, ki, 31);
        }
        if (lane == 0) {
            offsets[E] = rows;
            num_tiles[0] = nt;
            num_tiles[1] = rows;  // number of valid rows
        }
    }
}

// One CTA.  Invalid rows belong to no group and raise the status word.  Rows are counted per expert with integer atomics
// (the counts do not depend on their order); the grouping itself is stable without any: rows are placed 1024 at a time, a
// row's position among its expert's rows being that of the rows placed before, of the warps before its own (a table of
// counts per warp and expert, scanned by one thread per expert) and of the lanes before its own.  Latency-bound, one SM:
// 4.7 us for 32 rows of 32 experts.  More than kTableExperts experts (the table's size): one warp per expert walks all rows.
__global__ void __launch_bounds__(kRouteThreads)
moe_route_kernel(const int32_t* token_of_row, const int32_t* expert_of_row, int A, int T, int E, int tile_tokens,
                 int32_t* counts, int32_t* offsets, int32_t* sorted_rows, int32_t* num_tiles, int4* tiles, int* status) {
    __shared__ int s_cnt[kMaxExperts];
    __shared__ int s_off[kMaxExperts];
    __shared__ int s_table[kRouteThreads / 32][kTableExperts];
    // the gather and the grouped kernel may be made resident now; both wait for their predecessor
    // (griddepcontrol.wait) before they read anything this kernel writes
    sm100::grid_launch_dependents();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int e = tid; e < E; e += kRouteThreads) s_cnt[e] = 0;
    __syncthreads();
    sm100::grid_dependency_wait();      // the routing and, through an earlier call, the workspace are earlier kernels'
    list_tiles<kRouteThreads>(token_of_row, expert_of_row, A, T, E, tile_tokens, s_cnt, s_off, counts, offsets, num_tiles, tiles, status);
    __syncthreads();
    if (E <= kTableExperts) {
        for (int base = 0; base < A; base += kRouteThreads) {
            for (int i = tid; i < (kRouteThreads / 32) * E; i += kRouteThreads) s_table[i / E][i % E] = 0;
            __syncthreads();
            const int a = base + tid;
            const bool valid = a < A && row_valid(token_of_row, expert_of_row, a, T, E);
            const int e = valid ? expert_of_row[a] : -1;
            const unsigned same = __match_any_sync(0xFFFFFFFFu, e);
            const int before = __popc(same & ((1u << lane) - 1u));
            if (valid && before == 0) s_table[warp][e] = __popc(same);
            __syncthreads();
            if (tid < E) {
                int run = s_off[tid];
                for (int w = 0; w < kRouteThreads / 32; ++w) {
                    const int c = s_table[w][tid];
                    s_table[w][tid] = run;
                    run += c;
                }
                s_off[tid] = run;
            }
            __syncthreads();
            if (valid) sorted_rows[s_table[warp][e] + before] = a;
            __syncthreads();
        }
        return;
    }
    for (int e = warp; e < E; e += kRouteThreads / 32) {
        int pos = s_off[e];
        for (int base = 0; base < A; base += 32) {
            const int a = base + lane;
            const bool hit = a < A && expert_of_row[a] == e && row_valid(token_of_row, expert_of_row, a, T, E);
            const unsigned b = __ballot_sync(0xFFFFFFFFu, hit);
            if (hit) sorted_rows[pos + __popc(b & ((1u << lane) - 1u))] = a;
            pos += __popc(b);
        }
    }
}

// x_sorted[i][:] = x[token(sorted_rows[i])][:] for the valid rows; 16 bytes per thread.
// No __restrict__ here and in the routing kernel: both are resident while the kernels that write what they read still run,
// and a pointer marked so may be read through the non-coherent path, which wants data that nobody writes meanwhile.
__global__ void __launch_bounds__(256)
moe_gather_kernel(const uint4* x, const int32_t* token_of_row, const int32_t* sorted_rows, const int32_t* num_tiles,
                  uint4* x_sorted, int64_t k16) {
    sm100::grid_launch_dependents();
    sm100::grid_dependency_wait();   // sorted_rows and num_tiles come from the routing kernel
    const int valid = num_tiles[1];
    for (int i = blockIdx.x; i < valid; i += gridDim.x) {
        const int a = sorted_rows[i];
        const int64_t tok = token_of_row ? token_of_row[a] : a;
        const uint4* src = x + tok * k16;
        uint4* dst = x_sorted + (int64_t)i * k16;
        for (int64_t c = threadIdx.x; c < k16; c += blockDim.x) dst[c] = src[c];
    }
}

// Routing and gather in one launch, for up to kRankRows rows: every row has a block of its own, which finds the row's position
// among the sorted rows by itself -- the number of valid rows of smaller experts, and of its own expert in front of it -- and
// copies the activations there; one more block makes the tile list.  Two launches, each a chain of latencies that the next waits
// for, become one.  The positions cost A comparisons per row, which is the longer way for many rows.  A whole call with hardly any
// weights (256 rows x 4096, 8 experts / 256 x 2048, 64 experts), two launches against one, us: 2 rows 16.8 / 12.2 against 14.4 / 9.8,
// 128 rows 17.1 / 13.6 against 15.0 / 11.0, 512 20.6 / 14.8 against 19.2 / 12.9, 1024 23.5 / 15.6 against 23.4 / 14.4, 2048 27.1 / 20.8
// against 31.2 / 23.3, 4096 37.6 / 28.2 against 56.7 / 47.0.
constexpr int kRankRows = 1024;
constexpr int kRankThreads = 256;

__global__ void __launch_bounds__(kRankThreads)
moe_rank_gather_kernel(const uint4* x, const int32_t* token_of_row, const int32_t* expert_of_row, int A, int T, int E,
                       int tile_tokens, int32_t* counts, int32_t* offsets, int32_t* sorted_rows, int32_t* num_tiles, int4* tiles,
                       uint4* x_sorted, int64_t k16, int* status) {
    __shared__ int s_cnt[kMaxExperts];
    __shared__ int s_sum[kRankThreads / 32];
    sm100::grid_launch_dependents();
    const int tid = threadIdx.x;
    if (blockIdx.x == 0) {
        for (int e = tid; e < E; e += kRankThreads) s_cnt[e] = 0;
        __syncthreads();
        sm100::grid_dependency_wait();
        list_tiles<kRankThreads>(token_of_row, expert_of_row, A, T, E, tile_tokens, s_cnt, nullptr, counts, offsets, num_tiles, tiles, status);
        return;
    }
    const int a = (int)blockIdx.x - 1;
    sm100::grid_dependency_wait();      // the routing and, through an earlier call, the workspace are earlier kernels'
    if (!row_valid(token_of_row, expert_of_row, a, T, E)) return;       // (block 0 reports it)
    const int e = expert_of_row[a];
    const int64_t tok = token_of_row ? token_of_row[a] : a;
    const uint4* src = x + tok * k16;
    constexpr int kAhead = 4;           // pieces of the row requested before its position is known
    uint4 v[kAhead];
#pragma unroll
    for (int i = 0; i < kAhead; ++i)
        if (tid + i * kRankThreads < k16) v[i] = src[tid + i * kRankThreads];
    int before = 0;
#pragma unroll 4
    for (int b = tid; b < A; b += kRankThreads) {
        const int other = expert_of_row[b];
        before += (other < e || (other == e && b < a)) && row_valid(token_of_row, expert_of_row, b, T, E);
    }
    before = __reduce_add_sync(0xFFFFFFFFu, before);
    if ((tid & 31) == 0) s_sum[tid >> 5] = before;
    __syncthreads();
    int pos = 0;
#pragma unroll
    for (int i = 0; i < kRankThreads / 32; ++i) pos += s_sum[i];
    if (tid == 0) sorted_rows[pos] = a;
    uint4* dst = x_sorted + (int64_t)pos * k16;
#pragma unroll
    for (int i = 0; i < kAhead; ++i)
        if (tid + i * kRankThreads < k16) dst[tid + i * kRankThreads] = v[i];
    for (int64_t c = tid + kAhead * kRankThreads; c < k16; c += kRankThreads) dst[c] = src[c];
}

}  // namespace

size_t moe_workspace_bytes(int64_t A, int32_t E, int64_t K) {
    if (A < 0 || E <= 0 || E > kMaxExperts || A > (int64_t)1 << 30 || K <= 0 || K > (int64_t)1 << 31) return 0;
    return carve(nullptr, A, E, K).bytes;
}

cudaError_t launch_moe(int mode, const int32_t* enc_host, const void* x, const int32_t* token_of_row,
                       const int32_t* expert_of_row, const uint8_t* p, const uint8_t* r, void* y, int64_t A,
                       int64_t T, int64_t N, int64_t K, int32_t E, void* workspace, int* status,
                       cudaStream_t stream) {
    const Workspace w = carve(workspace, A, E, K);
    // CTA pairs or 128-row tiles, two CTAs per SM: pair_plan.h
    const bool pairs = pair_plan::grouped_on_pairs(mode == DPS_MODE_FULL, A, N, K, E, sm_count() / 2);
    const int tn = pairs ? pair_plan::grouped_width(mode == DPS_MODE_FULL, A, N, E, sm_count() / 2) : grouped_tile_tokens(A, E);
    cudaError_t err;
    // programmatic dependent launch, as the kernel behind them: each is resident early and waits before its first read
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    auto config = [&](int64_t blocks, int threads) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)blocks, 1, 1);
        cfg.blockDim = dim3((unsigned)threads, 1, 1);
        cfg.stream = stream;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        return cfg;
    };
    const uint4* rows_in = static_cast<const uint4*>(x);
    uint4* rows_out = reinterpret_cast<uint4*>(w.x_sorted);
    if (A <= kRankRows) {
        const cudaLaunchConfig_t cfg = config(A + 1, kRankThreads);
        err = cudaLaunchKernelEx(&cfg, moe_rank_gather_kernel, rows_in, token_of_row, expert_of_row, (int)A, (int)T, (int)E, tn,
                                 w.counts, w.offsets, w.sorted_rows, w.num_tiles, w.tiles, rows_out, (int64_t)(K / 8), status);
        count_launch();
        if (err != cudaSuccess) return err;
    } else {
        const cudaLaunchConfig_t route = config(1, kRouteThreads), gather = config(A < 4096 ? A : 4096, 256);
        err = cudaLaunchKernelEx(&route, moe_route_kernel, token_of_row, expert_of_row, (int)A, (int)T, (int)E, tn, w.counts,
                                 w.offsets, w.sorted_rows, w.num_tiles, w.tiles, status);
        count_launch();
        if (err != cudaSuccess) return err;
        err = cudaLaunchKernelEx(&gather, moe_gather_kernel, rows_in, token_of_row, (const int32_t*)w.sorted_rows,
                                 (const int32_t*)w.num_tiles, rows_out, (int64_t)(K / 8));
        count_launch();
        if (err != cudaSuccess) return err;
    }

    // 32 words of E5M2 bits, then 32 words of rounded-nest bits
    static_assert(kMaxExperts == 1024, "the grouped kernels take two 32-word masks");
    uint32_t mask[64];
    for (int i = 0; i < 64; ++i) mask[i] = 0;
    for (int e = 0; e < E; ++e) {
        if (enc_host[e] == DPS_ENC_E5M2 || enc_host[e] == DPS_ENC_E5M2_RN) mask[e >> 5] |= 1u << (e & 31);
        if (enc_host[e] == DPS_ENC_E4M3_RN || enc_host[e] == DPS_ENC_E5M2_RN) mask[32 + (e >> 5)] |= 1u << (e & 31);
    }
    // an upper bound on the number of token tiles that needs no device round trip
    const int max_tiles = (int)((A + tn - 1) / tn + E);
    if (pairs)
        return launch_pair_grouped(mode, mask, w.x_sorted, p, r, y, A, N, K, E, tn, w.tiles, w.num_tiles, w.sorted_rows,
                                   max_tiles < w.max_tiles ? max_tiles : (int)w.max_tiles, status, stream);
    return launch_umma_grouped(mode, mask, w.x_sorted, p, r, y, A, N, K, E, tn, w.tiles, w.num_tiles, w.sorted_rows,
                               max_tiles < w.max_tiles ? max_tiles : (int)w.max_tiles, status, stream);
}

}  // namespace dps

// ---- allocation-free variant ---------------------------------------------------------------------
// Scratch for dps_moe_linear_static: one fixed array per GPU that loads the library, held until the
// process exits.  In host code the array's name is only a stand-in; the device address is looked up
// once per device (with that device current) and handed to the kernels as an ordinary pointer.
namespace dps {
namespace {

constexpr size_t kStaticScratchBytes = (size_t)DPS_MOE_STATIC_SCRATCH_BYTES;
static __device__ __align__(256) unsigned char g_moe_static_scratch[kStaticScratchBytes];

// Device address of the array, per device.  Only a successful look-up is kept: a failed one (made
// inside a stream capture, say) is tried again by the next call.
std::mutex g_static_scratch_mutex;
unsigned char* g_static_scratch_ptr[kMaxDevices] = {};

cudaError_t static_scratch_address(unsigned char** out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_static_scratch_mutex);
    if (g_static_scratch_ptr[dev] == nullptr) {
        unsigned char* ptr = nullptr;
        e = cudaGetSymbolAddress((void**)&ptr, g_moe_static_scratch);
        if (e != cudaSuccess) {
            (void)cudaGetLastError();   // leave no sticky error behind: the next call tries again
            return e;
        }
        g_static_scratch_ptr[dev] = ptr;
    }
    *out = g_static_scratch_ptr[dev];
    return cudaSuccess;
}

}  // namespace
}  // namespace dps

extern "C" DPS_API dps_status dps_moe_linear_static(int32_t mode, const int32_t* enc_per_expert, const void* x,
                                                    const int32_t* token_of_row, const int32_t* expert_of_row,
                                                    const uint8_t* w_persist, const uint8_t* w_resid, void* y,
                                                    int64_t A, int64_t T, int64_t N, int64_t K, int32_t E,
                                                    void* cuda_stream) {
    using namespace dps;
    bool empty = false;
    const dps_status ok = check_moe_args(mode, enc_per_expert, x, token_of_row, expert_of_row, w_persist, w_resid, y, A, T,
                                         N, K, E, &empty);
    if (ok != DPS_OK) return ok;
    if (moe_workspace_bytes(A, E, K) > kStaticScratchBytes) return DPS_ERR_WORKSPACE;  // use dps_moe_linear instead
    if (empty) return DPS_OK;
    int* status = nullptr;
    const dps_status st = device_status_word(&status);
    if (st != DPS_OK) return st;
    unsigned char* scratch = nullptr;
    if (static_scratch_address(&scratch) != cudaSuccess || scratch == nullptr) return DPS_ERR_CUDA;
    const uint8_t* r = (mode == DPS_MODE_FULL) ? w_resid : nullptr;
    if (launch_moe(mode, enc_per_expert, x, token_of_row, expert_of_row, w_persist, r, y, A, T, N, K, E, scratch,
                   status, static_cast<cudaStream_t>(cuda_stream)) != cudaSuccess)
        return DPS_ERR_CUDA;
    return DPS_OK;
}
