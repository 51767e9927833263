// The C ABI of libdps: argument validation, the per-device status word, and dispatch of each
// call to a kernel family.  Nothing here allocates or frees device memory.
#include <atomic>
#include <cstdlib>
#include <cstring>
#include <mutex>

#include "sm100.cuh"

#include "bits.cuh"
#include "dps_internal.h"
#include "two_launches.h"

namespace dps {

namespace {

// Per-device words that kernels write: the status word (data-dependent errors) and the
// scratch word of the load-time magnitude statistic.
__device__ int g_status_word;
__device__ unsigned g_stat_word;
__device__ unsigned g_auto_flag;   // number of the last AUTO split that met a word out of E4M3 range

// Self-test of the bounded device-side waits: ONE warp initialises an mbarrier that nobody will ever
// arrive on and waits for it with the given limit -- the same wait (and the same reaction: set the
// status word, give up, return) as every pipeline wait in the tensor-core kernels.  No copy is in
// flight, no tensor memory is held, no other CTA is involved.
__global__ void wait_timeout_selftest_kernel(unsigned long long limit_ns, int* status) {
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x == 0) {
        sm100::mbar_init(sm100::smem_u32(&bar), 1);
        sm100::fence_barrier_init();
    }
    __syncwarp();
    if (!sm100::mbar_wait_limit(sm100::smem_u32(&bar), 0, limit_ns) && threadIdx.x == 0)
        atomicExch(status, (int)DPS_ERR_CUDA);
}

std::atomic<int64_t> g_launches{0};
std::mutex g_stat_mutex;  // the statistic words are shared by all AUTO / checked-E4M3 splits

struct DeviceInfo {
    std::once_flag once;
    cudaError_t err = cudaSuccess;
    int* status = nullptr;
    unsigned* stat = nullptr;
    unsigned* auto_flag = nullptr;
    unsigned* auto_host = nullptr;   // mapped host memory, one word, from the first AUTO split on (g_stat_mutex)
    unsigned auto_calls = 0;         // (g_stat_mutex)
    int sms = 0;
    int cc_major = 0;
};
DeviceInfo g_dev[kMaxDevices];

DeviceInfo* device_info() {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return nullptr;
    DeviceInfo& d = g_dev[dev];
    std::call_once(d.once, [&] {
        d.err = cudaGetSymbolAddress((void**)&d.status, g_status_word);
        if (d.err == cudaSuccess) d.err = cudaGetSymbolAddress((void**)&d.stat, g_stat_word);
        if (d.err == cudaSuccess) d.err = cudaGetSymbolAddress((void**)&d.auto_flag, g_auto_flag);
        if (d.err == cudaSuccess) d.err = cudaDeviceGetAttribute(&d.sms, cudaDevAttrMultiProcessorCount, dev);
        if (d.err == cudaSuccess) d.err = cudaDeviceGetAttribute(&d.cc_major, cudaDevAttrComputeCapabilityMajor, dev);
    });
    return &d;
}

// Tuning / debugging knob: DPS_FORCE_PATH=gemv, =umma, =stream or =pair pins the dense kernel family.
int forced_path() {
    static const int path = [] {
        const char* v = getenv("DPS_FORCE_PATH");
        if (!v) return 0;
        if (!strcmp(v, "gemv")) return 1;
        if (!strcmp(v, "umma")) return 2;
        if (!strcmp(v, "stream")) return 3;
        if (!strcmp(v, "pair")) return 4;
        return 0;
    }();
    return path;
}

inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

dps_status check_device(DeviceInfo*& d) {
    d = device_info();
    if (d == nullptr || d->err != cudaSuccess) return DPS_ERR_CUDA;
    if (d->cc_major != 10) return DPS_ERR_UNSUPPORTED;  // the kernels are built for sm_100a only
    return DPS_OK;
}

}  // namespace

void count_launch(int n) { g_launches.fetch_add(n, std::memory_order_relaxed); }

dps_status check_moe_args(int32_t mode, const int32_t* enc_per_expert, const void* x, const int32_t* token_of_row,
                          const int32_t* expert_of_row, const uint8_t* w_persist, const uint8_t* w_resid, const void* y,
                          int64_t A, int64_t T, int64_t N, int64_t K, int32_t E, bool* empty) {
    *empty = false;
    if (mode != DPS_MODE_FAST && mode != DPS_MODE_FULL) return DPS_ERR_MODE;
    if (A < 0 || T < 0 || N <= 0 || K <= 0 || E <= 0 || (K % 16) != 0 || (N % 8) != 0) return DPS_ERR_SHAPE;
    if (A > ((int64_t)1 << 30) || T > ((int64_t)1 << 30) || N >= ((int64_t)1 << 31) || K >= ((int64_t)1 << 31))
        return DPS_ERR_SHAPE;
    // the kernels address plane rows of all experts with 32-bit coordinates
    if ((int64_t)E * N >= ((int64_t)1 << 31)) return DPS_ERR_SHAPE;
    if (!enc_per_expert) return DPS_ERR_NULL;
    if (moe_workspace_bytes(A, E, K) == 0) return DPS_ERR_SHAPE;
    for (int32_t e = 0; e < E; ++e) {
        const int32_t enc = enc_per_expert[e];
        if (enc != DPS_ENC_E4M3 && enc != DPS_ENC_E5M2 && enc != DPS_ENC_E4M3_RN && enc != DPS_ENC_E5M2_RN)
            return DPS_ERR_ENCODING;
    }
    if (A == 0) {
        *empty = true;
        return DPS_OK;
    }
    if (!x || !expert_of_row || !w_persist || !y) return DPS_ERR_NULL;
    if (mode == DPS_MODE_FULL && !w_resid) return DPS_ERR_NULL;
    if (!aligned16(x) || !aligned16(w_persist) || !aligned16(y)) return DPS_ERR_ALIGN;
    if (mode == DPS_MODE_FULL && !aligned16(w_resid)) return DPS_ERR_ALIGN;
    if ((reinterpret_cast<uintptr_t>(expert_of_row) & 3u) || (reinterpret_cast<uintptr_t>(token_of_row) & 3u))
        return DPS_ERR_ALIGN;
    return DPS_OK;
}

dps_status device_status_word(int** status) {
    DeviceInfo* d = nullptr;
    const dps_status st = check_device(d);
    *status = (st == DPS_OK) ? d->status : nullptr;
    return st;
}

int sm_count() {
    DeviceInfo* d = device_info();
    return (d && d->sms > 0) ? d->sms : 148;
}

}  // namespace dps

using namespace dps;

namespace {
// 65-128 tokens: two 64-token decode tiles per 128 weight rows (K split over a cluster) instead of CTA pairs with 256-row
// tiles, where the latter would leave most SMs idle and the weights are few enough to be streamed out of L2 and rebuilt
// twice.  Fast / full mode, tiles against pairs, us: 96 tokens 4096 x 4096 10.3 / 13.9 against 11.1 / 12.7, 2048 x 2048 6.3 / 7.4 against
// 7.7 / 8.3, 6144 x 1024 6.6 / 8.0 against 6.7 / 7.8; 128 tokens 10.5 / 14.1 against 11.8 / 14.0, 6.4 / 7.5 against 8.3 / 9.2, 6.8 / 8.1
// against 6.4 / 7.1 (where the tiles are a little behind the line is older than the pairs' present start); beyond the line, 96 tokens, 3088 x
// 8336 in full mode 24.7 against 18.0, 4632 x 3088 15.4 / 22.4 against 10.8 / 12.6, 12288 x 4096 20.9 / 40.2 against 16.0 / 22.9.
bool decode_tiles_for_128(bool full, int64_t M, int64_t N, int64_t K) {
    return M <= 128 && ((N <= 4096 && N * K <= ((int64_t)1 << (full ? 24 : 26))) || N * K <= ((int64_t)1 << 23));
}
// 33-64 tokens: CTA pairs instead of the 64-token decode tiles where K is long and the pairs take no more turns over the chip
// (tile_plan.h: pairs_for_long_k, with what both sides take).  Fast / full mode, 64 tokens, tiles against pairs, us: 8192 x 28672 53.6 / 85.8 against 46.1 / 82.2,
// 12288 x 16384 54.7 / 85.8 against 47.1 / 75.8, 38144 x 16384 147.5 / 277.8 against 132.2 / 242.5; but 6144 x 16384 27.0 / 40.2 against
// 28.1 / 42.8, 8704 x 16384 32.8 / 51.6 against 44.7 / 66.0, 19200 x 16384 75.1 / 147.3 against 86.3 / 150.0.  With a shorter K the pairs' fixed
// costs show: 4096 x 14336 17.1 / 25.5 against 19.6 / 27.8, 10240 x 8192 24.3 / 36.3 against 26.5 / 39.6; at 20 tokens the 32-token tiles are
// faster here too: 43.0 / 78.0 against 45.0 / 80.2.  (All of these in bursts.  57344 x 8192, 93.7 / 170 against 95.4 / 174 so, takes 193 against 186 in
// full mode under the power cap, which is where the rule for tall matrices, share_rows, was measured.)  A pair sums a longer range of K in one
// accumulator: at 8192 x 28672 the error against 64 bits is 2.074e-4 of the output instead of 2.070e-4, of which the rounding to FP16 is 2.068e-4.
bool pairs_for_64(int32_t mode, int32_t enc, int64_t M, int64_t N, int64_t K) {
    if (M <= 32 || M > 64 || K < 16384 || N < 5120) return false;
    tile_plan::Turns pairs, tiles;
    return ask_pair_plan(mode, enc, M, N, K, {&pairs, nullptr}) == cudaSuccess && tile_turns_64(mode, enc, M, N, K, &tiles) == cudaSuccess &&
           tile_plan::pairs_for_long_k(pairs, tiles);
}
// More than a handful of tokens on rows of one matrix: decode tiles or CTA pairs.
cudaError_t launch_tensor(int32_t mode, int32_t enc, const void* x, const uint8_t* p, const uint8_t* r, void* y, int64_t ldy, int64_t M, int64_t N,
                          int64_t K, int* status, cudaStream_t stream, bool prepare_only = false) {
    const bool pairs = M > 64 ? !decode_tiles_for_128(mode == DPS_MODE_FULL, M, N, K) : pairs_for_64(mode, enc, M, N, K);
    return pairs ? launch_pair_linear(mode, enc, x, p, r, y, ldy, M, N, K, status, stream, prepare_only)
                 : launch_umma_linear(mode, enc, x, p, r, y, ldy, M, N, K, status, stream, prepare_only);
}
// The same for a whole matrix: the rows of whole rounds of pairs first, where the rest is better off by itself (pair_plan.h: share_rows).  The
// second launch depends on the first for nothing but the order; its planes are on their way while the first drains.  Two layers of hidden
// size 8192 at 64 tokens, full mode: 725 -> 686 us.
cudaError_t launch_rows(int32_t mode, int32_t enc, const void* x, const uint8_t* p, const uint8_t* r, void* y, int64_t M, int64_t N, int64_t K,
                        int* status, cudaStream_t stream) {
    pair_plan::RowShare share;
    if (pair_plan::may_share_rows(M, N, sm_count())) {
        const cudaError_t e = ask_pair_plan(mode, enc, M, N, K, {nullptr, &share});
        if (e != cudaSuccess) return e;
    }
    if (!share.pairs) return launch_tensor(mode, enc, x, p, r, y, N, M, N, K, status, stream);
    const int64_t rows = share.rows > 0 ? share.rows : N;
    auto whole_rounds = [&] { return launch_pair_linear(mode, enc, x, p, r, y, N, M, rows, K, status, stream); };
    if (rows == N) return whole_rounds();
    return launch_two(whole_rounds, [&](bool prepare_only) {
        return launch_tensor(mode, enc, x, p + rows * K, r != nullptr ? r + rows * K : nullptr, static_cast<uint16_t*>(y) + rows, N, M, N - rows, K, status,
                             stream, prepare_only);
    });
}
bool known_encoding(int32_t enc) {
    return enc == DPS_ENC_E4M3 || enc == DPS_ENC_E5M2 || enc == DPS_ENC_E4M3_RN || enc == DPS_ENC_E5M2_RN;
}
}  // namespace

extern "C" {

dps_status dps_split_weights(const void* w_fp16, uint8_t* w_persist, uint8_t* w_resid, int64_t rows, int64_t cols,
                             int32_t* enc_inout, void* cuda_stream) {
    if (enc_inout == nullptr) return DPS_ERR_NULL;
    const int32_t req = *enc_inout;
    if (req != DPS_ENC_AUTO && req != DPS_ENC_AUTO_RN && !known_encoding(req)) return DPS_ERR_ENCODING;
    if (rows < 0 || cols < 0 || (cols % 16) != 0) return DPS_ERR_SHAPE;
    if (rows > 0 && cols > 0 && rows > INT64_MAX / cols) return DPS_ERR_SHAPE;
    const int64_t n = rows * cols;
    if (n == 0) {
        if (req == DPS_ENC_AUTO) *enc_inout = DPS_ENC_E4M3;
        if (req == DPS_ENC_AUTO_RN) *enc_inout = DPS_ENC_E4M3_RN;
        return DPS_OK;
    }
    if (!w_fp16 || !w_persist || !w_resid) return DPS_ERR_NULL;
    if (!aligned16(w_fp16) || !aligned16(w_persist) || !aligned16(w_resid)) return DPS_ERR_ALIGN;
    DeviceInfo* d;
    dps_status st = check_device(d);
    if (st != DPS_OK) return st;
    cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
    int enc = req;
    if (req == DPS_ENC_AUTO) {
        // One pass: split as E4M3 while looking for words above 0x3F00 (|w| > 1.75); only a tensor that has one is
        // split again, as E5M2.  Every layer of a model goes through here once, four tensors of a Llama-7B layer
        // with the rebuilding that checks them 453 -> 308 us.  A word out of range costs the part of the first pass that
        // ran before it was met: a call on 12288 x 4096 weights takes 53 us without one, 75 / 81 / 90 us with one at the
        // start / middle / end (a statistics pass and then one split: 97 us), on 57344 x 8192 290, 437 / 510 / 576 us (507 us).
        // The kernel reports into mapped host memory, so the
        // host needs no copy after the wait that the choice of the encoding makes necessary anyway; after that wait
        // the planes are complete, so no fence launch is needed either.
        std::lock_guard<std::mutex> lock(g_stat_mutex);
        if (d->auto_host == nullptr) {
            void* word = nullptr;
            if (cudaHostAlloc(&word, sizeof(unsigned), cudaHostAllocPortable | cudaHostAllocMapped) != cudaSuccess) {
                (void)cudaGetLastError();
                return DPS_ERR_CUDA;
            }
            d->auto_host = static_cast<unsigned*>(word);
            *d->auto_host = 0;
        }
        const unsigned call = ++d->auto_calls ? d->auto_calls : ++d->auto_calls;   // 0 is what the words start with
        if (launch_split_auto(static_cast<const uint16_t*>(w_fp16), w_persist, w_resid, n, d->auto_flag, d->auto_host, call,
                              stream) != cudaSuccess)
            return DPS_ERR_CUDA;
        if (cudaStreamSynchronize(stream) != cudaSuccess) return DPS_ERR_CUDA;
        if (*static_cast<volatile unsigned*>(d->auto_host) != call) {
            *enc_inout = DPS_ENC_E4M3;
            return DPS_OK;
        }
        enc = DPS_ENC_E5M2;
    } else if (req != DPS_ENC_E5M2) {
        // Load-time statistics: max over the tensor of (word & 0x7FFF).  A word with the exponent
        // MSB set is >= 0x4000, so one maximum answers all questions:
        //   E4M3  -> legal iff max <  0x3F80 (exponent MSB clear and the byte is not 0x7F/0xFF)
        //   rounded nests: the same limits must hold after half a unit of the last kept bit is added
        //     E4M3_RN -> legal iff max + 0x40 < 0x3F80;  E5M2_RN -> legal iff max + 0x80 < 0x7C00 (no Inf code)
        std::lock_guard<std::mutex> lock(g_stat_mutex);
        unsigned maxmag = 0;
        if (cudaMemsetAsync(d->stat, 0, sizeof(unsigned), stream) != cudaSuccess) return DPS_ERR_CUDA;
        if (launch_magnitude_stat(static_cast<const uint16_t*>(w_fp16), n, d->stat, stream) != cudaSuccess)
            return DPS_ERR_CUDA;
        if (cudaMemcpyAsync(&maxmag, d->stat, sizeof(unsigned), cudaMemcpyDeviceToHost, stream) != cudaSuccess)
            return DPS_ERR_CUDA;
        if (cudaStreamSynchronize(stream) != cudaSuccess) return DPS_ERR_CUDA;
        if (req == DPS_ENC_AUTO_RN) {
            enc = (maxmag <= 0x3F00u) ? DPS_ENC_E4M3_RN : DPS_ENC_E5M2_RN;
            if (enc == DPS_ENC_E5M2_RN && maxmag + 0x80u >= 0x7C00u) return DPS_ERR_DATA;
        }
        else if (req == DPS_ENC_E4M3 && maxmag >= 0x3F80u) return DPS_ERR_DATA;
        else if (req == DPS_ENC_E4M3_RN && maxmag + 0x40u >= 0x3F80u) return DPS_ERR_DATA;
        else if (req == DPS_ENC_E5M2_RN && maxmag + 0x80u >= 0x7C00u) return DPS_ERR_DATA;
    }
    if (launch_split(static_cast<const uint16_t*>(w_fp16), w_persist, w_resid, n, enc, stream) != cudaSuccess)
        return DPS_ERR_CUDA;
    *enc_inout = enc;
    return DPS_OK;
}

dps_status dps_reconstruct(const uint8_t* w_persist, const uint8_t* w_resid, void* w_fp16_out, int64_t rows,
                           int64_t cols, int32_t enc, void* cuda_stream) {
    if (!known_encoding(enc)) return DPS_ERR_ENCODING;
    if (rows < 0 || cols < 0 || (cols % 16) != 0) return DPS_ERR_SHAPE;
    if (rows > 0 && cols > 0 && rows > INT64_MAX / cols) return DPS_ERR_SHAPE;
    const int64_t n = rows * cols;
    if (n == 0) return DPS_OK;
    if (!w_persist || !w_fp16_out) return DPS_ERR_NULL;
    if (!aligned16(w_persist) || !aligned16(w_resid) || !aligned16(w_fp16_out)) return DPS_ERR_ALIGN;
    DeviceInfo* d;
    dps_status st = check_device(d);
    if (st != DPS_OK) return st;
    if (launch_reconstruct(w_persist, w_resid, static_cast<uint16_t*>(w_fp16_out), n, enc,
                           static_cast<cudaStream_t>(cuda_stream)) != cudaSuccess)
        return DPS_ERR_CUDA;
    return DPS_OK;
}

dps_status dps_linear(int32_t mode, int32_t enc, const void* x, const uint8_t* w_persist, const uint8_t* w_resid,
                      void* y, int64_t M, int64_t N, int64_t K, void* cuda_stream) {
    if (mode != DPS_MODE_FAST && mode != DPS_MODE_FULL) return DPS_ERR_MODE;
    if (!known_encoding(enc)) return DPS_ERR_ENCODING;
    if (M < 0 || N <= 0 || K <= 0 || (K % 16) != 0 || (N % 8) != 0) return DPS_ERR_SHAPE;
    if (N >= ((int64_t)1 << 31) || K >= ((int64_t)1 << 31) || M >= ((int64_t)1 << 31)) return DPS_ERR_SHAPE;
    if (M == 0) return DPS_OK;
    if (!x || !w_persist || !y) return DPS_ERR_NULL;
    if (mode == DPS_MODE_FULL && !w_resid) return DPS_ERR_NULL;
    if (!aligned16(x) || !aligned16(w_persist) || !aligned16(y)) return DPS_ERR_ALIGN;
    if (mode == DPS_MODE_FULL && !aligned16(w_resid)) return DPS_ERR_ALIGN;
    DeviceInfo* d;
    dps_status st = check_device(d);
    if (st != DPS_OK) return st;
    cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
    const uint8_t* r = (mode == DPS_MODE_FULL) ? w_resid : nullptr;  // fast mode never sees the pointer
    // A handful of tokens makes the layer a pure weight stream: up to 8 tokens (one MMA column group) the
    // register-streaming kernel serves it.  For 9-16 tokens that kernel is the faster one for a single small matrix (4096 x
    // 4096: 4.9 us against 7.0), but not for a layer: it lives on a large L1, the tensor-core tiles on a large
    // shared memory, and an SM that changes its split drains first.  Four linears in turn at 12-13 tokens, streaming kernel
    // / tiles / the one or the other by N K < 2^25, which was the rule: hidden 3088 in full mode 57 / 46 / 98 us, 2048 in
    // fast mode 23.0 / 22.6 / 38, 4096 in full mode (16 tokens) 86 / 83 / 91; 1024 14.7 / 17.7, 512 9.3 / 13.2.  The smaller
    // side of the matrix is the hidden size in all four, so a rule on it keeps a layer in one family.  Matrices of 2^25 weights
    // and more with a small side, output heads, are the tiles' all the same (9 tokens, streaming kernel / tiles): 128256 x 1024
    // by itself 45.8 / 35.0 us in fast and 60.0 / 52.3 in full mode, behind twelve layers of hidden size 1024 198 / 184 and 260 / 246
    // for all; 57344 x 1536 behind eight layers 156 / 148 and 220 / 218.  (By itself, in full mode, 35.6 / 39.4.)
    // What the rule costs: a matrix beyond it that is called by itself.  2048 x 2048, 9 tokens, takes 4.5 us in fast and 5.4 in
    // full mode, the streaming kernel 3.4 and 3.9; 4096 x 4096 6.7 and 9.3 against 5.7 and 8.8.  With other programs' kernels
    // between the linears every launch of the tiles pays for the change of split, about 2 us: 2048 x 2048 7.0 against 4.2.
    // Beyond 16 tokens the tcgen05 tiles take over, beyond 64 tokens (33 for a long K, see pairs_for_64, from 17 on for tall matrices, see launch_rows) CTA
    // pairs.  Four linears of a layer, fast / full mode, tiles against pairs, us, in bursts: Llama-7B 64 tokens 61.8 / 96.5 against 66.7 / 95.1,
    // 96 tokens 89.0 / 147.4 against 69.6 / 98.8;
    // hidden size 2048, 64 tokens, 29.7 / 39.8 against 35.6 / 40.8, 96 tokens 37.8 / 53.7 against 37.9 / 46.1.  (The CUDA-core GEMV is kept as a cross-check.)
    const bool stream_mid = (N < K ? N : K) <= 1536 && N * K < ((int64_t)1 << 25);
    const int path = forced_path();
    cudaError_t err;
    if (path == 1) err = launch_gemv(mode, enc, x, w_persist, r, y, M, N, K, stream);
    else if (path == 2) err = launch_umma_linear(mode, enc, x, w_persist, r, y, N, M, N, K, d->status, stream);
    else if (path == 4) err = launch_pair_linear(mode, enc, x, w_persist, r, y, N, M, N, K, d->status, stream);
    else if (path == 3 || M <= 8 || (M <= 16 && stream_mid)) {
        if (M > 16) return DPS_ERR_UNSUPPORTED;      // (only reachable with DPS_FORCE_PATH=stream)
        err = launch_decode_mma(mode, enc, x, w_persist, r, y, M, N, K, stream);
    } else err = launch_rows(mode, enc, x, w_persist, r, y, M, N, K, d->status, stream);
    return err == cudaSuccess ? DPS_OK : DPS_ERR_CUDA;
}

size_t dps_moe_workspace_bytes(int64_t A, int32_t E, int64_t K) { return moe_workspace_bytes(A, E, K); }

dps_status dps_moe_linear(int32_t mode, const int32_t* enc_per_expert, const void* x, const int32_t* token_of_row,
                          const int32_t* expert_of_row, const uint8_t* w_persist, const uint8_t* w_resid, void* y,
                          int64_t A, int64_t T, int64_t N, int64_t K, int32_t E, void* workspace,
                          size_t workspace_bytes, void* cuda_stream) {
    bool empty = false;
    const dps_status ok = check_moe_args(mode, enc_per_expert, x, token_of_row, expert_of_row, w_persist, w_resid, y, A, T,
                                         N, K, E, &empty);
    if (ok != DPS_OK || empty) return ok;
    const size_t need = moe_workspace_bytes(A, E, K);
    if (!workspace || !aligned16(workspace) || workspace_bytes < need) return DPS_ERR_WORKSPACE;
    DeviceInfo* d;
    dps_status st = check_device(d);
    if (st != DPS_OK) return st;
    const uint8_t* r = (mode == DPS_MODE_FULL) ? w_resid : nullptr;
    if (launch_moe(mode, enc_per_expert, x, token_of_row, expert_of_row, w_persist, r, y, A, T, N, K, E, workspace,
                   d->status, static_cast<cudaStream_t>(cuda_stream)) != cudaSuccess)
        return DPS_ERR_CUDA;
    return DPS_OK;
}

dps_status dps_stream_status(void* cuda_stream) {
    DeviceInfo* d;
    dps_status st = check_device(d);
    if (st != DPS_OK) return st;
    cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
    int word = 0;
    if (cudaMemcpyAsync(&word, d->status, sizeof(int), cudaMemcpyDeviceToHost, stream) != cudaSuccess)
        return DPS_ERR_CUDA;
    if (cudaMemsetAsync(d->status, 0, sizeof(int), stream) != cudaSuccess) return DPS_ERR_CUDA;
    if (cudaStreamSynchronize(stream) != cudaSuccess) return DPS_ERR_CUDA;
    return word == 0 ? DPS_OK : (word == (int)DPS_ERR_DATA ? DPS_ERR_DATA : DPS_ERR_CUDA);
}

dps_status dps_quantize_activations(const void* x, uint8_t* x_fp8, float* scale, int64_t M, int64_t K,
                                    void* cuda_stream) {
    if (M < 0 || K <= 0 || (K % 16) != 0 || M >= ((int64_t)1 << 31) || K >= ((int64_t)1 << 31)) return DPS_ERR_SHAPE;
    if (M == 0) return DPS_OK;
    if (!x || !x_fp8 || !scale) return DPS_ERR_NULL;
    if (!aligned16(x) || !aligned16(x_fp8)) return DPS_ERR_ALIGN;
    DeviceInfo* d;
    dps_status st = check_device(d);
    if (st != DPS_OK) return st;
    return launch_quantize_activations(x, x_fp8, scale, M, K, d->status, static_cast<cudaStream_t>(cuda_stream)) ==
                   cudaSuccess
               ? DPS_OK
               : DPS_ERR_CUDA;
}

dps_status dps_linear_fp8act(int32_t enc, const uint8_t* x_fp8, const float* scale, const uint8_t* w_persist, void* y,
                             int64_t M, int64_t N, int64_t K, void* cuda_stream) {
    if (!known_encoding(enc)) return DPS_ERR_ENCODING;
    enc = base_enc(enc);   // the persistent byte of a rounded nest is an FP8 value like any other
    if (M < 0 || N <= 0 || K <= 0 || (K % 16) != 0 || (N % 8) != 0) return DPS_ERR_SHAPE;
    if (N >= ((int64_t)1 << 31) || K >= ((int64_t)1 << 31) || M >= ((int64_t)1 << 31)) return DPS_ERR_SHAPE;
    if (M == 0) return DPS_OK;
    if (!x_fp8 || !scale || !w_persist || !y) return DPS_ERR_NULL;
    if (!aligned16(x_fp8) || !aligned16(w_persist) || !aligned16(y)) return DPS_ERR_ALIGN;
    DeviceInfo* d;
    dps_status st = check_device(d);
    if (st != DPS_OK) return st;
    return launch_linear_fp8act(enc, x_fp8, scale, w_persist, y, M, N, K, d->status,
                                static_cast<cudaStream_t>(cuda_stream)) == cudaSuccess
               ? DPS_OK
               : DPS_ERR_CUDA;
}

namespace {
dps_status chunked_copy(void* dst, const void* src, size_t bytes, size_t chunk, cudaMemcpyKind kind, void* cuda_stream) {
    if (bytes == 0) return DPS_OK;
    if (!dst || !src) return DPS_ERR_NULL;
    if (chunk == 0) chunk = (size_t)4 << 20;
    cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
    for (size_t off = 0; off < bytes; off += chunk) {
        const size_t n = bytes - off < chunk ? bytes - off : chunk;
        if (cudaMemcpyAsync(static_cast<char*>(dst) + off, static_cast<const char*>(src) + off, n, kind, stream) !=
            cudaSuccess)
            return DPS_ERR_CUDA;
    }
    return DPS_OK;
}
}  // namespace

dps_status dps_backup_residual(const uint8_t* w_resid, uint8_t* backup_host, size_t bytes, size_t chunk_bytes,
                               void* cuda_stream) {
    return chunked_copy(backup_host, w_resid, bytes, chunk_bytes, cudaMemcpyDeviceToHost, cuda_stream);
}

dps_status dps_restore_residual(uint8_t* w_resid, const uint8_t* backup_host, size_t bytes, size_t chunk_bytes,
                                void* cuda_stream) {
    return chunked_copy(w_resid, backup_host, bytes, chunk_bytes, cudaMemcpyHostToDevice, cuda_stream);
}

dps_status dps_debug_wait_timeout(uint64_t limit_ns, void* cuda_stream) {
    if (limit_ns == 0 || limit_ns > 1000000000ull) return DPS_ERR_SHAPE;   // at most one second
    DeviceInfo* d;
    dps_status st = check_device(d);
    if (st != DPS_OK) return st;
    wait_timeout_selftest_kernel<<<1, 32, 0, static_cast<cudaStream_t>(cuda_stream)>>>(limit_ns, d->status);
    count_launch();
    return cudaGetLastError() == cudaSuccess ? DPS_OK : DPS_ERR_CUDA;
}

int64_t dps_launch_count(void) { return g_launches.load(std::memory_order_relaxed); }

const char* dps_status_string(dps_status status) {
    switch (status) {
        case DPS_OK: return "ok";
        case DPS_ERR_NULL: return "null pointer";
        case DPS_ERR_SHAPE: return "bad shape";
        case DPS_ERR_MODE: return "bad mode";
        case DPS_ERR_ENCODING: return "bad encoding";
        case DPS_ERR_ALIGN: return "misaligned pointer";
        case DPS_ERR_UNSUPPORTED: return "unsupported device or request";
        case DPS_ERR_CUDA: return "CUDA error";
        case DPS_ERR_DATA: return "data-dependent error";
        case DPS_ERR_WORKSPACE: return "workspace missing, misaligned or too small";
    }
    return "unknown status";
}

int dps_version(void) { return 1; }

}  // extern "C"
