// Load-time kernels: tensor statistics for the encoding choice, nested split, reconstruction.
// Paper: "Mapper: Semi-Unified Memory Abstraction" ("Persistent Region" paragraph) for the
// split; "Scheduler: Dual-Precision Execution" for the reconstruction and the per-layer
// encoding choice.  All are pure streams with fully coalesced accesses (consecutive lanes take
// consecutive items).
#include "bits.cuh"
#include "dps_internal.h"

namespace dps {

namespace {

constexpr int kThreads = 256;

__device__ __forceinline__ uint4 ldg_stream(const void* p) {
    uint4 v;
    asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p));
    return v;
}

__device__ __forceinline__ uint32_t max_mag2(uint32_t a, uint32_t m) {
    // per-half max of (word & 0x7FFF)
    a &= 0x7FFF7FFFu;
    return __vmaxu2(a, m);
}

__global__ void __launch_bounds__(kThreads) magnitude_stat_kernel(const uint4* __restrict__ w, int64_t n8,
                                                                   unsigned* stat) {
    uint32_t m = 0;
    for (int64_t i = blockIdx.x * (int64_t)kThreads + threadIdx.x; i < n8; i += (int64_t)gridDim.x * kThreads) {
        uint4 v = ldg_stream(w + i);
        m = max_mag2(v.x, m);
        m = max_mag2(v.y, m);
        m = max_mag2(v.z, m);
        m = max_mag2(v.w, m);
    }
    unsigned best = max(m & 0xFFFFu, m >> 16);
    for (int o = 16; o > 0; o >>= 1) best = max(best, __shfl_xor_sync(0xFFFFFFFFu, best, o));
    if ((threadIdx.x & 31) == 0 && best) atomicMax(stat, best);
}

// Streams of one block each: a block takes kUnits * kThreads consecutive items and is done, so the block
// scheduler balances the SMs and there is no last round of a grid-stride loop.  WIDE: an item is 16 weights --
// 32 bytes of FP16 (one 256-bit access) and 16 bytes of each plane; it needs the FP16 tensor on a 32-byte
// boundary.  Else an item is 8 weights: 16 bytes of FP16, 8 bytes of each plane, which a 16-byte boundary allows.
// Bound by HBM.  Split / rebuild of 90 M weights: 68.5 / 66.7 us as a grid-stride loop over 8-weight items, 58.7 /
// 57.6 us like this; a device-to-device copy of the FP16 tensor takes 57.7 us.
constexpr int kUnits = 2;

template <bool WIDE>
struct Item;
template <>
struct Item<true> {
    static constexpr int kPairs = 8;     // packed FP16 pairs
    static __device__ __forceinline__ void load(const uint32_t* p, uint32_t (&v)[8]) {
        asm volatile("ld.global.nc.L1::no_allocate.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                     : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
                     : "l"(p));
    }
    static __device__ __forceinline__ void store(uint32_t* p, const uint32_t (&v)[8]) {
        asm volatile("st.global.v8.b32 [%8], {%0,%1,%2,%3,%4,%5,%6,%7};" ::"r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]),
                     "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "l"(p)
                     : "memory");
    }
    static __device__ __forceinline__ void load_plane(const uint32_t* p, uint32_t (&v)[4]) {
        asm volatile("ld.global.nc.L1::no_allocate.v4.b32 {%0,%1,%2,%3}, [%4];"
                     : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3])
                     : "l"(p));
    }
    static __device__ __forceinline__ void store_plane(uint32_t* p, const uint32_t (&v)[4]) {
        *reinterpret_cast<uint4*>(p) = make_uint4(v[0], v[1], v[2], v[3]);
    }
};
template <>
struct Item<false> {
    static constexpr int kPairs = 4;
    static __device__ __forceinline__ void load(const uint32_t* p, uint32_t (&v)[4]) { Item<true>::load_plane(p, v); }
    static __device__ __forceinline__ void store(uint32_t* p, const uint32_t (&v)[4]) { Item<true>::store_plane(p, v); }
    static __device__ __forceinline__ void load_plane(const uint32_t* p, uint32_t (&v)[2]) {
        asm volatile("ld.global.nc.L1::no_allocate.v2.b32 {%0,%1}, [%2];" : "=r"(v[0]), "=r"(v[1]) : "l"(p));
    }
    static __device__ __forceinline__ void store_plane(uint32_t* p, const uint32_t (&v)[2]) {
        *reinterpret_cast<uint2*>(p) = make_uint2(v[0], v[1]);
    }
};

// The two words an encoding choice goes through: `flag` (device memory) and `host` (mapped host memory) receive
// `call`, the number of this call, from a block that meets a word above kAutoLimit.
struct AutoCheck {
    volatile unsigned* flag;
    volatile unsigned* host;
    unsigned call;
};
constexpr uint32_t kAutoLimit2 = 0x3F003F00u;   // |w| <= 1.75 in both halves of a register

// FP16 -> planes.  AUTO: the split and the statistic in ONE pass (4 bytes per weight instead of 2 + 4): the planes
// are written as E4M3 on the assumption that all weights are in range, which nearly all tensors are.  A block
// that meets a word out of range publishes that and stores nothing; blocks that start later see it and stop
// before they store, and the host then runs the E5M2 split over the whole tensor.
template <int ENC, bool WIDE, bool AUTO>
__global__ void __launch_bounds__(kThreads) split_kernel(const uint32_t* __restrict__ w, uint32_t* __restrict__ p,
                                                         uint32_t* __restrict__ r, int64_t items, AutoCheck check) {
    using I = Item<WIDE>;
    constexpr int kPairs = I::kPairs;
    const int64_t i0 = (int64_t)blockIdx.x * (kUnits * kThreads) + threadIdx.x;
    uint32_t a[kUnits][kPairs];
#pragma unroll
    for (int u = 0; u < kUnits; ++u)
        if (i0 + u * kThreads < items) I::load(w + (i0 + u * kThreads) * kPairs, a[u]);
    if (AUTO) {
        const bool stop = threadIdx.x == 0 && *check.flag == check.call;
        uint32_t m = 0;
#pragma unroll
        for (int u = 0; u < kUnits; ++u)
            if (i0 + u * kThreads < items) {
#pragma unroll
                for (int j = 0; j < kPairs; ++j) m = __vmaxu2(m, a[u][j] & 0x7FFF7FFFu);
            }
        const bool out = __vmaxu2(m, kAutoLimit2) != kAutoLimit2;
        if (out) {
            *check.flag = check.call;
            *check.host = check.call;
        }
        if (__syncthreads_or(out || stop)) return;
    }
#pragma unroll
    for (int u = 0; u < kUnits; ++u) {
        const int64_t i = i0 + u * kThreads;
        if (i < items) {
            uint32_t pp[kPairs / 2], rr[kPairs / 2];
#pragma unroll
            for (int j = 0; j < kPairs / 2; ++j) split4<ENC>(a[u][2 * j], a[u][2 * j + 1], pp[j], rr[j]);
            I::store_plane(p + i * (kPairs / 2), pp);
            I::store_plane(r + i * (kPairs / 2), rr);
        }
    }
}

template <int ENC, bool FULL, bool WIDE>
__global__ void __launch_bounds__(kThreads) reconstruct_kernel(const uint32_t* __restrict__ p,
                                                               const uint32_t* __restrict__ r, uint32_t* __restrict__ w,
                                                               int64_t items) {
    using I = Item<WIDE>;
    constexpr int kPairs = I::kPairs;
    const int64_t i0 = (int64_t)blockIdx.x * (kUnits * kThreads) + threadIdx.x;
    uint32_t pp[kUnits][kPairs / 2], rr[kUnits][kPairs / 2];
#pragma unroll
    for (int u = 0; u < kUnits; ++u) {
        const int64_t i = i0 + u * kThreads;
        if (i < items) {
            I::load_plane(p + i * (kPairs / 2), pp[u]);
            if (FULL) I::load_plane(r + i * (kPairs / 2), rr[u]);
        }
    }
#pragma unroll
    for (int u = 0; u < kUnits; ++u) {
        const int64_t i = i0 + u * kThreads;
        if (i < items) {
            uint32_t out[kPairs];
#pragma unroll
            for (int j = 0; j < kPairs / 2; ++j) join4<ENC, FULL>(pp[u][j], FULL ? rr[u][j] : 0u, out[2 * j], out[2 * j + 1]);
            I::store(w + i * kPairs, out);
        }
    }
}

inline bool wide_items(const void* w) { return (reinterpret_cast<uintptr_t>(w) & 31u) == 0; }
inline int64_t stream_blocks(int64_t items) { return (items + kUnits * kThreads - 1) / (kUnits * kThreads); }

template <int ENC, bool AUTO>
cudaError_t launch_split_enc(const uint16_t* w, uint8_t* p, uint8_t* r, int64_t n, AutoCheck check, cudaStream_t stream) {
    const uint32_t* ww = reinterpret_cast<const uint32_t*>(w);
    uint32_t* pp = reinterpret_cast<uint32_t*>(p);
    uint32_t* rr = reinterpret_cast<uint32_t*>(r);
    const bool wide = wide_items(w);
    const int64_t items = n / (wide ? 16 : 8);
    const dim3 grid((unsigned)stream_blocks(items));
    if (wide) split_kernel<ENC, true, AUTO><<<grid, kThreads, 0, stream>>>(ww, pp, rr, items, check);
    else split_kernel<ENC, false, AUTO><<<grid, kThreads, 0, stream>>>(ww, pp, rr, items, check);
    count_launch();
    return cudaGetLastError();
}

template <int ENC, bool FULL>
cudaError_t launch_reconstruct_enc(const uint8_t* p, const uint8_t* r, uint16_t* w, int64_t n, cudaStream_t stream) {
    const uint32_t* pp = reinterpret_cast<const uint32_t*>(p);
    const uint32_t* rr = reinterpret_cast<const uint32_t*>(r);
    uint32_t* ww = reinterpret_cast<uint32_t*>(w);
    const bool wide = wide_items(w);
    const int64_t items = n / (wide ? 16 : 8);
    const dim3 grid((unsigned)stream_blocks(items));
    if (wide) reconstruct_kernel<ENC, FULL, true><<<grid, kThreads, 0, stream>>>(pp, rr, ww, items);
    else reconstruct_kernel<ENC, FULL, false><<<grid, kThreads, 0, stream>>>(pp, rr, ww, items);
    count_launch();
    return cudaGetLastError();
}

int stream_grid(int64_t items) {
    int64_t blocks = (items + kThreads - 1) / kThreads;
    int64_t cap = (int64_t)sm_count() * 8;
    return (int)(blocks < cap ? (blocks > 0 ? blocks : 1) : cap);
}

// Empty kernel launched (as an ordinary, fully ordered launch) after the planes have been written.
// A linear kernel that follows on the stream may start early and fetch planes before it waits for
// its predecessor; with this launch in between, that predecessor is the fence, and the fence did
// not start before the split kernel had finished and its writes were visible.
__global__ void plane_fence_kernel() {}

}  // namespace

cudaError_t launch_magnitude_stat(const uint16_t* w, int64_t n, unsigned* stat, cudaStream_t stream) {
    int64_t n8 = n / 8;
    magnitude_stat_kernel<<<stream_grid(n8), kThreads, 0, stream>>>(reinterpret_cast<const uint4*>(w), n8, stat);
    count_launch();
    return cudaGetLastError();
}

cudaError_t launch_split(const uint16_t* w, uint8_t* p, uint8_t* r, int64_t n, int enc, cudaStream_t stream) {
    cudaError_t e;
    if (enc == kEncE4M3) e = launch_split_enc<kEncE4M3, false>(w, p, r, n, AutoCheck{}, stream);
    else if (enc == kEncE5M2) e = launch_split_enc<kEncE5M2, false>(w, p, r, n, AutoCheck{}, stream);
    else if (enc == kEncE4M3R) e = launch_split_enc<kEncE4M3R, false>(w, p, r, n, AutoCheck{}, stream);
    else e = launch_split_enc<kEncE5M2R, false>(w, p, r, n, AutoCheck{}, stream);
    if (e != cudaSuccess) return e;
    plane_fence_kernel<<<1, 32, 0, stream>>>();
    count_launch();
    return cudaGetLastError();
}

cudaError_t launch_split_auto(const uint16_t* w, uint8_t* p, uint8_t* r, int64_t n, unsigned* flag, unsigned* host,
                              unsigned call, cudaStream_t stream) {
    return launch_split_enc<kEncE4M3, true>(w, p, r, n, AutoCheck{flag, host, call}, stream);
}

cudaError_t launch_reconstruct(const uint8_t* p, const uint8_t* r, uint16_t* w, int64_t n, int enc,
                               cudaStream_t stream) {
    // without the residual plane the rounded nests read like their truncated siblings: P is an FP8 value
    if (!r) enc = base_enc(enc);
    if (enc == kEncE4M3)
        return r ? launch_reconstruct_enc<kEncE4M3, true>(p, r, w, n, stream)
                 : launch_reconstruct_enc<kEncE4M3, false>(p, r, w, n, stream);
    if (enc == kEncE5M2)
        return r ? launch_reconstruct_enc<kEncE5M2, true>(p, r, w, n, stream)
                 : launch_reconstruct_enc<kEncE5M2, false>(p, r, w, n, stream);
    if (enc == kEncE4M3R) return launch_reconstruct_enc<kEncE4M3R, true>(p, r, w, n, stream);
    return launch_reconstruct_enc<kEncE5M2R, true>(p, r, w, n, stream);
}

}  // namespace dps
