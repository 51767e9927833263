// Host-side construction of TMA tensor maps (cuTensorMapEncodeTiled through the runtime's driver
// entry-point query, so the library does not link against libcuda).
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace dps {

using EncodeTiledFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                   const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                   CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

inline EncodeTiledFn encode_fn() {
    static EncodeTiledFn fn = [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess)
            p = nullptr;
        return reinterpret_cast<EncodeTiledFn>(p);
    }();
    return fn;
}

// 2-D row-major tensor [rows][cols] of `elem_bytes`-sized elements, tiles of box_rows x box_cols;
// elements outside the tensor read as zero.  `promotion`: the stretch of memory L2 fetches for a missing line.
// Planes that are streamed from HBM once take 256 bytes: a tile is 64 or 128 bytes wide, and DRAM serves two
// neighbouring tiles of a row in one burst more cheaply than in two (Mixtral expert layers, 256 tokens: 383 /
// 215 -> 345 / 192 us in full mode, 217 / 124 -> 208 / 117 us in fast mode; hidden-8192 gate/up at 64 tokens 186 ->
// 169 us in full mode, 95 -> 92 us in fast mode; Llama-7B layers 0-2 %).  Planes that many token tiles share come
// out of L2 for the most part and keep 128 bytes (256: +1 % time at 256 tokens).
inline bool make_map_2d(CUtensorMap* map, const void* base, CUtensorMapDataType dt, int elem_bytes, uint64_t rows,
                        uint64_t cols, uint32_t box_rows, uint32_t box_cols, CUtensorMapSwizzle swizzle,
                        CUtensorMapL2promotion promotion = CU_TENSOR_MAP_L2_PROMOTION_L2_128B) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    const cuuint64_t dims[2] = {cols, rows};
    const cuuint64_t strides[1] = {cols * (uint64_t)elem_bytes};
    const cuuint32_t box[2] = {box_cols, box_rows};
    const cuuint32_t estr[2] = {1, 1};
    return fn(map, dt, 2, const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle,
              promotion, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace dps
