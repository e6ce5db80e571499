// Host side of bulk tensor copies (TMA): tensor maps over the [B,H,W,C] tensors of a call.
#pragma once

#include <cuda.h>

#include "bra_internal.h"

namespace bra {

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// The driver's encoder, looked up through the runtime (the library does not link against the driver).
inline EncodeTiledFn tma_encoder() {
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

// Tensor map over a [B,H0,W0,C] tensor of this GPU's memory (bf16 or fp32 by d.esize); box = (bc channels, bx, by
// tokens, 1 image); what a box covers outside the map is zero.
inline bool make_map(CUtensorMap* m, const void* base, const Dims& d, int bc, int bx, int by, CUtensorMapSwizzle sw) {
    EncodeTiledFn enc = tma_encoder();
    if (!enc) return false;
    const cuuint64_t tok = (cuuint64_t)d.C * d.esize;
    const cuuint64_t dims[4] = {(cuuint64_t)d.C, (cuuint64_t)d.W0, (cuuint64_t)d.H0, (cuuint64_t)d.B};
    const cuuint64_t strides[3] = {tok, d.W0 * tok, (cuuint64_t)d.H0 * d.W0 * tok};
    const cuuint32_t box[4] = {(cuuint32_t)bc, (cuuint32_t)bx, (cuuint32_t)by, 1};
    const cuuint32_t es[4] = {1, 1, 1, 1};
    return enc(m, d.esize == 2 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4,
               const_cast<void*>(base), dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, sw,
               CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace bra
