// Token rows of 32 channels in shared memory as bulk tensor copies leave them (64-byte rows, swizzled), read by ldmatrix without
// bank conflicts: as rows (contraction over channels) or transposed (contraction over tokens).
#pragma once

#include "direct_common.cuh"
#include "tma_map.h"

namespace bra {

// Offsets of a lane for ldmatrix, rows from a multiple of eight on: eight rows, a chunk of 16 bytes per matrix; 16 rows, two chunks
// (exclusive or with 32: the other two), which are the A fragment of 16 rows or, transposed, two B fragments.
__device__ __forceinline__ uint32_t row_swizzle(int row) { return (row >> 1) & 3; }
__device__ __forceinline__ uint32_t rows8_offset(int lane) { return (lane & 7) * 64 + (((lane >> 3) ^ row_swizzle(lane & 7)) << 4); }
__device__ __forceinline__ uint32_t rows16_offset(int lane) {
    const int row = lane & 15;
    return row * 64 + (((lane >> 4) ^ row_swizzle(row)) << 4);
}

// c (16 x 8) = A * B^T, B fragments of eight token rows: k step 0: b0, b1, k step 1: b0, b1
__device__ __forceinline__ void mma_rows8(float (&c)[4], const uint32_t (&a)[2][4], const uint32_t (&b)[4]) {
    mma_bf16_zero(c, a[0], b[0], b[1]);
    mma_bf16(c, a[1], b[2], b[3]);
}
// Row r of a tile's accumulators times f as bf16, 16 bytes (channels 8 t4 .. 8 t4 + 7 of a plane) per lane: the lanes of a quad
// hold a pair of every chunk and trade them for a whole one.
__device__ __forceinline__ uint4 pack_row_of_quad(const float (&acc)[4][4], int r, float f, int t4) {
    uint32_t w[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) w[i] = pack2_bf16(acc[i][2 * r] * f, acc[i][2 * r + 1] * f);
    const bool b0 = t4 & 1, b1 = t4 & 2;
    // 4 x 4 transpose over (register, lane): exchange of bit 0, then of bit 1
    uint32_t s0 = b0 ? w[0] : w[1], s1 = b0 ? w[2] : w[3];
    s0 = __shfl_xor_sync(0xffffffffu, s0, 1);
    s1 = __shfl_xor_sync(0xffffffffu, s1, 1);
    if (b0) { w[0] = s0; w[2] = s1; } else { w[1] = s0; w[3] = s1; }
    s0 = b1 ? w[0] : w[2]; s1 = b1 ? w[1] : w[3];
    s0 = __shfl_xor_sync(0xffffffffu, s0, 2);
    s1 = __shfl_xor_sync(0xffffffffu, s1, 2);
    if (b1) { w[0] = s0; w[1] = s1; } else { w[2] = s0; w[3] = s1; }
    return make_uint4(w[0], w[1], w[2], w[3]);
}

}  // namespace bra
