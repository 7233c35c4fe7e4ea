// The per-query terms of the backward, -lse/scale and -D with D_i = sum_c dO_ic O_ic, and the tile they are stored in.
// Shared by the pre kernel and the single-tile kernel, so that a row's terms are the same bits on either path.
#pragma once
#include <cstdint>
#include <cuda_bf16.h>

namespace dcp {

// A [128 queries x 16] bf16 tile in the MMA's shared-memory layout (8x8 core matrices, column halves 2048 bytes apart):
// columns 0-2 hold -lse/scale, 8-10 hold -D, each split into three bf16 parts whose sum carries 24 bits.  Rows past the
// sequence hold kNoRow and 0, which makes their probabilities vanish without masking.
constexpr int kTermTileBytes = 128 * 16 * 2;
constexpr float kNoRow = -1e30f;

// dO . O over eight columns.  D_i adds these partial sums in a tree, partners half the columns apart first, neighbours last.
__device__ __forceinline__ float chunk_dot(const uint4 a, const uint4 b) {
    const uint32_t aw[4] = {a.x, a.y, a.z, a.w}, bw[4] = {b.x, b.y, b.z, b.w};
    float sum = 0.f;
#pragma unroll
    for (int w = 0; w < 4; ++w) {
        const float2 x = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&aw[w]));
        const float2 y = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&bw[w]));
        sum += x.x * y.x + x.y * y.y;
    }
    return sum;
}

// Stores a term of row r into its tile (role 0: -lse/scale, 1: -D).
__device__ __forceinline__ void store_term(uint8_t* tile, int r, int role, float x) {
    const __nv_bfloat16 b0 = __float2bfloat16(x);
    const float r1 = x - __bfloat162float(b0);
    const __nv_bfloat16 b1 = __float2bfloat16(r1);
    const __nv_bfloat16 b2 = __float2bfloat16(r1 - __bfloat162float(b1));
    uint4 v;
    v.x = (uint32_t)__bfloat16_as_ushort(b0) | ((uint32_t)__bfloat16_as_ushort(b1) << 16);
    v.y = (uint32_t)__bfloat16_as_ushort(b2);
    v.z = 0u;
    v.w = 0u;
    *reinterpret_cast<uint4*>(tile + role * 2048 + (r / 8) * 128 + (r % 8) * 16) = v;
}

}  // namespace dcp
