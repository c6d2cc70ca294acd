// Weights of the proposal network's convolutions in the shared-memory layout of
// the tensor-core operands (k_conv_tc.cu), so that a CTA's copy is contiguous.
// Per layer: the forward operand (BF16, rows = output channels padded to 16 or
// 64, k = tap x input channel padded to 16 or 64) and the input gradient's
// (TF32 of the BF16 value, rows = 64 input channels, k = tap x output channel
// padded to 8 or 64).  Padding stays zero.
#pragma once
#include <cstddef>
#include <cuda_bf16.h>

namespace {

__host__ __device__ constexpr int pack_fwd_ci(int ci) { return ci <= 16 ? 16 : 64; }
__host__ __device__ constexpr int pack_fwd_co(int co) { return co <= 16 ? 16 : 64; }
__host__ __device__ constexpr int pack_bwd_co(int co) { return co <= 8 ? 8 : 64; }
__host__ __device__ constexpr size_t pack_fwd_bytes(int ci, int co) {
    return (size_t)pack_fwd_co(co) * 9 * pack_fwd_ci(ci) * 2;
}
__host__ __device__ constexpr size_t pack_bwd_bytes(int co) { return (size_t)64 * 9 * pack_bwd_co(co) * 4; }

// Byte offset of element (row, k): rows of KT elements of esz bytes in 8-row x
// 16-byte core matrices, consecutive along k.
__host__ __device__ __forceinline__ size_t pack_off(int row, int k, int KT, int esz) {
    const int per = 16 / esz;
    return (size_t)(row >> 3) * ((KT / per) * 128) + (size_t)(k / per) * 128 + (row & 7) * 16 + (k % per) * esz;
}

// Weight rel = (o ci + c) 9 + t of a layer, value v, into both operands (bwd
// may be null).
__device__ __forceinline__ void pack_weight(int ci, int co, int rel, float v, unsigned char* fwd, unsigned char* bwd) {
    const int o = rel / (ci * 9), c = rel / 9 % ci, t = rel % 9;
    const __nv_bfloat16 h = __float2bfloat16(v);
    *(__nv_bfloat16*)(fwd + pack_off(o, t * pack_fwd_ci(ci) + c, 9 * pack_fwd_ci(ci), 2)) = h;
    if (bwd) *(float*)(bwd + pack_off(c, t * pack_bwd_co(co) + o, 9 * pack_bwd_co(co), 4)) = __bfloat162float(h);
}

}  // namespace
