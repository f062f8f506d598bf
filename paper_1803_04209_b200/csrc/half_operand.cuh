// Operands of the emission products in half precision, as exact as tf32 ones wherever that can be seen.
//
// A value rounded to tf32 (or bf16) has at most 11 significant bits, which is what a half-precision number holds, so
// the only thing that keeps a tf32 operand from being stored in two bytes is its exponent.  Every row of an operand --
// a sample's hidden vector, a worker's weights -- is therefore multiplied by a power of two that brings its bound to
// [2^14, 2^15), and the product's row and column are divided by the two powers of two again (exactly) when the
// accumulator is read.  The products and their fp32 accumulation are those of tf32 operands, with one exception: an entry below
// 2^-28 of its row's bound may land among the half-precision subnormals and is then rounded by at most 2^-39 of the bound.
// The bound of a row of weights is its largest entry.  That of a hidden vector is one that the layer's weights and the
// sample's largest input allow, the row sums of |weights| and, for a ReLU layer, the largest positive bias (a unit that a large
// negative bias switches off must not push the others into the subnormals); it lies above the largest entry by as much as the
// terms of that unit cancel.  Half-precision operands take half the bytes from L2 to shared memory and half the
// tensor-core time.
#pragma once
#include <cstdint>
#include <cuda_fp16.h>

namespace cutoff {

// e with bound * 2^e in [2^14, 2^15), 2^e and 2^-e normal: every finite bound from 2^-112 on (a smaller one is scaled by 2^126).
__host__ __device__ inline int half_exponent(uint32_t bound_bits) {
    const int ex = static_cast<int>((bound_bits >> 23) & 0xffu) - 127, e = 14 - ex;
    return e > 126 ? 126 : (e < -113 ? -113 : e);
}
__host__ __device__ inline uint32_t pow2_bits(int e) { return static_cast<uint32_t>(127 + e) << 23; }

__device__ __forceinline__ void half_scale(float bound, float& scale, float& inv_scale) {
    const int e = half_exponent(__float_as_uint(bound));
    scale = __uint_as_float(pow2_bits(e));
    inv_scale = __uint_as_float(pow2_bits(-e));
}

// Two values as one word of two halves (the first in the low half).
__device__ __forceinline__ uint32_t pack_half2(float lo, float hi) {
    uint32_t r;
    asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}

// Rows of `cols` weights into rows of `ld` halves with a power of two per row, one warp per row (when weights are loaded).
// Entries from cols on are zeros.
__global__ void k_half_rows(const float* __restrict__ w, int rows, int cols, int ld, __half* __restrict__ out, float* __restrict__ inv_scale) {
    const int row = static_cast<int>((blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
    if (row >= rows) return;
    const float* src = w + static_cast<size_t>(row) * cols;
    uint32_t big = 0;                                       // bit pattern of the largest magnitude
    for (int k = lane; k < cols; k += 32) big = max(big, __float_as_uint(src[k]) & 0x7fffffffu);
    big = __reduce_max_sync(0xffffffffu, big);
    const int e = big ? half_exponent(big) : 0;
    const float scale = __uint_as_float(pow2_bits(e));
    for (int k = lane; k < ld; k += 32) out[static_cast<size_t>(row) * ld + k] = __float2half_rn(k < cols ? src[k] * scale : 0.0f);
    if (lane == 0) inv_scale[row] = __uint_as_float(pow2_bits(-e));
}

// A hidden vector as the emission products read it: halves with a row pitch of whole 16 bytes, one inverse scale per row,
// and the bound of a row's entries, |entry| <= bound[0] * (largest |input|) + bound[1].  The bound follows from the weights, so it is
// read from device memory: a captured graph outlives the weights it was captured with.
struct HalfRows {
    __half* p;              // [rows][ld]
    float* inv_scale;       // [rows]
    int ld;
    const float* bound;
};
__device__ __forceinline__ void half_scale(const HalfRows& rows, float largest_input, float& scale, float& inv_scale) {
    half_scale(1.01f * fmaf(__ldg(rows.bound), largest_input, __ldg(rows.bound + 1)), scale, inv_scale);
}

}  // namespace cutoff
