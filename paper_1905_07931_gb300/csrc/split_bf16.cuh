// Float32 factors as sums of three bf16 parts, for products of float32
// accuracy on the tensor cores (the dense weight gradient, the dense
// sparse-matrix products).
//
// x = x1 + x2 + x3, each the round to nearest of what is left. A part holds 8
// significant bits, so with 2^e the power of two at or below |x|: |x2| <=
// 2^(e-8), |x3| <= 2^(e-17), and nothing is left: the sum is x, all 24 bits.
// For that no part may fall below bf16's least value, so both factors are
// taken times 2^24 (exactly: float32's smallest value, 2^-149, becomes 2^-125,
// a normal number) and the product times 2^-48. The price is the range at the
// other end: values of 2^28 and more, infinities and NaN are left to the
// kernels of the CUDA cores (split_fits), as products and long sums of scaled
// ones would overflow.
//
// A product is taken as x1 y1 + (x1 y2 + x2 y1 + x2 y2 + x1 y3 + x3 y1). What
// is left out, x2 y3 + x3 y2 + x3 y3, is at most 2^-24 |x y|, one rounding of
// float32 (2^-28 of it on average over the significands).
//
// tcgen05.mma adds into its float32 accumulator with truncation (measured: 2
// bits beyond the accumulator's last place are kept, the sum is cut toward
// zero), which would cost a long chain more than its factors' bits are worth.
// So x1 y1 and the small products have an accumulator each. That of x1 y1 is
// read after every 64 columns (four steps) and added to float32 register sums
// with round to nearest; a single product x1 y1 has 16 bits and is exact
// there. The other's truncations are 2^-8 smaller: it is read after 512
// columns. (Sums of 32 columns: the additions' own rounding outweighs what
// truncation they save, error over 4096 columns 2.1e-7 against 1.6e-7, and the
// tensor cores wait for the reading back: 4096 x 4096 x 1024 161 us against
// 139 for the gradient.)
#pragma once

#include <cuda_bf16.h>

#include "common.cuh"

namespace csrt {

constexpr float kSplitUp = 0x1p24f;      // each factor times this
constexpr float kSplitDown = 0x1p-48f;   // their product times this
constexpr int kSplitChunk = 64;          // columns per sum of x1 y1
constexpr int kSplitFlush = 8;           // such chunks per sum of the small products
// The small products x3 y1, x1 y3, x2 y2, x2 y1, x1 y2: the parts (from 0) of
// both factors, a nibble each. (A loop over them: unrolled, their addresses
// spilled from the issuing warp's 32 registers, 10% of the gradient's time.)
constexpr int kSplitPartsA = 0x01102, kSplitPartsB = 0x10120;

// (NaN does not fit either)
__device__ __forceinline__ bool split_fits(float v) { return fabsf(v) < 0x1p28f; }

// The parts of two scaled factors.
__device__ __forceinline__ void split_bf16(float2 v, __nv_bfloat162 &p1, __nv_bfloat162 &p2, __nv_bfloat162 &p3) {
    v.x *= kSplitUp;
    v.y *= kSplitUp;
    p1 = __float22bfloat162_rn(v);
    const float2 f1 = __bfloat1622float2(p1);
    const float2 r1 = make_float2(v.x - f1.x, v.y - f1.y);
    p2 = __float22bfloat162_rn(r1);
    const float2 f2 = __bfloat1622float2(p2);
    p3 = __float22bfloat162_rn(make_float2(r1.x - f2.x, r1.y - f2.y));
}

}  // namespace csrt
