// Operand planes of the split-precision products: layout, scales and the
// hi / lo split of eight neighbouring elements, shared by the kernel that makes
// them from the FP64 values (k_tc.cu) and the compaction (k_compact.cu).
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <stdint.h>

namespace rdm {
namespace {

// element (r, c) of plane `plane` (0 hi, 1 lo) of a B x B block: the two
// planes' 8-row groups alternate (8 B elements each), so that one copy
// brings both and both are K-major core-matrix operands with a 32 B-byte
// stride between 8-row groups; inside a group, core matrix (c/8) at 64
// elements
template <int B>
__device__ __forceinline__ int pair_offset(int r, int c, int plane) {
    return (r >> 3) * (16 * B) + plane * (8 * B) + ((c >> 3) << 6) + ((r & 7) << 3) + (c & 7);
}

// operand scale of a matrix with largest block norm mx: 2^floor(log2(2^14 / mx))
// for fp16 (the largest element then sits below 2^14, far from fp16 overflow,
// and values down to ~1e-9 of it stay normal); 1 for bf16, whose exponent
// range is FP32's
__device__ __forceinline__ float matrix_scale(unsigned mxbits, bool fp16) {
    const float mx = __uint_as_float(mxbits);
    float s = 1.f;
    if (fp16 && mx > 0.f) {
        int e = (int)floorf(log2f(16384.f / mx));
        e = max(-60, min(60, e));
        s = ldexpf(1.f, e);
    }
    return s;
}

// x sc = hi + lo for columns c0 .. c0 + 7 (c0 a multiple of 8) of row r: one
// row of a core matrix of each plane
template <bool BF16, int B>
__device__ __forceinline__ void store_planes(uint16_t *blk, int r, int c0, const float (&xs)[8], float sc) {
    uint16_t h[8], l[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const float x = xs[k] * sc;
        if (BF16) {
            const __nv_bfloat16 bh = __float2bfloat16_rn(x);
            const __nv_bfloat16 bl = __float2bfloat16_rn(x - __bfloat162float(bh));
            h[k] = __bfloat16_as_ushort(bh);
            l[k] = __bfloat16_as_ushort(bl);
        } else {
            const __half hh = __float2half_rn(x);
            const __half hl = __float2half_rn(x - __half2float(hh));
            h[k] = __half_as_ushort(hh);
            l[k] = __half_as_ushort(hl);
        }
    }
    uint4 hv, lv;
    hv.x = h[0] | ((uint32_t)h[1] << 16); hv.y = h[2] | ((uint32_t)h[3] << 16);
    hv.z = h[4] | ((uint32_t)h[5] << 16); hv.w = h[6] | ((uint32_t)h[7] << 16);
    lv.x = l[0] | ((uint32_t)l[1] << 16); lv.y = l[2] | ((uint32_t)l[3] << 16);
    lv.z = l[4] | ((uint32_t)l[5] << 16); lv.w = l[6] | ((uint32_t)l[7] << 16);
    *reinterpret_cast<uint4 *>(blk + pair_offset<B>(r, c0, 0)) = hv;
    *reinterpret_cast<uint4 *>(blk + pair_offset<B>(r, c0, 1)) = lv;
}

}  // namespace
}  // namespace rdm
