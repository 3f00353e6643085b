// FP32 <-> FP64 conversions in integer arithmetic, bit for bit the results of
// the conversion instructions.  The conversions run on the FP64 pipe, which on
// this part retires 2 of them per clock and SM (measured; FP64 FMA 2, FP32 FMA
// 113), so a kernel that converts every element it moves is bound by them: the
// 32,768 outputs of one 128 x 256 tile take 16,000 clocks, as long as the
// tile's tensor-core work.  The integer forms take 6 and 11 operations on the
// integer pipes.  Values outside the common case (FP32 subnormals,
// infinities, NaN, overflow) take the instruction.
#pragma once

#include <stdint.h>

namespace rdm {
namespace {

__device__ __forceinline__ double f32_to_f64(float x) {
    const uint32_t u = __float_as_uint(x);
    const uint32_t m = u & 0x7fffffffu;
    // normal numbers: the exponent re-biased by 896, the fraction shifted by 29
    uint32_t hi = (u & 0x80000000u) | ((m >> 3) + 0x38000000u);
    uint32_t lo = u << 29;
    if (m - 0x00800000u >= 0x7f000000u) {   // zero, subnormal, infinity or NaN
        if (m == 0u) {
            hi = u;
            lo = 0u;
        } else {
            return (double)x;
        }
    }
    return __hiloint2double((int)hi, (int)lo);
}

// round to nearest even
__device__ __forceinline__ float f64_to_f32(double x) {
    const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
    const uint32_t e = (hi >> 20) & 0x7ffu;
    if (e - 897u > 253u) {                  // not a normal FP32 number
        if (((hi & 0x7fffffffu) | lo) == 0u) return __uint_as_float(hi);
        return (float)x;
    }
    // the 29 fraction bits that go: half a unit (less one, plus the kept last
    // bit) is added below them and the carry runs up, into the exponent too
    const uint64_t v = (((uint64_t)(hi & 0x7fffffffu)) << 32 | lo) + (0x0fffffffu + ((lo >> 29) & 1u));
    const uint32_t t = (uint32_t)(v >> 29) - 0xc0000000u;   // exponent bias 1023 -> 127 (modulo 2^32)
    return __uint_as_float(t | (hi & 0x80000000u));
}

// 32 bytes of global memory (32-byte aligned)
__device__ __forceinline__ void ld_f64x4(const double *p, double (&v)[4]) {
    asm volatile("ld.global.v4.f64 {%0,%1,%2,%3}, [%4];"
                 : "=d"(v[0]), "=d"(v[1]), "=d"(v[2]), "=d"(v[3])
                 : "l"(p)
                 : "memory");
}
__device__ __forceinline__ void st_f64x4(double *p, const double (&v)[4]) {
    asm volatile("st.global.v4.f64 [%0], {%1,%2,%3,%4};" ::"l"(p), "d"(v[0]), "d"(v[1]), "d"(v[2]), "d"(v[3]) : "memory");
}

}  // namespace
}  // namespace rdm
