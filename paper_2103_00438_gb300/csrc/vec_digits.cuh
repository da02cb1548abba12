// Signed 7-bit digits of a real vector for the digit-slice GEMV (gemv_digits.cu), shared with the
// kernels that produce vectors.
#pragma once

#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cstdint>

namespace wfq {

constexpr int kVecDigits = 8;
constexpr int kVecNotFinite = 1 << 20;   // exponent of a vector with an Inf or NaN

// v 2^(54 - E) rounded to an integer, |v| < 2^E (half up in magnitude); on the bits, since a
// conversion would run on the FP64 pipe.
__device__ __forceinline__ int64_t fixed_point54(double v, int E) {
    const uint32_t hi = (uint32_t)__double2hiint(v), lo = (uint32_t)__double2loint(v);
    const int ex = (int)((hi >> 20) & 0x7ffu);
    const uint32_t mh = (hi & 0xfffffu) | (ex ? 0x100000u : 0u);
    int sh = 1022 + E - (ex ? ex : 1);
    sh = (unsigned)sh > 63u ? 63 : sh;
    const uint64_t f = (((((uint64_t)(mh << 2 | lo >> 30) << 32) | (lo << 2)) >> sh) + 1) >> 1;
    return (hi >> 31) ? -(int64_t)f : (int64_t)f;
}

// Exponent e of a vector, |x| < 2^e, from the bit pattern of its largest magnitude.
__device__ __forceinline__ int vec_exp(unsigned long long bits) {
    const int ex = (int)(bits >> 52);
    return ex == 0x7ff ? kVecNotFinite : ex > 0 ? ex - 1022 : -1021;
}

// x = 2^(e - 5) sum_m e_m 2^(-7 m), |e_m| <= 64, as fp16 at dst[m * stride]
__device__ __forceinline__ void put_vec_digits(double x, int e, __half *dst, int64_t stride) {
    const uint64_t bias = 0x81020408102040ull;   // 64 (128^8 - 1) / 127
    const uint64_t g = e == kVecNotFinite ? bias : (uint64_t)fixed_point54(x, e) + bias;
#pragma unroll
    for (int m = 0; m < kVecDigits; ++m) {
        const unsigned short u = (unsigned short)(0x6400u | (uint32_t)((g >> (7 * (kVecDigits - 1 - m))) & 127u));
        dst[m * stride] = __hsub(__ushort_as_half(u), __ushort_as_half(0x6440u));   // 1024 + u - 1088
    }
}

}  // namespace wfq
