// Signed 7-bit digits of a real vector for the digit-slice GEMV (gemv_digits.cu), shared with the
// kernels that produce vectors.
#pragma once

#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cstdint>

#include "dfloat.cuh"
#include "common.h"

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

// x = 2^(e - 5) sum_m e_m 2^(-7 m), |e_m| <= 64, as fp16 at dst[m * stride].  Returns
// floor(2^8 |x| / 2^e).
__device__ __forceinline__ unsigned put_vec_digits(double x, int e, __half *dst, int64_t stride) {
    const uint64_t bias = 0x81020408102040ull;   // 64 (128^8 - 1) / 127
    const int64_t f = e == kVecNotFinite ? 0 : fixed_point54(x, e);
    const uint64_t g = (uint64_t)f + bias;
#pragma unroll
    for (int m = 0; m < kVecDigits; ++m) {
        const unsigned short u = (unsigned short)(0x6400u | (uint32_t)((g >> (7 * (kVecDigits - 1 - m))) & 127u));
        dst[m * stride] = __hsub(__ushort_as_half(u), __ushort_as_half(0x6440u));   // 1024 + u - 1088
    }
    return (unsigned)((uint64_t)(f < 0 ? -f : f) >> 46);
}

// Row i, vector d of C from the symmetric product's partial sums: the items of tile row K = i / 64,
// then the tiles (I, K), I < K, in double-float in that order.
__device__ __forceinline__ double dsymv_sum(const SymPartials &p, int C, int64_t i, int d) {
    const int64_t K = i / kSymTile, r = i % kSymTile;
    float sh = 0.f, sl = 0.f;
    for (int q = p.item_start[K]; q < p.item_start[K + 1]; ++q) {
        const float2 v = p.rowpart[((int64_t)q * kSymTile + r) * C + d];
        df_add(sh, sl, v.x, v.y);
    }
    for (int64_t I = 0; I < K; ++I) {
        const float2 v = p.colpart[(sym_tile(I, K, p.T) * kSymTile + r) * C + d];
        df_add(sh, sl, v.x, v.y);
    }
    return (double)sh + (double)sl;
}

}  // namespace wfq
