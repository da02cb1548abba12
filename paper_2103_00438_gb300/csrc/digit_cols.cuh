// Which columns of X the digit-slice products serve, and which plain sums take instead.
//
// Digits hold D_ij to a fraction of 2^E_i (its row's bound) and x_j to one of 2^e (its column's): what
// is left out is at most u_d 2^(E + e) per nonzero x_j, however small D_ij x_j is.  Plain sums err by at
// most u |D_ij| |x_j| per entry and step (u = 2^-53 in FP64, 2^-48 in double-float).  So a column that a
// few entries dominate loses bits in the rows far from them.  With dmin a lower bound of all entries of
// D (erf(r / s) / r at the structure's diagonal), the digits' bound is no larger than the plain one if
//     sum_j |x_j| >= (u_d / u) 2^(E + e) / dmin:
// a column is taken in digits only then (the sum may be that of the other part of the complex
// column: its error stands beside the same |y|).  csum: sum_j floor(2^8 |x_j| / 2^e), from the splitting kernel;
// thr = 2^8 (u_d / u) 2^max(E) / dmin.  A 20000-atom tube of carbon asks for an average |x_j| of 0.004
// of 2^e in FP64 blocks (u_d / u = 2^-5, eight digits), 0.03 (2^-2, seven digits) or 0.0002 (2^-9, eight)
// in double-float ones; normal random columns have 0.1 to 0.2, the charges of a solve down to 0.01.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

namespace wfq {

struct DigitCols {
    unsigned long long *cmax;   // bits of the largest |x| of each column (null: no columns to sort out)
    unsigned *csum;
    unsigned thr;
    unsigned thr7;   // seven digits do when every column of the digits has this sum
};

// Whether real column c (its sum and largest magnitude) or its partner in a complex column, whose rows it
// shares, has the sum: the errors of both parts are beside the same |y|.  Magnitudes' exponents are
// compared (ex: biased, of the largest |x|).
__device__ __forceinline__ bool sum_suffices(unsigned own, unsigned other, unsigned long long mown, unsigned long long mother,
                                             unsigned thr) {
    if (own >= thr) return true;
    if (mother == 0ull || mother >= 0x7ff0000000000000ull) return false;
    const int up = max((int)(mother >> 52), 1) - max((int)(mown >> 52), 1);   // other's unit is 2^up own's
    if (up >= 0) return up > 31 || ((unsigned long long)other << up) >= thr;
    return -up < 32 && (other >> -up) >= thr;
}

constexpr unsigned kSumOfOne = 128;   // csum of a column that is not zero: at least its largest entry's

enum ColState { COL_ZERO, COL_DIGITS, COL_PLAIN, COL_NOT_FINITE };

__device__ __forceinline__ ColState col_state(const DigitCols &d, int64_t c) {
    const unsigned long long m = d.cmax[c];
    if (m == 0ull) return COL_ZERO;
    if (m >= 0x7ff0000000000000ull) return COL_NOT_FINITE;
    return sum_suffices(d.csum[c], d.csum[c ^ 1], m, d.cmax[c ^ 1], d.thr) ? COL_DIGITS : COL_PLAIN;
}

// The plain kernels' share: dominated columns, and for FP64 sums (not_finite) those with an Inf or
// NaN, whose signs and NaNs they reproduce; every column when there are none to sort out.
__device__ __forceinline__ bool col_plain(const DigitCols &d, int64_t c, bool not_finite) {
    if (!d.cmax) return true;
    const ColState s = col_state(d, c);
    return s == COL_PLAIN || (not_finite && s == COL_NOT_FINITE);
}

// The same for groups of C <= 4 vectors (gemv_digits.cu, u_d = 2^-53 of the bounds, u = 2^-48): a group is
// left to double-float sums if any of its vectors is dominated.  vsum: sum_j floor(2^8 |v_j| / 2^e) or a
// lower bound; all ones for a vector of zeros and one that is not finite (NaN either way).  vmax: largest
// magnitudes of the parts of complex columns, two by two; null: real vectors.
struct VecSums {
    const unsigned *vsum;
    const unsigned long long *vmax;
    unsigned thr;
    __device__ __forceinline__ bool plain(int C) const {
        bool any = false;
        for (int c = 0; c < C; ++c) {
            const bool ok = vmax ? sum_suffices(vsum[c], vsum[c ^ 1], vmax[c], vmax[c ^ 1], thr) : vsum[c] >= thr;
            any = any || !ok;
        }
        return any;
    }
};

}  // namespace wfq
