// Which columns of X the digit-slice products serve, and which plain sums take instead.
//
// Digits hold D_ij to a fraction of 2^E_i (its row's bound) and x_j to one of 2^e (its column's): what
// is left out is at most u_d 2^(E + e) per nonzero x_j, however small D_ij x_j is.  Plain sums err by at
// most u |D_ij| |x_j| per entry and step (u = 2^-53 in FP64, 2^-48 in double-float).  So a column that a
// few entries dominate loses bits in the rows far from them.  With dmin a lower bound of all entries of
// D (erf(r / s) / r at the structure's diagonal), the digits' bound is no larger than the plain one if
//     sum_j |x_j| >= (u_d / u) 2^(E + e) / dmin:
// a column is taken in digits only then.  csum: sum_j floor(2^8 |x_j| / 2^e), from the splitting kernel;
// thr = 2^8 (u_d / u) 2^max(E) / dmin.  A 20000-atom tube of carbon asks for an average |x_j| of 0.004
// (u_d / u = 2^-5) or 0.03 (2^-2) of 2^e; normal random columns have 0.1 to 0.2.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

namespace wfq {

struct DigitCols {
    unsigned long long *cmax;   // bits of the largest |x| of each column (null: no columns to sort out)
    unsigned *csum;
    unsigned thr;
};

enum ColState { COL_ZERO, COL_DIGITS, COL_PLAIN, COL_NOT_FINITE };

__device__ __forceinline__ ColState col_state(const DigitCols &d, int64_t c) {
    const unsigned long long m = d.cmax[c];
    if (m == 0ull) return COL_ZERO;
    if (m >= 0x7ff0000000000000ull) return COL_NOT_FINITE;
    return d.csum[c] < d.thr ? COL_PLAIN : COL_DIGITS;
}

// The plain kernels' share: dominated columns, and for FP64 sums (not_finite) those with an Inf or
// NaN, whose signs and NaNs they reproduce; every column when there are none to sort out.
__device__ __forceinline__ bool col_plain(const DigitCols &d, int64_t c, bool not_finite) {
    if (!d.cmax) return true;
    const ColState s = col_state(d, c);
    return s == COL_PLAIN || (not_finite && s == COL_NOT_FINITE);
}

}  // namespace wfq
