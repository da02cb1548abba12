// Dense FP64-grade products U = D X of many columns on the tensor cores (sm_103a), by exact
// digit slices (the error-free splitting of Ozaki, Ogita, Oishi and Rump, Numer. Algorithms 59,
// 2012, with integer digits).
//
// D_ij (scaled by its row's power of two) and x_jc (scaled by its column's) are written as S
// signed 8-bit digits,
//     D_ij = 2^(E_i - 8S + 2) sum_a d_a 2^(8 (S-1-a)),   |d_a| <= 128,
// and likewise x.  Digits are exact in fp16, their products and the sums of up to 128 x 8 of
// them stay below 2^24, so the FP32 accumulators of the tensor cores hold every partial sum
// exactly.  The digit products d_a e_b with a + b = w < S share one accumulator (weight
// 2^(-8w)); each 128-atom chunk's accumulators are read back, converted to integers and added
// to a 96-bit integer per output.  Nothing is rounded before the final conversion to FP64 (but
// for S = 7 the weights 4 to 6 of a chunk, as one float), and a chunk's sum is one integer, so
// the result does not depend on how the work is split; what is left out is the digits past the
// S-th (2^-62 or 2^-54 of the row's and column's bound) and the digit products with
// a + b >= S.  S = 8 stands for FP64 products, S = 7 for double-float ones (8 for blocks with a
// column that needs it; X is always split into 8); columns whose sum of
// magnitudes is too small beside their largest entry for the bounds above to be below those of plain
// sums are left to plain kernels (digit_cols.cuh).
//
// Why: GB300 has about 2 FP64 FMAs per clock per SM (0.5e12/s) and the double-float product
// costs 12 FP32 operations; the tensor cores do 36 (S = 8) or 28 (S = 7) fp16 digit products
// in less time than either: 20000 atoms x 384 real columns from the pair planes 7.3 ms (69.9 ms
// for double-float FMAs), a 10k-atom sphere x 32 real columns in FP64 0.38 ms (20.5 ms).
//
// Structure (one CTA per SM, 28 warps, stream-K over (column group, row tile, 128-atom chunk)):
//   warps 0-15  epilogue: 8 warps for each of two TMEM slots (S accumulators of 128 x 32), read
//               after each chunk; a thread keeps the 96-bit sums of 16 columns of its row in
//               registers; 64-bit integer atomics onto a zeroed buffer at the end of a tile.
//   warps 16-23 converters: read D (FP64, or the FP32 pairs) one stage ahead into registers,
//               write the S digit planes of a 128 x 32 stage into 64-byte-swizzled shared
//               memory.
//   warp 24     one lane loads the X digit planes by TMA; allocates TMEM.
//   warp 25     one lane issues the MMAs: digit plane a of D against the first S - a digit
//               planes of X, which are consecutive rows of the operand, so that one
//               instruction of N = 32 (S - a) updates the accumulators a .. S-1.
// Registers: launched with 72 a thread (64512); the epilogue keeps 64, warps 24-27 keep 56 and
// the converters take 96: 512 x 64 + 128 x 56 + 256 x 96 = 64512.
// A column group is 64 columns in two halves, each with its own TMEM slot: one half is read
// back while the other's products run.  A group of one half alternates the slots by chunk.
// Every barrier wait is bounded, as in gemm_tc.cuh.
//
// Bound: the conversion and read-back arithmetic about as much as the MMAs (cnt20k, S = 7: 7.0 ms
// in this kernel, 8.1 before the MMAs were issued from a warp-uniform loop; then 7.7 without the
// conversions' loads, 6.9 with one MMA in seven, 7.2 with one read-back column in 16).  Measured
// slower: a third D stage, L2 prefetch of the next chunk (0.5 ms), 16-atom D stages (more
// fences), two converter groups on alternate stages with three register sets (instruction-cache
// misses), skipping the leading digit plane where it is all zeros.
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>

#include "common.h"
#include "digit_cols.cuh"
#include "gemm_tc.cuh"

namespace wfq {
namespace {

using tc::BK;
using tc::BM;
using tc::Params;
using tc::ROWB;

constexpr int DG_CHUNK = 128;          // atoms per accumulator read-back: 2^14 * 8 * 128 = 2^24
constexpr int DG_HALF = 32;            // columns per TMEM slot
constexpr int DG_DIGITS = 8;           // digit planes of X (seven digits: the first seven)
constexpr int DG_STAGES = 2;           // a third D stage (it fits for S = 7) measured slower: less L1
constexpr int DG_EPI_WARPS = 16, DG_CONV_WARPS = 8;
constexpr int DG_EPI_COLS = 2 * DG_HALF / (DG_EPI_WARPS / 4);   // columns an epilogue thread sums
constexpr int DG_THREADS = 32 * (DG_EPI_WARPS + DG_CONV_WARPS + 4);
constexpr int DG_TMA_WARP = DG_EPI_WARPS + DG_CONV_WARPS;
constexpr int DG_ROWS = BM / (4 * DG_CONV_WARPS);             // rows a converter lane handles per stage
constexpr uint32_t DG_A_BYTES = BM * ROWB;                   // one digit plane of a stage

enum DigitSource { SRC_FP64 = 0, SRC_PAIRS = 1 };

struct DigitParams {
    Params p;            // n, err, timeout_ns
    int64_t C;           // real columns
    int nhalf;           // halves of 32 columns
    int mtiles, kchunks;
    int64_t units;       // groups * mtiles * kchunks
    const double *D64;   // SRC_FP64: n x n
    const float *Fh, *Fl;   // SRC_PAIRS: n x ld planes, zero past column n
    int64_t ld;
    const int *dexp;     // n: |D_ij| < 2^dexp[i]
    unsigned long long *acc;   // [n][C][2]: sums in units of 2^-24 and of 2^-56
    DigitCols cols;
};

// v 2^(8S - 2 - E) as an integer (|v| < 2^E), truncated for S = 8, rounded for S = 7; done on
// the bits, since a conversion would run on the FP64 pipe.
template <int S>
__device__ __forceinline__ int64_t fixed_point(double v, int E) {
    const uint32_t hi = (uint32_t)__double2hiint(v), lo = (uint32_t)__double2loint(v);
    const int ex = (int)((hi >> 20) & 0x7ffu);
    const uint32_t mh = (hi & 0xfffffu) | (ex ? 0x100000u : 0u);
    int sh = 1022 + E - (ex ? ex : 1);
    sh = (unsigned)sh > 63u ? 63 : sh;   // (negative only for memory past column n)
    uint64_t f;
    if constexpr (S == 8) {
        f = (((uint64_t)(mh << 9 | lo >> 23) << 32) | (lo << 9)) >> sh;
    } else {
        f = (((uint64_t)(mh << 2 | lo >> 30) << 32) | (lo << 2)) >> sh;
        f = (f + 1) >> 1;
    }
    return (hi >> 31) ? -(int64_t)f : (int64_t)f;
}

// Digit a (0: most significant) of a fixed-point value f is byte S - 1 - a of f + bias, less 128.
template <int S>
__device__ __forceinline__ uint64_t biased(int64_t f) {
    return (uint64_t)f + (S == 8 ? 0x8080808080808080ull : 0x0080808080808080ull);
}

// biased<7> of a float pair h + l, |h| < 2^E, in units of 2^(E - 53): h in units of 2^(E - 22) by
// a magic sum (a conversion would take the 16-per-clock pipe), its remainder and l in units of
// 2^(E - 53).  sh = 2^(22 - E), sl = 2^(53 - E).  The bias is split over the two parts.
__device__ __forceinline__ uint64_t biased_pair(float h, float l, float sh, float sl) {
    constexpr float magic = 12582912.f;   // 1.5 2^23
    const float v = h * sh;
    const float t = __fadd_rn(v, magic);
    const float r = __fsub_rn(v, __fsub_rn(t, magic));   // exact, |r| <= 1/2
    const int it = __float_as_int(t) - (0x4b400000 - 0x01010101);
    const int ib = __float2int_rn(r * 2147483648.f) + __float2int_rn(l * sl) + 0x00808080;
    return (uint64_t)((int64_t)it * 2147483648ll + ib);
}

// v 2^(61 - E) as an integer, truncated; |v| < 2^E.
__device__ __forceinline__ int64_t fixed_float(float v, int E) {
    const uint32_t b = __float_as_uint(v);
    const int ex = (int)((b >> 23) & 0xffu), sh = max(ex, 1) - 89 - E;   // v = m 2^(ex - 150)
    const uint64_t m = (b & 0x7fffffu) | (ex ? 0x800000u : 0u);
    const int64_t f = (int64_t)(sh >= 0 ? m << min(sh, 38) : m >> min(-sh, 31));   // (38: memory past column n)
    return (int)b < 0 ? -f : f;
}

// biased<8> of a float pair in units of 2^(E - 61).
__device__ __forceinline__ uint64_t biased_pair8(float h, float l, int E) {
    return (uint64_t)(fixed_float(h, E) + fixed_float(l, E)) + 0x8080808080808080ull;
}

// Two digits, bytes q and q + 1 of w (q = 0 or 2), as fp16: 0x6400 | u is 1024 + u.
__device__ __forceinline__ uint32_t digits_f16(uint32_t w, bool upper) {
    const uint32_t b = __byte_perm(w, 0x64646464u, upper ? 0x4342u : 0x4140u);
    const __half2 d = __hsub2(*reinterpret_cast<const __half2 *>(&b), __half2half2(__ushort_as_half(0x6480)));   // 1152
    return *reinterpret_cast<const uint32_t *>(&d);
}

__device__ __forceinline__ void tmem_ld1(uint32_t taddr, float &v) {
    uint32_t r;
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=r"(r) : "r"(taddr));
    v = __uint_as_float(r);
}

// (t2:t1) += v
__device__ __forceinline__ void add64(uint32_t &t1, uint32_t &t2, int64_t v) {
    asm("add.cc.u32 %0, %0, %2;\n\taddc.u32 %1, %1, %3;"
        : "+r"(t1), "+r"(t2)
        : "r"((uint32_t)v), "r"((uint32_t)((uint64_t)v >> 32)));
}
// (t2:t1:t0) += v
__device__ __forceinline__ void add96(uint32_t &t0, uint32_t &t1, uint32_t &t2, int64_t v) {
    const uint32_t v1 = (uint32_t)((uint64_t)v >> 32);
    asm("add.cc.u32 %0, %0, %3;\n\taddc.cc.u32 %1, %1, %4;\n\taddc.u32 %2, %2, %5;"
        : "+r"(t0), "+r"(t1), "+r"(t2)
        : "r"((uint32_t)v), "r"(v1), "r"((uint32_t)((int32_t)v1 >> 31)));
}

template <int S, int SRC>
__device__ __forceinline__ void gemm_digits(const CUtensorMap &tm_x, const DigitParams &dp) {
    const Params &p = dp.p;
    constexpr uint32_t A_STAGE = S * DG_A_BYTES;
    constexpr uint32_t B_HALF = S * DG_HALF * ROWB;   // one half's X digit planes of a stage
    constexpr int NA = DG_STAGES;
    constexpr uint32_t B_OFF = NA * A_STAGE;          // X digits follow the D digit stages
    extern __shared__ unsigned char smem_raw[];
    unsigned char *smem =
        reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint64_t *b_full = reinterpret_cast<uint64_t *>(smem + B_OFF + DG_STAGES * 2 * B_HALF);
    uint64_t *b_empty = b_full + DG_STAGES;
    uint64_t *a_full = b_empty + DG_STAGES;
    uint64_t *a_empty = a_full + NA;
    uint64_t *acc_full = a_empty + NA;   // one per TMEM slot
    uint64_t *acc_empty = acc_full + 2;
    uint64_t *drain = acc_empty + 2;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(drain + 1);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);

    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    const int64_t u_begin = dp.units * (int64_t)blockIdx.x / gridDim.x;
    const int64_t u_end = dp.units * ((int64_t)blockIdx.x + 1) / gridDim.x;
    if (threadIdx.x == 0) {
        for (int s = 0; s < DG_STAGES; ++s) {
            tc::mbar_init(tc::smem_u32(b_full + s), 1);
            tc::mbar_init(tc::smem_u32(b_empty + s), 1);
        }
        for (int s = 0; s < NA; ++s) {
            tc::mbar_init(tc::smem_u32(a_full + s), DG_CONV_WARPS);
            tc::mbar_init(tc::smem_u32(a_empty + s), 1);
        }
        for (int e = 0; e < 2; ++e) {
            tc::mbar_init(tc::smem_u32(acc_full + e), 1);
            tc::mbar_init(tc::smem_u32(acc_empty + e), DG_EPI_WARPS / 2);
        }
        tc::mbar_init(tc::smem_u32(drain), 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == DG_TMA_WARP) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc::smem_u32(tmem_slot)),
                     "r"(512)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    const uint32_t smem_base = tc::smem_u32(smem);
    // position of a work unit, advanced unit by unit
    struct Cursor {
        int kc, tile, grp;
    };
    Cursor cur;
    {
        const int64_t per_group = (int64_t)dp.mtiles * dp.kchunks, rem = u_begin % per_group;
        cur.grp = (int)(u_begin / per_group);
        cur.tile = (int)(rem / dp.kchunks);
        cur.kc = (int)(rem % dp.kchunks);
    }
    const int nunits = (int)(u_end - u_begin);
    auto advance = [&] {
        if (++cur.kc == dp.kchunks) {
            cur.kc = 0;
            if (++cur.tile == dp.mtiles) {
                cur.tile = 0;
                ++cur.grp;
            }
        }
    };
    auto halves = [&] { return 2 * cur.grp + 1 < dp.nhalf ? 2 : 1; };

    if (warp < DG_EPI_WARPS) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 64;");
        // ---------------------------------------------------------- epilogue
        const int e = (warp >> 2) & 1, quad = warp & 3, col = (warp >> 3) * DG_EPI_COLS;
        const uint32_t base = tmem + (uint32_t)(e * 256 + col) + ((uint32_t)(quad * 32) << 16);
        uint32_t t0[DG_EPI_COLS], t1[DG_EPI_COLS], t2[DG_EPI_COLS];
#pragma unroll
        for (int c = 0; c < DG_EPI_COLS; ++c) t0[c] = t1[c] = t2[c] = 0u;
        uint32_t uses = 0;
        for (int u = 0; u < nunits; ++u, advance()) {
            const int nh = halves();
            if (nh == 2 || (u & 1) == e) {
                if (!tc::mbar_wait_warp(tc::smem_u32(acc_full + e), uses & 1u, p, 4, abort_flag)) break;
                ++uses;
                tc::tc_fence_after();
#pragma unroll
                for (int c = 0; c < DG_EPI_COLS; ++c) {
                    // |s_w| <= (w + 1) 2^21: the first two pairs combine in 32 bits.  Four weights
                    // at a time, which keeps the sums of 16 columns in registers.
                    float v[4];
#pragma unroll
                    for (int w = 0; w < 4; ++w) tmem_ld1(base + (uint32_t)(w * DG_HALF + c), v[w]);
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                    const int s01 = __float2int_rn(v[0]) * 256 + __float2int_rn(v[1]);
                    const int s23 = __float2int_rn(v[2]) * 256 + __float2int_rn(v[3]);
                    add64(t1[c], t2[c], (int64_t)s01 * 65536 + s23);
#pragma unroll
                    for (int w = 4; w < S; ++w) tmem_ld1(base + (uint32_t)(w * DG_HALF + c), v[w - 4]);
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                    int64_t lo;
                    if constexpr (S == 8) {
                        lo = (int64_t)__float2int_rn(v[0]) * 16777216 + (int64_t)__float2int_rn(v[1]) * 65536 +
                             (int64_t)__float2int_rn(v[2]) * 256 + __float2int_rn(v[3]);
                    } else {
                        // weights 4 to 6 as one float in units of 2^-7 of weight 4: exact below
                        // 2^24 units (as for digits of varying signs), else rounded at 2^-24 of
                        // s_4, at most 2^-52 of the bounds' product per nonzero entry
                        const float f = fmaf(v[0], 128.f, fmaf(v[1], 0.5f, v[2] * 0.001953125f));
                        lo = (int64_t)__float2int_rn(f) * 131072;
                    }
                    add96(t0[c], t1[c], t2[c], lo);
                }
                tc::tc_fence_before();
                __syncwarp();
                if (lane == 0) tc::mbar_arrive(tc::smem_u32(acc_empty + e));
            }
            if (cur.kc == dp.kchunks - 1 || u + 1 == nunits) {
                // end of this CTA's share of the tile: integer sums, any order gives the same
                const int64_t row = (int64_t)cur.tile * BM + quad * 32 + lane;
                const int64_t col0 = (int64_t)(2 * cur.grp + (nh == 2 ? e : 0)) * DG_HALF + col;
#pragma unroll
                for (int c = 0; c < DG_EPI_COLS; ++c) {
                    if (row < p.n && col0 + c < dp.C) {
                        unsigned long long *a = dp.acc + 2 * (row * dp.C + col0 + c);
                        atomicAdd(a, ((unsigned long long)t2[c] << 32) | t1[c]);
                        atomicAdd(a + 1, (unsigned long long)t0[c]);
                    }
                    t0[c] = t1[c] = t2[c] = 0u;
                }
            }
        }
    } else if (warp < DG_EPI_WARPS + DG_CONV_WARPS) {
        // ---------------------------------------------------------- converters
        asm volatile("setmaxnreg.inc.sync.aligned.u32 96;");
        const int cw = warp - DG_EPI_WARPS;
        // A lane takes 4 consecutive atoms of DG_ROWS rows, 8 lanes a row's 32 atoms; the stage
        // after the one being converted is on its way into the other register set.  (The code is
        // kept to two copies of the conversion: four times as much, with deeper prefetch, ran
        // into instruction-cache misses and was half as fast.)
        const int lr = cw * 4 + (lane >> 3), lk = (lane & 7) * 4;
        const bool vec = (p.n & 1) == 0;   // FP64 rows are 16-byte aligned
        const int nst = nunits * (DG_CHUNK / BK);
        const int64_t nn = p.n * p.n;
        struct Regs {   // (h, l) of 4 atoms per row, or their 4 doubles; the rows' exponents, a byte each
            float4 a[DG_ROWS], b[DG_ROWS];
            uint32_t ex;
        };
        static_assert(DG_ROWS == 4, "four exponents to a word");
        int sub = 0, ex_tile = -1;   // stage within the cursor's chunk; tile of exps
        uint32_t exps = 0;
        // The cursor's stage; advances it.  Rows past n read the last row (never stored); entries
        // past column n meet zero digits of X, so whatever is in memory there will do.
        auto load = [&](Regs &f) {
            const int64_t k = (int64_t)cur.kc * DG_CHUNK + sub * BK + lk;
            const int64_t r0 = (int64_t)cur.tile * BM + lr;
            if (cur.tile != ex_tile) {
                ex_tile = cur.tile;
                exps = 0;
#pragma unroll
                for (int q = 0; q < DG_ROWS; ++q)
                    exps |= (uint32_t)(__ldg(dp.dexp + min(r0 + q * 4 * DG_CONV_WARPS, p.n - 1)) & 0xff) << (8 * q);
            }
            f.ex = exps;
#pragma unroll
            for (int q = 0; q < DG_ROWS; ++q) {
                const int64_t i = min(r0 + q * 4 * DG_CONV_WARPS, p.n - 1);
                if constexpr (SRC == SRC_PAIRS) {
                    f.a[q] = __ldg(reinterpret_cast<const float4 *>(dp.Fh + i * dp.ld + k));
                    f.b[q] = __ldg(reinterpret_cast<const float4 *>(dp.Fl + i * dp.ld + k));
                } else if (vec) {
                    const int64_t o = i * p.n + k;
                    f.a[q] = __ldg(reinterpret_cast<const float4 *>(dp.D64 + min(o, nn - 2)));
                    f.b[q] = __ldg(reinterpret_cast<const float4 *>(dp.D64 + min(o + 2, nn - 2)));
                } else {
                    const int64_t o = i * p.n + k;
                    auto get = [&](int64_t at, float &l, float &h) {
                        const float2 v = __ldg(reinterpret_cast<const float2 *>(dp.D64 + min(at, nn - 1)));
                        l = v.x;
                        h = v.y;
                    };
                    get(o, f.a[q].x, f.a[q].y);
                    get(o + 1, f.a[q].z, f.a[q].w);
                    get(o + 2, f.b[q].x, f.b[q].y);
                    get(o + 3, f.b[q].z, f.b[q].w);
                }
            }
            if (++sub == DG_CHUNK / BK) {
                sub = 0;
                advance();
            }
        };
        auto convert = [&](const Regs &f, uint32_t base) {
#pragma unroll
            for (int q = 0; q < DG_ROWS; ++q) {
                const int ex = (int)(f.ex << (24 - 8 * q)) >> 24;
                uint64_t g[4];
                if constexpr (SRC == SRC_PAIRS && S == 8) {
                    g[0] = biased_pair8(f.a[q].x, f.b[q].x, ex);
                    g[1] = biased_pair8(f.a[q].y, f.b[q].y, ex);
                    g[2] = biased_pair8(f.a[q].z, f.b[q].z, ex);
                    g[3] = biased_pair8(f.a[q].w, f.b[q].w, ex);
                } else if constexpr (SRC == SRC_PAIRS) {
                    const float sh = __int_as_float((127 + 22 - ex) << 23);
                    const float sl = __int_as_float((127 + 53 - ex) << 23);
                    g[0] = biased_pair(f.a[q].x, f.b[q].x, sh, sl);
                    g[1] = biased_pair(f.a[q].y, f.b[q].y, sh, sl);
                    g[2] = biased_pair(f.a[q].z, f.b[q].z, sh, sl);
                    g[3] = biased_pair(f.a[q].w, f.b[q].w, sh, sl);
                } else {
                    auto dbl = [](float l, float h) { return __hiloint2double(__float_as_int(h), __float_as_int(l)); };
                    g[0] = biased<S>(fixed_point<S>(dbl(f.a[q].x, f.a[q].y), ex));
                    g[1] = biased<S>(fixed_point<S>(dbl(f.a[q].z, f.a[q].w), ex));
                    g[2] = biased<S>(fixed_point<S>(dbl(f.b[q].x, f.b[q].y), ex));
                    g[3] = biased<S>(fixed_point<S>(dbl(f.b[q].z, f.b[q].w), ex));
                }
                const int row = q * 4 * DG_CONV_WARPS + lr;
                // 64-byte swizzle: 16-byte chunk index XOR (row / 2) mod 4
                const uint32_t off =
                    base + (uint32_t)row * ROWB + (uint32_t)(((lk >> 3) ^ ((lr >> 1) & 3)) * 16) + (uint32_t)(lk & 4) * 2;
#pragma unroll
                for (int w = 0; w < 2; ++w) {   // low words: digits S-1 .. S-4; high words: the others
                    uint32_t v[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k) v[k] = (uint32_t)(g[k] >> (32 * w));
#pragma unroll
                    for (int b2 = 0; b2 < 2; ++b2) {   // bytes 2 b2 and 2 b2 + 1 of the word
                        const uint32_t p01 = __byte_perm(v[0], v[1], b2 ? 0x7362u : 0x5140u);
                        const uint32_t p23 = __byte_perm(v[2], v[3], b2 ? 0x7362u : 0x5140u);
#pragma unroll
                        for (int b = 0; b < 2; ++b) {
                            const int digit = S - 1 - (4 * w + 2 * b2 + b);
                            if (digit < 0) continue;
                            asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(off + (uint32_t)digit * DG_A_BYTES),
                                         "r"(digits_f16(p01, b != 0)), "r"(digits_f16(p23, b != 0))
                                         : "memory");
                        }
                    }
                }
            }
        };
        uint32_t buf = 0, par = 0;
        auto step = [&](int j, const Regs &now, Regs &next) -> bool {
            if (j + 1 < nst) load(next);
            if (!tc::mbar_wait_warp(tc::smem_u32(a_empty + buf), par ^ 1u, p, 1, abort_flag)) return false;
            convert(now, smem_base + buf * A_STAGE);
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(tc::smem_u32(a_full + buf));
            if (++buf == NA) {
                buf = 0;
                par ^= 1u;
            }
            return true;
        };
        Regs r0, r1;
        load(r0);
#pragma unroll 1
        for (int j = 0; j < nst; j += 2) {
            if (!step(j, r0, r1)) break;
            if (!step(j + 1, r1, r0)) break;   // the number of stages is even
        }
    } else {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 56;");
        if (warp == DG_TMA_WARP && lane == 0) {
            // ---------------------------------------------------------- TMA producer (X digits)
            uint32_t it = 0;
            bool aborted = false;
            for (int u = 0; u < nunits && !aborted; ++u, advance()) {
                const int nh = halves();
                for (int st = 0; st < DG_CHUNK / BK; ++st, ++it) {
                    const uint32_t s = it & 1u;
                    if (!tc::mbar_wait(tc::smem_u32(b_empty + s), ((it >> 1) & 1u) ^ 1u, p, 1, abort_flag)) {
                        aborted = true;
                        break;
                    }
                    const uint32_t fb = tc::smem_u32(b_full + s);
                    tc::mbar_expect_tx(fb, (uint32_t)nh * B_HALF);
                    for (int h = 0; h < nh; ++h)
                        tc::tma_load_2d(smem_base + B_OFF + (2 * s + (uint32_t)h) * B_HALF, &tm_x, fb,
                                        cur.kc * DG_CHUNK + st * BK, (2 * cur.grp + h) * DG_DIGITS * DG_HALF);
                }
            }
            if (aborted) {   // wait (bounded) for the copies of the last stages issued
                volatile int no_abort = 0;
                for (uint32_t j = it > DG_STAGES ? it - DG_STAGES : 0; j < it; ++j)
                    tc::mbar_wait(tc::smem_u32(b_full + (j & 1u)), (j >> 1) & 1u, p, 1, &no_abort);
            }
        } else if (warp == DG_TMA_WARP + 1) {
            const bool el = tc::elect_one();
            // ---------------------------------------------------------- MMA issuer
            uint32_t it = 0, uses = 0, abuf = 0, apar = 0;   // uses: phase of each slot's barriers, a bit each
            bool aborted = false;
            for (int u = 0; u < nunits && !aborted; ++u, advance()) {
                const int nh = halves();
                for (int st = 0; st < DG_CHUNK / BK && !aborted; ++st, ++it) {
                    const uint32_t s = it & 1u;
                    aborted = !tc::mbar_wait(tc::smem_u32(b_full + s), (it >> 1) & 1u, p, 2, abort_flag) ||
                              !tc::mbar_wait(tc::smem_u32(a_full + abuf), apar, p, 2, abort_flag);
                    if (aborted) break;
                    tc::tc_fence_after();
                    // shared-memory descriptors hold the address in units of 16 bytes
                    const uint64_t da = tc::desc_k_sw64(smem_base + abuf * A_STAGE);
                    for (int h = 0; h < nh; ++h) {
                        const int slot = nh == 2 ? h : (u & 1);
                        if (st == 0) {
                            aborted = !tc::mbar_wait(tc::smem_u32(acc_empty + slot), ((uses >> slot) & 1u) ^ 1u, p, 3, abort_flag);
                            if (aborted) break;
                            tc::tc_fence_after();
                        }
                        const uint64_t db = tc::desc_k_sw64(smem_base + B_OFF + (2 * s + (uint32_t)h) * B_HALF);
                        const uint32_t d = tmem + (uint32_t)(slot * 256);
#pragma unroll 1
                        for (int ks = 0; ks < 2; ++ks) {
#pragma unroll
                            for (int a = 0; a < S; ++a) {
                                // fp16 operands, FP32 accumulator, N = 32 (S - a)
                                const uint32_t idesc =
                                    (1u << 4) | ((uint32_t)((S - a) * DG_HALF >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
                                if (el) tc::umma_bf16(d + (uint32_t)(a * DG_HALF),
                                              da + (uint64_t)(uint32_t)(a * (DG_A_BYTES >> 4) + ks * 2), db + (uint64_t)(ks * 2),
                                              idesc, (a == 0 && st == 0 && ks == 0) ? 0u : 1u);
                            }
                        }
                        if (st == DG_CHUNK / BK - 1) {
                            if (el) tc::umma_commit(tc::smem_u32(acc_full + slot));
                            uses ^= 1u << slot;
                        }
                    }
                    if (aborted) break;
                    if (el) tc::umma_commit(tc::smem_u32(a_empty + abuf));
                    if (el) tc::umma_commit(tc::smem_u32(b_empty + s));
                    if (++abuf == NA) {
                        abuf = 0;
                        apar ^= 1u;
                    }
                }
            }
            if (el) tc::umma_commit(tc::smem_u32(drain));
            volatile int no_abort = 0;
            tc::mbar_wait(tc::smem_u32(drain), 0u, p, 5, &no_abort);
        }
    }
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    if (warp == DG_TMA_WARP) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
    }
}

// Eight digits; or seven if they do for every column, else eight -- in one launch (DG_BOTH), or in two of
// which one finds nothing to do (4 us): with both bodies in a kernel its registers spill, which
// costs 4% (20000 atoms x 384 real columns 8.79 ms against 8.45).
enum DigitMode { DG_EIGHT, DG_BOTH, DG_IF_SEVEN, DG_IF_EIGHT };
constexpr int64_t DG_BOTH_MAX = 4096;   // atoms
template <int SRC, DigitMode MODE>
__global__ void __launch_bounds__(DG_THREADS, 1)
    k_gemm_digits(const __grid_constant__ CUtensorMap tm7, const __grid_constant__ CUtensorMap tm8, const DigitParams dp) {
    const DigitCols &cols = dp.cols;
    if constexpr (MODE == DG_IF_EIGHT) wait_for_previous();
    bool mine = false, low = false;
    for (int64_t c = threadIdx.x; c < dp.C; c += DG_THREADS)
        if (col_state(cols, c) == COL_DIGITS) {
            mine = true;
            if constexpr (MODE != DG_EIGHT)
                low = low || !sum_suffices(cols.csum[c], cols.csum[c ^ 1], cols.cmax[c], cols.cmax[c ^ 1], cols.thr7);
        }
    if (!__syncthreads_or(mine)) return;   // plain sums take every column
    const bool eight = MODE == DG_EIGHT || __syncthreads_or(low);
    if constexpr (MODE == DG_BOTH || MODE == DG_IF_SEVEN) {
        if (!eight) {
            gemm_digits<7, SRC>(tm7, dp);
            return;
        }
    }
    if constexpr (MODE != DG_IF_SEVEN) {
        if (eight) gemm_digits<8, SRC>(tm8, dp);
    }
}

// cmax[c] = the largest |x| of column c as its bit pattern (monotonic; 0x7ff0... and above:
// not finite).  X: n x C row-major.  Block: 32 columns x 8 row lanes over a run of rows.
__global__ void __launch_bounds__(256) k_col_absmax(int64_t n, int64_t C, int64_t rpb, const double *__restrict__ X,
                                                    unsigned long long *__restrict__ cmax) {
    __shared__ unsigned long long sm[8][33];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int64_t c = (int64_t)blockIdx.y * 32 + tx;
    const int64_t r0 = (int64_t)blockIdx.x * rpb, r1 = min(n, r0 + rpb);
    unsigned long long m = 0;
    if (c < C)
        for (int64_t r = r0 + ty; r < r1; r += 8) {
            const unsigned long long b = (unsigned long long)__double_as_longlong(X[r * C + c]) & 0x7fffffffffffffffull;
            m = b > m ? b : m;
        }
    sm[ty][tx] = m;
    __syncthreads();
    if (ty == 0 && c < C) {
#pragma unroll
        for (int q = 1; q < 8; ++q) m = sm[q][tx] > m ? sm[q][tx] : m;
        atomicMax(cmax + c, m);
    }
}

// Exponent e of a column, |x| < 2^e, from the bit pattern of its largest magnitude.
__device__ __forceinline__ int col_exp(unsigned long long bits) {
    const int ex = (int)(bits >> 52);
    return ex > 0 ? ex - 1022 : -1021;
}

// X digits: planes [half][digit][32 columns][npad] fp16, zero past row n and column C.  Block:
// 64 atoms x 32 columns.
__global__ void __launch_bounds__(256) k_split_digits(int64_t n, int64_t npad, int64_t C, const double *__restrict__ X,
                                                      DigitCols cols, __half *__restrict__ planes) {
    constexpr int S = DG_DIGITS;
    __shared__ uint64_t t[64][33];
    __shared__ unsigned qsum[8][33];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int64_t a0 = (int64_t)blockIdx.x * 64, c = (int64_t)blockIdx.y * 32 + tx;
    const unsigned long long mb = c < C ? cols.cmax[c] : 0ull;
    const bool finite = mb < 0x7ff0000000000000ull;
    const int e = col_exp(mb);
    unsigned q = 0;   // 2^8 |x| / 2^e
#pragma unroll
    for (int r = ty; r < 64; r += 8) {
        const int64_t a = a0 + r;
        const double v = (a < n && c < C && finite) ? X[a * C + c] : 0.0;
        const int64_t f = fixed_point<S>(v, e);
        q += (unsigned)((uint64_t)(f < 0 ? -f : f) >> (8 * S - 10));
        t[r][tx] = biased<S>(f);
    }
    qsum[ty][tx] = q;
    __syncthreads();
    if (ty == 0 && c < C) {
#pragma unroll
        for (int k = 1; k < 8; ++k) q += qsum[k][tx];
        atomicAdd(cols.csum + c, q);
    }
#pragma unroll
    for (int cr = ty; cr < 32; cr += 8) {
        const uint64_t v0 = t[2 * tx][cr], v1 = t[2 * tx + 1][cr];
#pragma unroll
        for (int d = 0; d < S; ++d) {
            const int sft = 8 * (S - 1 - d);
            const uint32_t w = (uint32_t)((v0 >> sft) & 0xffu) | ((uint32_t)((v1 >> sft) & 0xffu) << 8);
            const int64_t row = ((int64_t)blockIdx.y * S + d) * DG_HALF + cr;
            *reinterpret_cast<uint32_t *>(planes + row * npad + a0 + 2 * tx) = digits_f16(w, false);
        }
    }
}

// U = 2^(E_i + e_c + unit) (acc0 + acc1 2^-32); a column that is not finite gives NaN; columns of
// the plain sums are left to them.
__global__ void __launch_bounds__(256) k_digits_finish(int64_t n, int64_t C, const unsigned long long *__restrict__ acc,
                                                       const int *__restrict__ dexp, DigitCols cols, int unit,
                                                       double *__restrict__ U) {
    wait_for_previous();
    const int64_t e = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (e >= n * C) return;
    const int64_t i = e / C, c = e - i * C;
    const ColState st = col_state(cols, c);
    if (st == COL_PLAIN) return;
    if (st == COL_NOT_FINITE) {
        U[e] = __longlong_as_double(0x7ff8000000000000ll);
        return;
    }
    const ulonglong2 a = reinterpret_cast<const ulonglong2 *>(acc)[e];
    // the low words of the shares sum to less than 2^32 x CTAs: carry their upper part exactly
    const long long hi = (long long)a.x + (long long)(a.y >> 32);
    const unsigned lo = (unsigned)a.y;
    const double v = fma((double)lo, 0x1p-32, (double)hi);
    U[e] = scalbn(v, dexp[i] + col_exp(cols.cmax[c]) + unit);
}

template <int SRC, DigitMode MODE>
int launch_digits(const __half *planes, const DigitParams &dp, int64_t npad, int grid, cudaStream_t s) {
    constexpr int S = DG_DIGITS;
    constexpr size_t smem = (size_t)DG_STAGES * S * DG_A_BYTES + (size_t)DG_STAGES * 2 * S * DG_HALF * ROWB + 1024 + 256;
    static_assert(smem <= (size_t)tc::kMaxDynSmem, "digit stages exceed shared memory");
    std::string msg;
    CUtensorMap m7, m8;
    const uint64_t rows = (uint64_t)dp.nhalf * DG_DIGITS * DG_HALF;
    if (!tc::make_map(&m7, planes, (uint64_t)npad, rows, (uint64_t)npad, 7u * DG_HALF, &msg) ||
        !tc::make_map(&m8, planes, (uint64_t)npad, rows, (uint64_t)npad, 8u * DG_HALF, &msg))
        return fail(WFQ_ECUDA, "digit-slice GEMM: " + msg);
    static std::atomic<uint64_t> smem_set{0};
    cudaError_t e = tc::allow_max_smem(k_gemm_digits<SRC, MODE>, smem_set);
    if (e == cudaSuccess) {
        note_launch();
        if constexpr (MODE == DG_IF_EIGHT) {
            e = launch_overlapped(k_gemm_digits<SRC, MODE>, dim3((unsigned)grid), dim3(DG_THREADS), smem, s, m7, m8, dp);
        } else {
            k_gemm_digits<SRC, MODE><<<(unsigned)grid, DG_THREADS, smem, s>>>(m7, m8, dp);
            e = cudaGetLastError();
        }
    }
    if (e != cudaSuccess) {
        cudaGetLastError();
        return fail(WFQ_ECUDA, std::string("digit-slice GEMM: ") + cudaGetErrorString(e));
    }
    return WFQ_OK;
}

template <int SRC>
int launch_double_float(const __half *planes, const DigitParams &dp, int64_t npad, int grid, cudaStream_t s) {
    if (dp.p.n <= DG_BOTH_MAX) return launch_digits<SRC, DG_BOTH>(planes, dp, npad, grid, s);
    WFQ_TRY((launch_digits<SRC, DG_IF_SEVEN>(planes, dp, npad, grid, s)));
    return launch_digits<SRC, DG_IF_EIGHT>(planes, dp, npad, grid, s);
}

}  // namespace

unsigned digit_sum_threshold(const wfq_geom *g, int log2_ratio) {
    const double t = std::ceil(std::ldexp(1.0, 8 + log2_ratio + g->dexp_max) / g->dmin);
    return t < 4294967295.0 ? (unsigned)t : 4294967295u;
}

static size_t plane_elems(const wfq_geom *g, int64_t C) {
    return (size_t)((C + DG_HALF - 1) / DG_HALF) * DG_DIGITS * DG_HALF * g->npad;
}
static size_t sum_words(const wfq_geom *g, int64_t C) { return (size_t)2 * g->n * C + C + (C + 1) / 2; }

size_t digits_workspace(const wfq_geom *g, int64_t C) {
    return g->digits_ok && (g->D64 || g->Dfh) ? plane_elems(g, C) * sizeof(__half) + sum_words(g, C) * sizeof(unsigned long long) : 0;
}

int digits_product(const wfq_geom *g, bool fp64, int64_t C, const double *X, double *U, DigitColsBuf &cols, cudaStream_t s,
                   int *err) {
    wfq_ctx *ctx = g->ctx;
    const int64_t n = g->n, npad = g->npad;
    const int nhalf = (int)((C + DG_HALF - 1) / DG_HALF);
    const bool pairs = !fp64 && g->Dfh != nullptr;
    DevBuf<__half> planes;
    const size_t words = sum_words(g, C);
    WFQ_TRY(planes.alloc(ctx, plane_elems(g, C), s));
    WFQ_TRY(cols.buf.alloc(ctx, words, s));
    unsigned long long *acc = cols.buf.ptr, *cmax = acc + 2 * n * C;
    // What is left out per entry, in 2^(E + e): products with a + b = S, (S - 1) 2^(14 - 8 S) against 2^12
    // (2^11 from pairs), the truncated or rounded last digits and, S = 7, the float of weights 4 to 6 (2^-24
    // of 5 2^14 2^7 in its units): below 2^-57 (S = 8), 2^-50 (S = 7); against 2^-53 or 2^-48.
    cols.dc = fp64 ? DigitCols{cmax, reinterpret_cast<unsigned *>(cmax + C), digit_sum_threshold(g, -58 + 53), 0}
                   : DigitCols{cmax, reinterpret_cast<unsigned *>(cmax + C), digit_sum_threshold(g, -57 + 48),
                               digit_sum_threshold(g, -50 + 48)};
    WFQ_CUDA(cudaMemsetAsync(acc, 0, sizeof(unsigned long long) * words, s));
    const int64_t rpb = std::max<int64_t>(32, round_up((n + 4 * ctx->num_sms - 1) / (4 * ctx->num_sms), 8));
    k_col_absmax<<<dim3((unsigned)((n + rpb - 1) / rpb), (unsigned)nhalf), 256, 0, s>>>(n, C, rpb, X, cmax);
    note_launch();
    k_split_digits<<<dim3((unsigned)(npad / 64), (unsigned)nhalf), 256, 0, s>>>(n, npad, C, X, cols.dc, planes.ptr);
    note_launch();
    WFQ_CUDA(cudaGetLastError());
    DigitParams dp{};
    dp.p.n = n;
    dp.p.err = err ? err : ctx->dev_err;
    dp.p.timeout_ns = 4000000000ull;
    dp.C = C;
    dp.nhalf = nhalf;
    dp.mtiles = (int)(npad / BM);
    dp.kchunks = (int)(npad / DG_CHUNK);
    dp.units = (int64_t)((nhalf + 1) / 2) * dp.mtiles * dp.kchunks;
    dp.D64 = g->D64;
    dp.Fh = g->Dfh;
    dp.Fl = g->Dfl;
    dp.ld = g->ldf;
    dp.dexp = g->dexp;
    dp.acc = acc;
    dp.cols = cols.dc;
    const int grid = (int)std::min<int64_t>(ctx->num_sms, dp.units);
    if (fp64)
        WFQ_TRY((launch_digits<SRC_FP64, DG_EIGHT>(planes.ptr, dp, npad, grid, s)));
    else if (pairs)
        WFQ_TRY(launch_double_float<SRC_PAIRS>(planes.ptr, dp, npad, grid, s));
    else
        WFQ_TRY(launch_double_float<SRC_FP64>(planes.ptr, dp, npad, grid, s));
    WFQ_CUDA(launch_overlapped(k_digits_finish, dim3((unsigned)((n * C + 255) / 256)), dim3(256), 0, s, n, C, acc, g->dexp,
                               cols.dc, pairs ? -35 : -36, U));
    note_launch();
    WFQ_CUDA(cudaGetLastError());
    return WFQ_OK;
}

}  // namespace wfq
