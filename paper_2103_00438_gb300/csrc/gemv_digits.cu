// U = D V for up to 4 real vectors on the tensor cores by exact digit slices (sm_103a): the D
// product of the shifted solver and of few-column applies from the stored float pairs.
//
// As gemm_digits.cu, D and the vectors are split into signed digits that fp16 holds exactly and
// that multiply and add without rounding in the FP32 accumulators, here
//     D_ij = 2^(E - 10) sum_k d_k 2^(-11 k),  k < 5,  |d_k| <= 2048,
//     v_j  = 2^(e - 5)  sum_m e_m 2^(-7 m),   m < 8,  |e_m| <= 64,
// with one accumulator per (k, m, vector): sums of 128 products stay within 2^24.  The terms
// with 11 k + 7 m <= 56 are kept (digits and terms left out: 2^-53 of the bounds' product at
// most); each read-back adds them to 64-bit integers, so the result does not depend on the split
// of the work.  Vectors that few entries dominate, for which that bound can exceed the
// double-float sums', are left to those (VecSums).
//
// Why: the double-float multiply-adds cost 12 FP32 operations per entry and vector.  A digit
// split costs 12.5 packed instructions per entry for all vectors, and D being symmetric
// (Eq. 3) every entry above the diagonal serves two products from the same shared-memory tile:
// D_IJ v_J (rows as M, K-major) and D_IJ^T v_I (columns as M, the same bytes as an MN-major
// operand).  So only the upper triangle is read, of the symmetric tiles or of the full planes:
// 4 bytes per entry of the full matrix instead of 8.  20000 atoms, 3 vectors: 385 us (675 from
// the full planes with double-float multiply-adds, 701 from the tiles); 15000 (tiles): 444 -> 213.
//
// Bound (20000 atoms, us): HBM 236, the conversions alone 238, the products alone 305 (40 clocks
// each on average, M = 64 and 128, N = 16 and 32: small ones cost their operand reads), all
// together 385; with two stages of 80 KiB a stage's conversion and products overlap only in
// part.  Measured slower or equal: 16 converter warps with symmetry, prefetching the planes into
// L2 (a bulk prefetch per row: 1190), a single row slot.
//
// Work unit (stage): 128 rows (block a) x 64 columns (block J), J >= 2 a; for J = 2 a the lower
// 64 x 64 half lies below the diagonal (zero here, its transpose belongs to J = 2 a + 1).
// One CTA per SM takes a contiguous range of units:
//   warps 0-3   row epilogue, warps 4-7 column epilogue: tensor memory -> integers; the rows'
//               sums stay in registers to the end of the block, the columns' go out per unit,
//               both by 64-bit integer atomics.
//   warps 8-15  converters: float pairs -> 5 digit planes of 128 x 64 (128-byte swizzle).
//   warp 16     vector digits by TMA, the tiles ahead into L2.
//   warp 17     MMAs.
#include <cuda_fp16.h>

#include <algorithm>

#include "common.h"
#include "gemm_tc.cuh"
#include "vec_digits.cuh"

namespace wfq {
namespace {

using tc::Params;

constexpr int SV_M = 128, SV_K = 64;                 // rows and columns of a stage
constexpr int SV_ND = 5;                             // digits of D (a vector has 8)
constexpr int SV_ROWS = 32;                          // rows of the vector digit planes: m * C + v
constexpr uint32_t SV_PLANE = SV_M * SV_K * 2;       // one digit plane of a stage
constexpr uint32_t SV_A = SV_ND * SV_PLANE;
constexpr uint32_t SV_B = SV_ROWS * SV_K * 2;        // vector digits of 64 atoms
constexpr int SV_STAGES = 2;
constexpr int SV_AHEAD = 3;                           // units the pairs are prefetched ahead
constexpr int SV_CONV = 8;                           // converter warps (16 measured 412 against 390 us)
constexpr int SV_Q = 64 / (2 * SV_CONV);             // rows a converter lane has in a register set
constexpr int SV_TMA_WARP = 8 + SV_CONV;
constexpr int SV_THREADS = 32 * (SV_TMA_WARP + 4);
// digits m of the vector that digit plane k of D meets: 11 k + 7 m <= 56
__host__ __device__ constexpr int sv_terms(int k) { return k == 0 ? 8 : k == 1 ? 7 : k == 2 ? 5 : k == 3 ? 4 : 2; }
__host__ __device__ constexpr int sv_n(int k, int C) { return (sv_terms(k) * C + 15) / 16 * 16; }
// first tensor-memory column of plane k in a slot (of 128)
__host__ __device__ constexpr int sv_col(int k, int C) {
    return (k > 0 ? sv_n(0, C) : 0) + (k > 1 ? sv_n(1, C) : 0) + (k > 2 ? sv_n(2, C) : 0) + (k > 3 ? sv_n(3, C) : 0);
}

struct SymvParams {
    Params p;
    int T;                  // 64-column blocks
    int64_t units;
    const float *Dsym;      // symmetric tiles, or
    const float *Fh, *Fl;   // full planes of ld columns, zero past column n
    int64_t ld;
    int E;                  // |D_ij| < 2^E
    unsigned long long *acc;   // [C][n][2]: units 2^-28 and 2^-56
    VecSums sums;
};

// descriptor of a tile of 128-byte rows with the 128-byte swizzle: 8-row groups 1024 bytes apart
// (K-major: M or N rows; MN-major: K rows, one 64-element block along M)
__device__ __forceinline__ uint64_t desc_sw128(uint32_t saddr) {
    uint64_t d = 0;
    d |= static_cast<uint64_t>((saddr & 0x3FFFFu) >> 4);
    d |= static_cast<uint64_t>(1u) << 16;
    d |= static_cast<uint64_t>(1024u >> 4) << 32;
    d |= static_cast<uint64_t>(1u) << 46;
    d |= static_cast<uint64_t>(2u) << 61;
    return d;
}

// fp16 operands, FP32 accumulator; a_mn: A is MN-major
__device__ __forceinline__ uint32_t idesc_f16(int m, int n, bool a_mn) {
    return (1u << 4) | (a_mn ? 1u << 15 : 0u) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float *v) {
    uint32_t r[8];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr));
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
}

// hi[v] += terms of weight 2^-28 and above (units 2^-28), lo[v] += the others (units 2^-56), of
// the accumulators of one row at `base`
template <int C>
__device__ __forceinline__ void read_terms(uint32_t base, int64_t (&hi)[C], int64_t (&lo)[C]) {
#pragma unroll
    for (int k = 0; k < SV_ND; ++k) {
#pragma unroll
        for (int b = 0; b < sv_terms(k) * C; b += 8) {
            float x[8];
            tmem_ld8(base + (uint32_t)(sv_col(k, C) + b), x);
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int m = (b + q) / C, v = (b + q) % C, w = 11 * k + 7 * m;
                if (m >= sv_terms(k)) continue;
                const int s = __float2int_rn(x[q]);
                if (w <= 28)
                    hi[v] += (int64_t)s * (1 << (w <= 28 ? 28 - w : 0));
                else
                    lo[v] += (int64_t)s * (1 << (w > 28 ? 56 - w : 0));
            }
        }
    }
}

template <int C, bool TILES>
__global__ void __launch_bounds__(SV_THREADS, 1) k_gemv_digits(const __grid_constant__ CUtensorMap tm_x, const SymvParams sp) {
    const bool skip = sp.sums.plain(C);   // read while the block sets up
    const Params &p = sp.p;
    extern __shared__ unsigned char smem_raw[];
    unsigned char *smem =
        reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    constexpr uint32_t SLOT = 128;   // tensor-memory columns of a slot
    constexpr uint32_t BJ_OFF = SV_STAGES * SV_A, BI_OFF = BJ_OFF + SV_STAGES * SV_B;
    uint64_t *a_full = reinterpret_cast<uint64_t *>(smem + BI_OFF + 2 * 2 * SV_B);
    uint64_t *a_empty = a_full + SV_STAGES;
    uint64_t *bj_full = a_empty + SV_STAGES;
    uint64_t *bi_full = bj_full + SV_STAGES;
    uint64_t *bi_empty = bi_full + 2;
    uint64_t *row_full = bi_empty + 2;   // tensor-memory slots: two for rows, two for columns
    uint64_t *row_empty = row_full + 2;
    uint64_t *col_full = row_empty + 2;
    uint64_t *col_empty = col_full + 2;
    uint64_t *drain = col_empty + 2;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(drain + 1);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);

    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    const int64_t u_begin = sp.units * (int64_t)blockIdx.x / gridDim.x;
    const int64_t u_end = sp.units * ((int64_t)blockIdx.x + 1) / gridDim.x;
    const int nunits = (int)(u_end - u_begin);

    if (threadIdx.x == 0) {
        for (int s = 0; s < SV_STAGES; ++s) {
            tc::mbar_init(tc::smem_u32(a_full + s), SV_CONV);
            tc::mbar_init(tc::smem_u32(a_empty + s), 1);
            tc::mbar_init(tc::smem_u32(bj_full + s), 1);
        }
        for (int s = 0; s < 2; ++s) {
            tc::mbar_init(tc::smem_u32(bi_full + s), 1);
            tc::mbar_init(tc::smem_u32(bi_empty + s), 1);
            tc::mbar_init(tc::smem_u32(col_full + s), 1);
            tc::mbar_init(tc::smem_u32(col_empty + s), 4);
            tc::mbar_init(tc::smem_u32(row_full + s), 1);
            tc::mbar_init(tc::smem_u32(row_empty + s), 4);
        }
        tc::mbar_init(tc::smem_u32(drain), 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == SV_TMA_WARP) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc::smem_u32(tmem_slot)),
                     "r"(512)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    if (skip) {
        if (warp == SV_TMA_WARP)
            asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
        return;
    }
    const uint32_t smem_base = tc::smem_u32(smem);

    // position of a unit: row block a, column block J from 2 a, advanced in order
    struct Cursor {
        int a, J;
    };
    Cursor cur;
    {
        // units before block a: a T - a (a - 1)
        int lo = 0, hi = (sp.T + 1) / 2;
        while (hi - lo > 1) {
            const int mid = (lo + hi) / 2;
            if ((int64_t)mid * sp.T - (int64_t)mid * (mid - 1) <= u_begin) lo = mid;
            else hi = mid;
        }
        cur.a = lo;
        cur.J = 2 * lo + (int)(u_begin - ((int64_t)lo * sp.T - (int64_t)lo * (lo - 1)));
    }
    auto advance = [&] {
        if (++cur.J == sp.T) {
            ++cur.a;
            cur.J = 2 * cur.a;
        }
    };
    // K steps of 16 rows of the transposed product
    auto col_steps = [&] { return cur.J == 2 * cur.a ? 0 : cur.J == 2 * cur.a + 1 ? 4 : 8; };
    auto block_end = [&](int u) { return cur.J == sp.T - 1 || u + 1 == nunits; };
    // the rows' accumulators are read every 128 columns at the latest
    auto row_read = [&](int u) { return (cur.J & 1) || block_end(u); };

    if (warp < 4) {
        // ---------------------------------------------------------- row epilogue
        int64_t hi[C], lo[C];
#pragma unroll
        for (int v = 0; v < C; ++v) hi[v] = lo[v] = 0;
        const uint32_t base = tmem + ((uint32_t)(warp * 32) << 16);
        uint32_t uses = 0;
        for (int u = 0; u < nunits; ++u, advance()) {
            if (!row_read(u)) continue;
            const uint32_t slot = uses & 1u;
            if (!tc::mbar_wait_warp(tc::smem_u32(row_full + slot), (uses >> 1) & 1u, p, 4, abort_flag)) break;
            ++uses;
            tc::tc_fence_after();
            read_terms<C>(base + slot * SLOT, hi, lo);
            tc::tc_fence_before();
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(tc::smem_u32(row_empty + slot));
            if (block_end(u)) {
                const int64_t i = (int64_t)cur.a * SV_M + warp * 32 + lane;
#pragma unroll
                for (int v = 0; v < C; ++v) {
                    if (i < p.n) {
                        unsigned long long *a = sp.acc + 2 * ((int64_t)v * p.n + i);
                        atomicAdd(a, (unsigned long long)hi[v]);
                        atomicAdd(a + 1, (unsigned long long)lo[v]);
                    }
                    hi[v] = lo[v] = 0;
                }
            }
        }
    } else if (warp < 8) {
        // ---------------------------------------------------------- column epilogue
        // M = 64: rows 16 q .. 16 q + 15 of the product in lanes 0-15 of quadrant q
        const int quad = warp & 3;
        uint32_t uses = 0;
        for (int u = 0; u < nunits; ++u, advance()) {
            if (col_steps() == 0) continue;
            const uint32_t slot = uses & 1u;
            if (!tc::mbar_wait_warp(tc::smem_u32(col_full + slot), (uses >> 1) & 1u, p, 4, abort_flag)) break;
            ++uses;
            tc::tc_fence_after();
            int64_t hi[C], lo[C];
#pragma unroll
            for (int v = 0; v < C; ++v) hi[v] = lo[v] = 0;
            read_terms<C>(tmem + (2 + slot) * SLOT + ((uint32_t)(quad * 32) << 16), hi, lo);
            tc::tc_fence_before();
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(tc::smem_u32(col_empty + slot));
            const int64_t j = (int64_t)cur.J * SV_K + quad * 16 + lane;
            if (lane < 16 && j < p.n) {
#pragma unroll
                for (int v = 0; v < C; ++v) {
                    unsigned long long *a = sp.acc + 2 * ((int64_t)v * p.n + j);
                    atomicAdd(a, (unsigned long long)hi[v]);
                    atomicAdd(a + 1, (unsigned long long)lo[v]);
                }
            }
        }
    } else if (warp < SV_TMA_WARP) {
        // ---------------------------------------------------------- converters
        // A lane takes 4 consecutive columns of a row, 16 lanes a row's 64, a warp 2 rows at a
        // time; a register set is half a stage (64 rows), the other half's set and the next
        // stage's are on their way while one is converted.
        const int cw = warp - 8;
        const int lr = cw * 2 + (lane >> 4), lk = (lane & 15) * 4;
        struct Regs {
            float4 h[SV_Q], l[SV_Q];
        };
        int half = 0;   // next load: half of the cursor's stage
        auto load = [&](Regs &f) {
            const bool zero = cur.J == 2 * cur.a && half == 1;
            if (zero) {
#pragma unroll
                for (int q = 0; q < SV_Q; ++q) f.h[q] = f.l[q] = make_float4(0.f, 0.f, 0.f, 0.f);
            } else if constexpr (TILES) {
                const int I = 2 * cur.a + half;
                const float *t = sp.Dsym + sym_tile(I, cur.J, sp.T) * 2 * kSymTile * kSymTile;
#pragma unroll
                for (int q = 0; q < SV_Q; ++q) {
                    f.h[q] = f.l[q] = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (I < sp.T) {
                        f.h[q] = __ldcs(reinterpret_cast<const float4 *>(t + (q * 2 * SV_CONV + lr) * kSymTile + lk));
                        f.l[q] = __ldcs(reinterpret_cast<const float4 *>(t + kSymTile * kSymTile + (q * 2 * SV_CONV + lr) * kSymTile + lk));
                    }
                }
            } else {
#pragma unroll
                for (int q = 0; q < SV_Q; ++q) {
                    // rows past n meet zero digits of the vectors, and are not stored
                    const int64_t i = min((int64_t)cur.a * SV_M + half * 64 + q * 2 * SV_CONV + lr, p.n - 1);
                    f.h[q] = __ldcs(reinterpret_cast<const float4 *>(sp.Fh + i * sp.ld + (int64_t)cur.J * SV_K + lk));
                    f.l[q] = __ldcs(reinterpret_cast<const float4 *>(sp.Fl + i * sp.ld + (int64_t)cur.J * SV_K + lk));
                }
            }
            half ^= 1;
            if (half == 0) advance();
        };
        auto convert = [&](const Regs &f, uint32_t base, int hf) {
            const float2 magic = make_float2(12582912.f, 12582912.f), nmagic = make_float2(-12582912.f, -12582912.f);
            const float2 s11 = make_float2(2048.f, 2048.f);
#pragma unroll
            for (int q = 0; q < SV_Q; ++q) {
                const float sh1 = __int_as_float((127 + 10 - sp.E) << 23), sl1 = __int_as_float((127 + 32 - sp.E) << 23);
                const float2 sh = make_float2(sh1, sh1), sl = make_float2(sl1, sl1);
                uint32_t dig[SV_ND][2];
#pragma unroll
                for (int b = 0; b < 2; ++b) {
                    const float2 h = b ? make_float2(f.h[q].z, f.h[q].w) : make_float2(f.h[q].x, f.h[q].y);
                    const float2 l = b ? make_float2(f.l[q].z, f.l[q].w) : make_float2(f.l[q].x, f.l[q].y);
                    auto put = [&](int k, float2 d) {
                        const __half2 hd = __floats2half2_rn(d.x, d.y);
                        dig[k][b] = *reinterpret_cast<const uint32_t *>(&hd);
                    };
                    auto neg = [](float2 a) { return make_float2(-a.x, -a.y); };
                    // every remainder is exact: it is representable, and fma rounds once
                    const float2 v = __fmul2_rn(h, sh);
                    const float2 d0 = __fadd2_rn(__fadd2_rn(v, magic), nmagic);
                    float2 r = __fadd2_rn(v, neg(d0));
                    put(0, d0);
                    const float2 d1 = __fadd2_rn(__ffma2_rn(r, s11, magic), nmagic);
                    r = __ffma2_rn(r, s11, neg(d1));
                    put(1, d1);
                    // the third digit: what is left of h, and l from here on
                    const float2 dh = __fadd2_rn(__ffma2_rn(r, s11, magic), nmagic);
                    r = __ffma2_rn(r, s11, neg(dh));
                    const float2 dl = __fadd2_rn(__ffma2_rn(l, sl, magic), nmagic);
                    put(2, __fadd2_rn(dh, dl));
                    r = __fadd2_rn(r, __ffma2_rn(l, sl, neg(dl)));   // rounded at 2^-57 of the bound
                    const float2 d3 = __fadd2_rn(__ffma2_rn(r, s11, magic), nmagic);
                    r = __ffma2_rn(r, s11, neg(d3));
                    put(3, d3);
                    put(4, __fadd2_rn(__ffma2_rn(r, s11, magic), nmagic));
                }
                const int row = hf * 64 + q * 2 * SV_CONV + lr;
                // 128-byte swizzle: 16-byte chunk index XOR row mod 8
                const uint32_t off =
                    base + (uint32_t)row * 128u + (uint32_t)(((lk >> 3) ^ (row & 7)) * 16) + (uint32_t)(lk & 4) * 2;
#pragma unroll
                for (int k = 0; k < SV_ND; ++k)
                    asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(off + (uint32_t)k * SV_PLANE), "r"(dig[k][0]),
                                 "r"(dig[k][1])
                                 : "memory");
            }
        };
        Regs r0, r1;
        load(r0);
        load(r1);
#pragma unroll 1
        for (int u = 0; u < nunits; ++u) {
            const uint32_t s = u & 1, ph = (u >> 1) & 1;
            const uint32_t base = smem_base + s * SV_A;
            if (!tc::mbar_wait_warp(tc::smem_u32(a_empty + s), ph ^ 1u, p, 1, abort_flag)) break;
            convert(r0, base, 0);
            if (u + 1 < nunits) load(r0);
            convert(r1, base, 1);
            if (u + 1 < nunits) load(r1);
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(tc::smem_u32(a_full + s));
        }
    } else {
        if (warp == SV_TMA_WARP) {
        // ---------------------------------------------------------- TMA producer (vector digits)
        // and, all lanes, the tiles SV_AHEAD units on into L2 (not the planes: a bulk prefetch per
        // 256-byte row segment measured twice as slow as none).
        Cursor ahead = cur;
        int ahead_u = 0;
        auto prefetch = [&] {   // unit `ahead`; advances it
            if (ahead_u < nunits) {
                if constexpr (TILES) {
                    // 4 KiB of a 16 KiB plane a lane: (tile row, plane, quarter)
                    const int I = 2 * ahead.a + (lane >> 3);
                    if (lane < 16 && I < sp.T && !(ahead.J == 2 * ahead.a && lane >= 8)) {
                        const float *t = sp.Dsym + sym_tile(I, ahead.J, sp.T) * 2 * kSymTile * kSymTile + (lane & 7) * 1024;
                        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(t), "r"(4096u) : "memory");
                    }
                }
            }
            ++ahead_u;
            if (++ahead.J == sp.T) {
                ++ahead.a;
                ahead.J = 2 * ahead.a;
            }
        };
        for (int k = 0; k < SV_AHEAD; ++k) prefetch();
        uint32_t blocks = 0;
        int u = 0;
        bool aborted = false;
        for (; u < nunits; ++u, advance()) {
            const uint32_t s = u & 1, ph = (u >> 1) & 1;
            prefetch();
            if (u == 0 || cur.J == 2 * cur.a) {   // a block's own rows, for the transposed products
                const uint32_t bs = blocks & 1;
                if (!tc::mbar_wait_warp(tc::smem_u32(bi_empty + bs), ((blocks >> 1) & 1) ^ 1u, p, 1, abort_flag)) {
                    aborted = true;
                    break;
                }
                if (lane == 0) {
                    tc::mbar_expect_tx(tc::smem_u32(bi_full + bs), 2 * SV_B);
                    for (int h = 0; h < 2; ++h)
                        tc::tma_load_2d(smem_base + BI_OFF + (2 * bs + h) * SV_B, &tm_x, tc::smem_u32(bi_full + bs),
                                        cur.a * SV_M + h * SV_K, 0);
                }
                ++blocks;
            }
            if (!tc::mbar_wait_warp(tc::smem_u32(a_empty + s), ph ^ 1u, p, 1, abort_flag)) {
                aborted = true;
                break;
            }
            if (lane == 0) {
                tc::mbar_expect_tx(tc::smem_u32(bj_full + s), SV_B);
                tc::tma_load_2d(smem_base + BJ_OFF + s * SV_B, &tm_x, tc::smem_u32(bj_full + s), cur.J * SV_K, 0);
            }
            __syncwarp();
        }
        if (aborted && lane == 0) {   // wait (bounded) for the copies issued
            volatile int no_abort = 0;
            for (int j = u > 2 ? u - 2 : 0; j < u; ++j)
                tc::mbar_wait(tc::smem_u32(bj_full + (j & 1)), (j >> 1) & 1, p, 1, &no_abort);
            for (uint32_t j = blocks > 2 ? blocks - 2 : 0; j < blocks; ++j)
                tc::mbar_wait(tc::smem_u32(bi_full + (j & 1)), (j >> 1) & 1, p, 1, &no_abort);
        }
        } else if (warp == SV_TMA_WARP + 1) {
        const bool el = tc::elect_one();
        // ---------------------------------------------------------- MMA issuer
        uint32_t blocks = 0, cuses = 0, ruses = 0;
        bool aborted = false, fresh = true;
        for (int u = 0; u < nunits && !aborted; ++u, advance()) {
            const uint32_t s = u & 1, ph = (u >> 1) & 1;
            if (u == 0 || cur.J == 2 * cur.a) {
                aborted = !tc::mbar_wait(tc::smem_u32(bi_full + (blocks & 1)), (blocks >> 1) & 1, p, 2, abort_flag);
                ++blocks;
            }
            aborted = aborted || !tc::mbar_wait(tc::smem_u32(a_full + s), ph, p, 2, abort_flag) ||
                      !tc::mbar_wait(tc::smem_u32(bj_full + s), ph, p, 2, abort_flag);
            if (aborted) break;
            tc::tc_fence_after();
            const uint64_t da = desc_sw128(smem_base + s * SV_A);
            // Small products wait on their accumulator's previous one, so the row and the column
            // products, which share none, are issued in turn.
            const int steps = col_steps();
            const uint32_t slot = cuses & 1u;
            if (steps > 0) {
                aborted = !tc::mbar_wait(tc::smem_u32(col_empty + slot), ((cuses >> 1) & 1u) ^ 1u, p, 3, abort_flag);
                ++cuses;
            }
            if (fresh) aborted = aborted || !tc::mbar_wait(tc::smem_u32(row_empty + (ruses & 1u)), ((ruses >> 1) & 1u) ^ 1u, p, 3, abort_flag);
            if (aborted) break;
            tc::tc_fence_after();
            const uint64_t dbi = desc_sw128(smem_base + BI_OFF + 2 * ((blocks - 1) & 1) * SV_B);
            const uint64_t dbj = desc_sw128(smem_base + BJ_OFF + s * SV_B);
            const uint32_t drow = tmem + (ruses & 1u) * SLOT, dcol = tmem + (2 + slot) * SLOT;
#pragma unroll 1
            for (int ks = 0; ks < SV_K / 16; ++ks) {
#pragma unroll
                for (int k = 0; k < SV_ND; ++k)
                    if (el) tc::umma_bf16(drow + (uint32_t)sv_col(k, C), da + (uint64_t)((k * SV_PLANE + ks * 32u) >> 4),
                                  dbj + (uint64_t)(ks * 2), idesc_f16(SV_M, sv_n(k, C), false), fresh && ks == 0 ? 0u : 1u);
                for (int kc = ks; kc < steps; kc += 4) {
#pragma unroll
                    for (int k = 0; k < SV_ND; ++k)
                        if (el)
                            tc::umma_bf16(dcol + (uint32_t)sv_col(k, C), da + (uint64_t)((k * SV_PLANE + kc * 2048u) >> 4),
                                          dbi + (uint64_t)(((kc >> 2) * SV_B + (kc & 3) * 32u) >> 4),
                                          idesc_f16(64, sv_n(k, C), true), kc > 0 ? 1u : 0u);
                }
            }
            if (steps > 0 && el) tc::umma_commit(tc::smem_u32(col_full + slot));
            fresh = row_read(u);
            if (fresh) {
                if (el) tc::umma_commit(tc::smem_u32(row_full + (ruses & 1u)));
                ++ruses;
            }
            if (el) tc::umma_commit(tc::smem_u32(a_empty + s));
            if (block_end(u) && el) tc::umma_commit(tc::smem_u32(bi_empty + ((blocks - 1) & 1)));
        }
        if (el) tc::umma_commit(tc::smem_u32(drain));
        volatile int no_abort = 0;
        tc::mbar_wait(tc::smem_u32(drain), 0u, p, 5, &no_abort);
        }
    }
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    if (warp == SV_TMA_WARP) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
    }
}

// Largest |x| of each of C vectors (element i of vector c at i si + c sc) as a bit pattern.
__global__ void __launch_bounds__(256) k_vec_absmax(int64_t n, int64_t si, int64_t sc, const double *__restrict__ X,
                                                    unsigned long long *__restrict__ vmax) {
    __shared__ unsigned long long sm[8];
    const int c = blockIdx.y;
    unsigned long long m = 0;
    for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < n; i += (int64_t)gridDim.x * 256) {
        const unsigned long long b = (unsigned long long)__double_as_longlong(X[i * si + c * sc]) & 0x7fffffffffffffffull;
        m = b > m ? b : m;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long q = __shfl_xor_sync(0xffffffffu, m, o);
        m = q > m ? q : m;
    }
    if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int q = 1; q < 8; ++q) m = sm[q] > m ? sm[q] : m;
        atomicMax(vmax + c, m);
    }
}

__global__ void __launch_bounds__(256) k_vec_digits(int64_t n, int64_t npad, int C, int64_t si, int64_t sc,
                                                    const double *__restrict__ X, const unsigned long long *__restrict__ vmax,
                                                    __half *__restrict__ planes, int *__restrict__ xexp,
                                                    unsigned *__restrict__ vsum, float *__restrict__ xh,
                                                    float *__restrict__ xl) {
    const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
    const int c = blockIdx.y, cg = min(4, C - (c & ~3));
    const unsigned long long mb = vmax[c];
    const int e = vec_exp(mb);
    __half *dst = planes + (int64_t)(c >> 2) * SV_ROWS * npad + (int64_t)(c & 3) * npad + i;
    unsigned q = 0;
    if (i < n) {
        const double x = X[i * si + c * sc];
        q = put_vec_digits(x, e, dst, (int64_t)cg * npad);
        if (xh) df_split(x, xh[c * n + i], xl[c * n + i]);
    }
    q = __reduce_add_sync(0xffffffffu, q);
    if ((threadIdx.x & 31) == 0 && q > 0) atomicAdd(vsum + c, q);
    if (i == 0) {
        xexp[c] = e;
        if (mb == 0ull || e == kVecNotFinite) vsum[c] = 0xffffffffu;   // nothing is added for these
    }
}

// U[i si + c sc] = 2^(E + e_c - 43) (acc0 + acc1 2^-28), and the sums are cleared for the next
// product; a group left to double-float sums takes theirs.
__global__ void __launch_bounds__(256) k_gemv_digits_finish(int64_t n, int C, int64_t si, int64_t sc,
                                                            unsigned long long *__restrict__ acc, int E,
                                                            const int *__restrict__ xexp, const VecSums sums,
                                                            const SymPartials sym, const double *ud, double *U) {
    wait_for_previous();
    const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
    const int c = blockIdx.y;
    if (i >= n) return;
    if (sums.plain(C)) {
        if (sym.rowpart) U[i * si + c * sc] = dsymv_sum(sym, C, i, c);
        else if (ud) U[i * si + c * sc] = ud[c * n + i];
        return;
    }
    ulonglong2 *a = reinterpret_cast<ulonglong2 *>(acc) + (int64_t)c * n + i;
    const ulonglong2 s = *a;
    *a = make_ulonglong2(0ull, 0ull);
    const int e = xexp[c];
    const double v = fma((double)(long long)s.y, 0x1p-28, (double)(long long)s.x);
    U[i * si + c * sc] = e == kVecNotFinite ? __longlong_as_double(0x7ff8000000000000ll)
                                            : scalbn(v, E + e - 43);
}

bool make_x_map(CUtensorMap *m, const __half *planes, uint64_t npad, std::string *msg) {
    tc::EncodeTiledFn fn = tc::encode_fn(msg);
    if (!fn) return false;
    cuuint64_t dims[2] = {npad, (cuuint64_t)SV_ROWS};
    cuuint64_t strides[1] = {npad * 2};
    cuuint32_t box[2] = {(cuuint32_t)SV_K, (cuuint32_t)SV_ROWS};
    cuuint32_t estr[2] = {1, 1};
    const CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, const_cast<__half *>(planes), dims, strides, box, estr,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS && msg) *msg = "cuTensorMapEncodeTiled failed with code " + std::to_string((int)r);
    return r == CUDA_SUCCESS;
}

template <int C, bool TILES>
cudaError_t launch_ct(const CUtensorMap &m, const SymvParams &sp, int grid, cudaStream_t s) {
    constexpr size_t smem = SV_STAGES * (size_t)(SV_A + SV_B) + 4 * SV_B + 1024 + 512;
    static_assert(smem <= (size_t)tc::kMaxDynSmem, "digit stages exceed shared memory");
    static std::atomic<uint64_t> smem_set{0};
    cudaError_t e = tc::allow_max_smem(k_gemv_digits<C, TILES>, smem_set);
    if (e != cudaSuccess) return e;
    k_gemv_digits<C, TILES><<<(unsigned)grid, SV_THREADS, smem, s>>>(m, sp);
    return cudaGetLastError();
}

template <int C>
cudaError_t launch_c(const CUtensorMap &m, const SymvParams &sp, int grid, cudaStream_t s) {
    return sp.Fh ? launch_ct<C, false>(m, sp, grid, s) : launch_ct<C, true>(m, sp, grid, s);
}

}  // namespace

// Needs a symmetric D (not the BEM operator: with every column block and no transposed products it
// gained 10% there, but its Krylov spaces amplify the rounding of either product past 1e-9 of q).  All
// rows share one exponent (a column's sum runs over the rows), so the rows' bounds must not differ
// by more than 2^3: a row then loses at most 3 of its 55 bits.
bool gemv_digits_usable(const wfq_geom *g) {
    return g->digits_ok && (g->Dfh || g->Dsym) && g->dexp_max - g->dexp_min <= 3;
}

size_t gemv_digits_plane_elems(const wfq_geom *g) { return (size_t)SV_ROWS * g->npad; }

// What is left out per entry, in 2^(E + e): the terms with 11 k + 7 m > 56 (2^-55 at most), the last
// digits of D and of the vector (2^-55 each) and the rounding of D's fourth remainder (2^-57): below 2^-53,
// against 2^-48 |D_ij v_j| of double-float sums.
unsigned gemv_digits_threshold(const wfq_geom *g) { return digit_sum_threshold(g, -53 + 48); }

int gemv_digits_split(const wfq_geom *g, int C, const double *X, int64_t si, int64_t sc, const GemvDigits &w, float *xh,
                      float *xl, cudaStream_t s) {
    WFQ_CUDA(cudaMemsetAsync(w.vmax, 0, (sizeof(unsigned long long) + sizeof(unsigned)) * C, s));
    const unsigned nb = (unsigned)std::min<int64_t>((g->n + 255) / 256, 64);
    k_vec_absmax<<<dim3(nb, (unsigned)C), 256, 0, s>>>(g->n, si, sc, X, w.vmax);
    note_launch();
    k_vec_digits<<<dim3((unsigned)((g->n + 255) / 256), (unsigned)C), 256, 0, s>>>(
        g->n, g->npad, C, si, sc, X, w.vmax, reinterpret_cast<__half *>(w.planes), w.xexp, w.vsum, xh, xl);
    note_launch();
    WFQ_CUDA(cudaGetLastError());
    return WFQ_OK;
}

int gemv_digits_product(const wfq_geom *g, int C, const GemvDigits &w, cudaStream_t s, int *err) {
    const int64_t n = g->n;
    SymvParams sp{};
    sp.p.n = n;
    sp.p.err = err ? err : g->ctx->dev_err;
    sp.p.timeout_ns = 4000000000ull;
    sp.T = (int)((n + SV_K - 1) / SV_K);
    const int64_t A = (sp.T + 1) / 2;
    sp.units = A * sp.T - A * (A - 1);
    sp.Dsym = g->Dsym;
    sp.Fh = g->Dfh;
    sp.Fl = g->Dfl;
    sp.ld = g->ldf;
    sp.E = g->dexp_max;
    sp.acc = w.acc;
    sp.sums = w.sums();
    std::string msg;
    CUtensorMap m;
    if (!make_x_map(&m, reinterpret_cast<const __half *>(w.planes), (uint64_t)g->npad, &msg)) return fail(WFQ_ECUDA, "digit-slice GEMV: " + msg);
    const int grid = (int)std::min<int64_t>(g->ctx->num_sms, sp.units);
    cudaError_t e = C == 1 ? launch_c<1>(m, sp, grid, s) : C == 2 ? launch_c<2>(m, sp, grid, s)
                    : C == 3 ? launch_c<3>(m, sp, grid, s) : launch_c<4>(m, sp, grid, s);
    note_launch();
    if (e != cudaSuccess) {
        cudaGetLastError();
        return fail(WFQ_ECUDA, std::string("digit-slice GEMV: ") + cudaGetErrorString(e));
    }
    return WFQ_OK;
}

int gemv_digits_finish(const wfq_geom *g, int C, const GemvDigits &w, const SymPartials &sym, const double *ud, double *U,
                       int64_t si, int64_t sc, cudaStream_t s) {
    WFQ_CUDA(launch_overlapped(k_gemv_digits_finish, dim3((unsigned)((g->n + 255) / 256), (unsigned)C), dim3(256), 0, s, g->n, C,
                               si, sc, w.acc, g->dexp_max, w.xexp, w.sums(), sym, ud, U));
    note_launch();
    WFQ_CUDA(cudaGetLastError());
    return WFQ_OK;
}

}  // namespace wfq
