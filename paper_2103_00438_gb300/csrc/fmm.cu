// Far-field-compressed D product: a fast multipole method for U = D X at large N.
//
// The paper's conclusions name the O(N^2) matrix-vector product as the first bottleneck
// of the method and the fast multipole method as the way past it; the paper gives no FMM
// of its own.  This is the Chebyshev-interpolation ("black-box") FMM of Fong and Darve
// (J. Comput. Phys. 228, 2009), written from its published description:
//
//   * a uniform tree over the bounding cube (a quadtree over the bounding square when all
//     atoms share one z, as for a flat graphene disk), as deep as leaves of side
//     h >= r_far = 6 max_ij s_ij allow (s_ij = sqrt(w_i^2 + w_j^2), widths from Eq. 4):
//     erf(r / s_ij) is 1 in FP64 beyond r_far, so every pair the far field handles has
//     D_ij = 1 / r_ij exactly (Eq. 3);
//   * near field: pairs in the same or adjacent leaves, Eq. 3 directly (D_ii = eta_i);
//   * far field: 1 / |t - s| interpolated at p Chebyshev nodes per dimension in target and
//     source boxes: P2M (atoms to their leaf's nodes), M2M (child to parent nodes), M2L
//     (1 / |t - s| between the nodes of the boxes of each interaction list), L2L (parent to
//     child nodes), L2P (leaf nodes to atoms), with the weights
//         S_p(x_m, y) = 1/p + (2/p) sum_{k=1}^{p-1} T_k(x_m) T_k(y);
//   * interaction list of a box at level l >= 2: boxes of level l whose parents are
//     adjacent to (or are) its parent and which are not adjacent to it.
//
// The tree is built on the host in FP64 with the same arithmetic as the oracle's, so both
// put every atom in the same leaf.  The passes run in FP32 on the device (the far field's
// truncation error at p = 6 is ~1e-6 of sum_j |D_ij x_j|, the same order as the 3xBF16
// products of the mixed precision): one launch for P2M, one per level for M2M and L2L,
// one for every M2L of all levels, one for L2P with the near field.  Coordinates reach the
// kernels relative to their leaf's centre, so the near-field differences keep FP32
// precision at any distance from the origin.
#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <memory>
#include <numeric>
#include <unordered_map>
#include <vector>

#include "common.h"

namespace wfq {

struct Fmm {
    int dim = 3, p = 0, P = 0, L = 0;
    double side = 0.0, h = 0.0, r_far = 0.0;
    std::vector<int64_t> lvl0;       // first global box index of each level, L + 2 entries
    int64_t nbox = 0, nleaf = 0, nil = 0, nnear = 0;
    // device arrays
    int32_t *perm = nullptr;         // n: original index of the atom at sorted position k
    int32_t *leaf_start = nullptr;   // nleaf + 1: sorted atom range of each leaf
    float4 *atl = nullptr;           // n (sorted): position relative to the leaf centre, width
    float *eta = nullptr;            // n (sorted): eta_i (the diagonal of D)
    int32_t *parent = nullptr;       // nbox: parent's global index (-1 at level 0)
    int32_t *child_lo = nullptr;     // nbox: children's global index range [lo, hi)
    int32_t *child_hi = nullptr;
    int8_t *octant = nullptr;        // nbox: which child of its parent (bit d: upper half in d)
    // M2L: the boxes of levels >= 2 by octant (boxes of one octant have the same offsets in the
    // same order, the slots) and each slot's source box
    int nslots = 0;                  // 27 (quadtree) or 189 (octree)
    int64_t nm2l = 0;
    int32_t oct_first[9] = {};       // first list position of each octant
    int32_t *m2l_box = nullptr;      // nm2l: global box index
    int8_t *m2l_level = nullptr;     // nm2l
    int32_t *m2l_src = nullptr;      // nslots x nm2l: source box, -1: none
    int16_t *slot_off = nullptr;     // 2^dim x nslots: offset code, sum_d (src_d - tgt_d + 3) 7^d
    int32_t *near_start = nullptr;   // nleaf + 1: near leaves of each leaf (CSR)
    int32_t *near_leaf = nullptr;    // nnear: leaf index
    int8_t *near_delta = nullptr;    // nnear: offset code, sum_d (src_d - tgt_d + 1) 3^d
    int64_t ngroups = 0;             // targets of the near field: up to 32 atoms of one leaf
    int32_t *tgt_leaf = nullptr;     // ngroups: leaf index
    int32_t *tgt_first = nullptr;    // ngroups: first atom
    float *Tm = nullptr;             // 2^dim x P x Pp: M2M weights [octant][child node][parent node]
    float *Tl = nullptr;             // 2^dim x P x Pp: the same [octant][parent node][child node], for L2L
    float *K = nullptr;              // 7^dim x P x P: M2L kernel for boxes of half-width 1
    float *cheb = nullptr;           // p x p: T_k(x_m)
    size_t bytes = 0;
};

namespace {

constexpr double kPi = 3.14159265358979323846;

inline uint64_t spread2(uint64_t v) {   // bits of v at even positions
    uint64_t r = 0;
    for (int b = 0; b < 31; ++b) r |= ((v >> b) & 1ull) << (2 * b);
    return r;
}
inline uint64_t spread3(uint64_t v) {
    uint64_t r = 0;
    for (int b = 0; b < 21; ++b) r |= ((v >> b) & 1ull) << (3 * b);
    return r;
}
inline uint64_t morton(int dim, const int64_t *c) {
    return dim == 2 ? (spread2(c[0]) << 1) | spread2(c[1])
                    : (spread3(c[0]) << 2) | (spread3(c[1]) << 1) | spread3(c[2]);
}
inline void unmorton(int dim, uint64_t k, int64_t *c) {
    for (int d = 0; d < dim; ++d) {
        c[d] = 0;
        const int sh = dim - 1 - d;
        for (int b = 0; b < (dim == 2 ? 31 : 21); ++b) c[d] |= (int64_t)((k >> (dim * b + sh)) & 1ull) << b;
    }
}

// S_p(x_m, y) for the p Chebyshev nodes x_m of [-1, 1].
void cheb_weights(int p, double y, double *S) {
    for (int m = 0; m < p; ++m) {
        const double th = (2.0 * m + 1.0) * kPi / (2.0 * p);
        double s = 1.0 / p;
        for (int k = 1; k < p; ++k) s += 2.0 / p * std::cos(k * th) * std::cos(k * std::acos(std::max(-1.0, std::min(1.0, y))));
        S[m] = s;
    }
}

template <class T>
int upload(wfq_ctx *ctx, Fmm *f, T **dst, const std::vector<T> &src) {
    const size_t bytes = std::max<size_t>(src.size(), 1) * sizeof(T);
    cudaError_t e = cudaMalloc(reinterpret_cast<void **>(dst), bytes);
    if (e != cudaSuccess) {
        cudaGetLastError();
        *dst = nullptr;
        return fail(WFQ_ENOMEM, "FMM allocation of " + std::to_string(bytes) + " bytes failed");
    }
    f->bytes += bytes;
    if (!src.empty()) WFQ_CUDA(cudaMemcpy(*dst, src.data(), src.size() * sizeof(T), cudaMemcpyHostToDevice));
    (void)ctx;
    return WFQ_OK;
}

// ------------------------------------------------------------------ kernels

struct FmmDev {
    int dim, p, P, L;
    float h;                          // leaf side
    int nslots;
    const int32_t *perm, *leaf_start, *parent, *child_lo, *child_hi, *m2l_box, *m2l_src;
    const int32_t *near_start, *near_leaf, *tgt_leaf, *tgt_first;
    const int16_t *slot_off;
    const int8_t *octant, *near_delta, *m2l_level;
    const float4 *atl;
    const float *eta, *Tm, *Tl, *K, *cheb;
    int64_t leaf0;                    // global index of the first leaf
};

constexpr int kMaxP = 16;   // nodes per dimension the kernels hold in registers

// Node weights of one coordinate: W[m] = S_p(x_m, y).
__device__ __forceinline__ void node_weights(const FmmDev &f, float y, float *W) {
    float tk[kMaxP];
    tk[0] = 1.f;
    if (f.p > 1) tk[1] = y;
    for (int k = 2; k < f.p; ++k) tk[k] = 2.f * y * tk[k - 1] - tk[k - 2];
    const float inv = 1.f / f.p;
    for (int m = 0; m < f.p; ++m) {
        float s = 0.f;
        for (int k = 1; k < f.p; ++k) s = fmaf(f.cheb[m * f.p + k], tk[k], s);
        W[m] = inv + 2.f * inv * s;
    }
}

// node index m -> per-dimension node indices (last dimension fastest)
__device__ __forceinline__ float node_product(const FmmDev &f, int m, const float *W0, const float *W1,
                                              const float *W2) {
    if (f.dim == 2) return W0[m / f.p] * W1[m % f.p];
    return W0[m / (f.p * f.p)] * W1[(m / f.p) % f.p] * W2[m % f.p];
}

// Rows of X in sorted order, padded with zeros to Cp columns (a multiple of 4).
__global__ void k_fmm_sort_x(int64_t n, int64_t C, int64_t Cp, const int32_t *__restrict__ perm, const float *__restrict__ X,
                             float *__restrict__ Xs) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n * Cp) return;
    const int64_t k = e / Cp, r = e - k * Cp;
    Xs[e] = r < C ? X[(int64_t)perm[k] * C + r] : 0.f;
}

// P2M: one block per leaf; multipole coefficients M[leaf][m][r] = sum_i S(m, y_i) x_i[r]
// (X in sorted order).
__global__ void k_fmm_p2m(FmmDev f, int64_t C, const float *__restrict__ X, float *__restrict__ M) {
    extern __shared__ float sm[];
    const int64_t b = blockIdx.x;
    const int k0 = f.leaf_start[b], k1 = f.leaf_start[b + 1];
    const float a = 0.5f * f.h;
    constexpr int KCH = 32;
    float *W = sm;                                   // [KCH][3][kMaxP]
    float *xs = sm + KCH * 3 * kMaxP;                // [KCH][C]
    const int64_t PC = (int64_t)f.P * C;
    float *Mb = M + (f.leaf0 + b) * PC;
    for (int64_t o = threadIdx.x; o < PC; o += blockDim.x) Mb[o] = 0.f;
    for (int c0 = k0; c0 < k1; c0 += KCH) {
        const int nk = min(KCH, k1 - c0);
        __syncthreads();
        for (int t = threadIdx.x; t < nk * f.dim; t += blockDim.x) {
            const int k = t / f.dim, d = t % f.dim;
            const float4 q = f.atl[c0 + k];
            const float y = (d == 0 ? q.x : d == 1 ? q.y : q.z) / a;
            node_weights(f, y, W + (k * 3 + d) * kMaxP);
        }
        for (int64_t t = threadIdx.x; t < (int64_t)nk * C; t += blockDim.x) {
            const int k = (int)(t / C);
            const int64_t r = t % C;
            xs[t] = X[(int64_t)(c0 + k) * C + r];
        }
        __syncthreads();
        for (int64_t o = threadIdx.x; o < PC; o += blockDim.x) {
            const int m = (int)(o / C);
            const int64_t r = o % C;
            float acc = 0.f;
            for (int k = 0; k < nk; ++k) {
                const float *Wk = W + k * 3 * kMaxP;
                acc = fmaf(node_product(f, m, Wk, Wk + kMaxP, Wk + 2 * kMaxP), xs[(int64_t)k * C + r], acc);
            }
            Mb[o] += acc;
        }
    }
}

// acc[0..7] += the rows r0 .. r0 + 7 of Tt^T In for one column: Tt is P x Pp (rows past P zero),
// In this column of a P x Cp array.  Eight rows share each load of In; Tt is uniform in a warp.
__device__ __forceinline__ void node_rows(int P, int Pp, int64_t Cp, const float *__restrict__ Tt, int r0,
                                          const float *__restrict__ In, float (&acc)[8]) {
#pragma unroll 6
    for (int k = 0; k < P; ++k) {
        const float4 a = __ldg(reinterpret_cast<const float4 *>(Tt + (int64_t)k * Pp + r0));
        const float4 b = __ldg(reinterpret_cast<const float4 *>(Tt + (int64_t)k * Pp + r0 + 4));
        const float v = In[(int64_t)k * Cp];
        acc[0] = fmaf(a.x, v, acc[0]);
        acc[1] = fmaf(a.y, v, acc[1]);
        acc[2] = fmaf(a.z, v, acc[2]);
        acc[3] = fmaf(a.w, v, acc[3]);
        acc[4] = fmaf(b.x, v, acc[4]);
        acc[5] = fmaf(b.y, v, acc[5]);
        acc[6] = fmaf(b.z, v, acc[6]);
        acc[7] = fmaf(b.w, v, acc[7]);
    }
}

// M2M at one level: a block per (parent box, 32 columns), its warps over groups of 8 nodes.
// (One output per thread with two loads per multiply-add took 418 us over the levels of the
// 250k-atom disk, order 6, 32 columns, against 255; L2L 358 against 219.)
__global__ void __launch_bounds__(256) k_fmm_m2m(FmmDev f, int Pp, int64_t C, int64_t box0, float *__restrict__ M) {
    const int64_t g = box0 + blockIdx.x;
    const int64_t r = (int64_t)blockIdx.y * 32 + (threadIdx.x & 31);
    if (r >= C) return;
    const int64_t PC = (int64_t)f.P * C;
    const int c0 = f.child_lo[g], c1 = f.child_hi[g];
    for (int r0 = (threadIdx.x >> 5) * 8; r0 < f.P; r0 += blockDim.x / 4) {
        float acc[8] = {};
        for (int ch = c0; ch < c1; ++ch)
            node_rows(f.P, Pp, C, f.Tm + (int64_t)f.octant[ch] * f.P * Pp, r0, M + (int64_t)ch * PC + r, acc);
#pragma unroll
        for (int i = 0; i < 8; ++i)
            if (r0 + i < f.P) M[g * PC + (int64_t)(r0 + i) * C + r] = acc[i];
    }
}

// L2L at one level (l >= 3): a block per (box, 32 columns); L[child] += T[oct]^T L[parent].
__global__ void __launch_bounds__(256) k_fmm_l2l(FmmDev f, int Pp, int64_t C, int64_t box0, float *__restrict__ Lc) {
    const int64_t g = box0 + blockIdx.x;
    const int64_t r = (int64_t)blockIdx.y * 32 + (threadIdx.x & 31);
    if (r >= C) return;
    const int64_t PC = (int64_t)f.P * C;
    for (int r0 = (threadIdx.x >> 5) * 8; r0 < f.P; r0 += blockDim.x / 4) {
        float acc[8] = {};
        node_rows(f.P, Pp, C, f.Tl + (int64_t)f.octant[g] * f.P * Pp, r0, Lc + (int64_t)f.parent[g] * PC + r, acc);
#pragma unroll
        for (int i = 0; i < 8; ++i)
            if (r0 + i < f.P) Lc[g * PC + (int64_t)(r0 + i) * C + r] += acc[i];
    }
}

// M2L for every box of levels 2..L.  A block takes boxes of one octant, which meet the same
// offsets slot by slot, so one kernel tile K[offset] in shared memory serves all of them; a lane
// owns one column of M2L_NB boxes and 2 RP nodes (packed FP32x2 pairs of nodes), reading its
// column of the sources' multipoles straight from L2 and K as a broadcast.  K[-offset] is the
// transpose of K[offset] (1 / |x_m - x_s - 2 d| with m and s exchanged), so its rows hold the
// target nodes of one source node consecutively.  lpb lanes per box (a power of two >= the
// columns of a block, at most 32).  blockIdx.z: group of 2 RP target nodes.
//
// Bound: FP32 FMAs (455544 tiles of 36 x 36 x 32 for the 250k-atom disk, order 6: 0.53 ms) and
// the K broadcasts (one 16-byte shared load per 8 FMAs of a lane): 1.00 ms.  A block per box with
// 4 x 4 register tiles, both operands staged, took 4.66 ms.  Unrolling the source nodes by 6
// keeps enough loads in flight (4: 1.67 ms, 12: 1.02); one box per lane 1.3 to 1.7 ms; prefetching
// the next nodes into registers 1.5 to 2.1 ms.
struct M2lGrid {
    int32_t first[9];   // octant's first list position, then the end
    int32_t tile[9];    // octant's first block
    float inv_a[24];    // 1 / half-width of the boxes of each level
};
constexpr int M2L_WARPS = 8, M2L_NB = 2;

template <int RP>
__global__ void __launch_bounds__(32 * M2L_WARPS, 2)
    k_fmm_m2l(FmmDev f, int64_t C, int64_t nm2l, int noct, M2lGrid gr, int lpb, const float *__restrict__ M,
              float *__restrict__ Lc) {
    extern __shared__ __align__(16) float sK[];   // [P][2 RP]
    constexpr int RW = 2 * RP;
    const int P = f.P, r0 = blockIdx.z * RW;
    int oc = 0;
    while (oc + 1 < noct && (int)blockIdx.x >= gr.tile[oc + 1]) ++oc;
    const int bpw = 32 / lpb;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t col = (int64_t)blockIdx.y * 32 + (lane & (lpb - 1));
    const int64_t PC = (int64_t)P * C;
    int64_t pos[M2L_NB];
    bool ok[M2L_NB];
#pragma unroll
    for (int b = 0; b < M2L_NB; ++b) {
        pos[b] = gr.first[oc] + (((int64_t)blockIdx.x - gr.tile[oc]) * M2L_WARPS + warp) * (M2L_NB * bpw) + b * bpw + lane / lpb;
        ok[b] = pos[b] < gr.first[oc + 1] && col < C;
    }
    float2 acc[M2L_NB][RP];
#pragma unroll
    for (int b = 0; b < M2L_NB; ++b)
#pragma unroll
        for (int q = 0; q < RP; ++q) acc[b][q] = make_float2(0.f, 0.f);
    const int total = f.dim == 2 ? 6 * 8 : 6 * 57;   // offset code of -d: total - code
    for (int sl = 0; sl < f.nslots; ++sl) {
        const float *Ko = f.K + (int64_t)(total - f.slot_off[oc * f.nslots + sl]) * P * P;
        __syncthreads();
        for (int q = threadIdx.x; q < P * RW; q += blockDim.x) {
            const int k = q / RW, m = q - k * RW;
            sK[q] = r0 + m < P ? __ldg(Ko + (int64_t)k * P + r0 + m) : 0.f;
        }
        int32_t src[M2L_NB];
        bool any = false;
#pragma unroll
        for (int b = 0; b < M2L_NB; ++b) {
            src[b] = ok[b] ? __ldg(f.m2l_src + (int64_t)sl * nm2l + pos[b]) : -1;
            any = any || src[b] >= 0;
        }
        __syncthreads();
        if (!__any_sync(0xffffffffu, any)) continue;
        const float *Ms[M2L_NB];
#pragma unroll
        for (int b = 0; b < M2L_NB; ++b) Ms[b] = M + (int64_t)(src[b] < 0 ? 0 : src[b]) * PC + col;
#pragma unroll 6
        for (int k = 0; k < P; ++k) {
            float2 mv[M2L_NB];
#pragma unroll
            for (int b = 0; b < M2L_NB; ++b) {
                const float v = src[b] >= 0 ? __ldg(Ms[b] + (int64_t)k * C) : 0.f;
                mv[b] = make_float2(v, v);
            }
            const float2 *kr = reinterpret_cast<const float2 *>(sK + k * RW);
#pragma unroll
            for (int q = 0; q < RP; ++q) {
                const float2 kv = kr[q];
#pragma unroll
                for (int b = 0; b < M2L_NB; ++b) acc[b][q] = __ffma2_rn(kv, mv[b], acc[b][q]);
            }
        }
    }
#pragma unroll
    for (int b = 0; b < M2L_NB; ++b) {
        if (!ok[b]) continue;
        const float scale = gr.inv_a[f.m2l_level[pos[b]]];
        float *o = Lc + (int64_t)f.m2l_box[pos[b]] * PC + col;
#pragma unroll
        for (int q = 0; q < RP; ++q) {
            const int m = r0 + 2 * q;
            if (m < P) o[(int64_t)m * C] = scale * acc[b][q].x;
            if (m + 1 < P) o[(int64_t)(m + 1) * C] = scale * acc[b][q].y;
        }
    }
}

// M2L of small trees, where the boxes of an octant fill few blocks (k_fmm_m2l waits for L2 in every slot, 5
// to 7 us, whatever the number of boxes): a block per (box, 32 columns, 64 or more target nodes).  Steps
// of MB_KC source nodes of a slot: K's rows for the block's target nodes and the source's multipoles come by
// asynchronous copies into two stages of shared memory, one step ahead.  Warps over groups of 8
// target nodes, a lane per column (lpb of them; 32 / lpb node groups a warp).  The same sums in the same
// order as k_fmm_m2l.
constexpr int MB_KC = 32;
__device__ __forceinline__ void copy_async(float *dst, const float *src, bool vec) {
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
    if (vec) asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
    else asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d), "l"(src) : "memory");
}
__global__ void __launch_bounds__(256) k_fmm_m2l_box(FmmDev f, int64_t C, int64_t nm2l, int noct, M2lGrid gr, int lpb,
                                                     int rows, const float *__restrict__ M, float *__restrict__ Lc) {
    extern __shared__ __align__(16) float sm[];   // two stages of K [MB_KC][rows], M [MB_KC][lpb]
    const int P = f.P, stage = MB_KC * (rows + lpb);
    const int64_t pos = blockIdx.x, PC = (int64_t)P * C, col0 = (int64_t)blockIdx.y * 32;
    int oc = 0;
    while (oc + 1 < noct && pos >= gr.first[oc + 1]) ++oc;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rb = blockIdx.z * rows, nr = min(rows, P - rb);
    const int c = lane & (lpb - 1), r0 = (warp * (32 / lpb) + lane / lpb) * 8;
    const bool ok = col0 + c < C && r0 < nr;
    const bool vec = (P & 3) == 0;   // rows of K by 16 bytes (C is a multiple of 4)
    const int total = f.dim == 2 ? 6 * 8 : 6 * 57;  // offset code of -d: total - code
    const int nc = (int)min((int64_t)lpb, C - col0);
    auto source = [&](int sl) { return __ldg(f.m2l_src + (int64_t)sl * nm2l + pos); };
    auto next_slot = [&](int sl) {
        while (sl < f.nslots && source(sl) < 0) ++sl;
        return sl;
    };
    auto fetch = [&](int sl, int k0, float *dst) {   // K[-offset] is K[offset] transposed: its rows are source nodes
        const int nk = min(MB_KC, P - k0), w = vec ? 4 : 1;
        const float *Ko = f.K + ((int64_t)(total - f.slot_off[oc * f.nslots + sl]) * P + k0) * P + rb;
        for (int q = threadIdx.x; q < nk * (nr / w); q += 256) {
            const int k = q / (nr / w), r = (q - k * (nr / w)) * w;
            copy_async(dst + k * rows + r, Ko + (int64_t)k * P + r, vec);
        }
        const float *Ms = M + (int64_t)source(sl) * PC + (int64_t)k0 * C + col0;
        float *dm = dst + MB_KC * rows;
        for (int q = threadIdx.x; q < nk * (nc / 4); q += 256) {
            const int k = q / (nc / 4), r = (q - k * (nc / 4)) * 4;
            copy_async(dm + k * lpb + r, Ms + (int64_t)k * C + r, true);
        }
    };
    float acc[8] = {};
    int sl = next_slot(0), k0 = 0, buf = 0;
    if (sl < f.nslots) fetch(sl, 0, sm);
    asm volatile("cp.async.commit_group;" ::: "memory");
    while (sl < f.nslots) {
        const int nk = min(MB_KC, P - k0);
        k0 += MB_KC;
        if (k0 >= P) {
            k0 = 0;
            sl = next_slot(sl + 1);
        }
        if (sl < f.nslots) fetch(sl, k0, sm + (buf ^ 1) * stage);
        asm volatile("cp.async.commit_group;" ::: "memory");
        asm volatile("cp.async.wait_group 1;" ::: "memory");   // this step's copies; the next one's go on
        __syncthreads();
        if (ok) {
            const float *sK = sm + buf * stage + r0, *sM = sm + buf * stage + MB_KC * rows + c;
#pragma unroll 4
            for (int k = 0; k < nk; ++k) {
                const float m = sM[k * lpb];
                const float4 a = *reinterpret_cast<const float4 *>(sK + k * rows);
                const float4 b = *reinterpret_cast<const float4 *>(sK + k * rows + 4);
                acc[0] = fmaf(a.x, m, acc[0]);
                acc[1] = fmaf(a.y, m, acc[1]);
                acc[2] = fmaf(a.z, m, acc[2]);
                acc[3] = fmaf(a.w, m, acc[3]);
                acc[4] = fmaf(b.x, m, acc[4]);
                acc[5] = fmaf(b.y, m, acc[5]);
                acc[6] = fmaf(b.z, m, acc[6]);
                acc[7] = fmaf(b.w, m, acc[7]);
            }
        }
        __syncthreads();   // before the next fetch overwrites this stage
        buf ^= 1;
    }
    if (!ok) return;
    const float scale = gr.inv_a[f.m2l_level[pos]];
    float *o = Lc + (int64_t)f.m2l_box[pos] * PC + col0 + c;
#pragma unroll
    for (int i = 0; i < 8; ++i)
        if (rb + r0 + i < P && r0 + i < nr) o[(int64_t)(rb + r0 + i) * C] = scale * acc[i];
}

// L2P and the near field: a warp per 32 atoms of a leaf (tgt_leaf, tgt_first), a lane per target
// atom, 4 CQ columns (blockIdx.y) in registers, so a pair's D_ij is computed once for them (once per 8 columns: 1431 us for the
// 250k-atom disk, order 6, 32 columns, against 726; sources staged by 32 took the apply from 2.57
// to 2.41 ms).  X rows and the leaf's local coefficients are uniform in the warp and come through L1.
// Bound by the chain of each source (distance, erf, multiply-adds) where warps are few: a leaf
// to a warp took 116 ms for an apply of 16 columns of a 15k-atom sphere (64 leaves) that takes 2.3.
template <int CQ>
__global__ void __launch_bounds__(128) k_fmm_l2p_near(FmmDev f, int64_t ngroups, int64_t C, int64_t Cp, int far,
                                                      const float *__restrict__ Xs, const float *__restrict__ Lc,
                                                      float *__restrict__ U) {
    __shared__ float sW[4][3][kMaxP][32];
    __shared__ float4 sS[4][32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t grp = (int64_t)blockIdx.x * 4 + warp;
    if (grp >= ngroups) return;
    const int64_t b = f.tgt_leaf[grp];
    const int64_t col0 = (int64_t)blockIdx.y * (4 * CQ);
    const int k1 = f.leaf_start[b + 1];
    const float a = 0.5f * f.h;
    const int i = f.tgt_first[grp] + lane;
    const bool act = i < k1;
    const float4 qi = act ? f.atl[i] : make_float4(0.f, 0.f, 0.f, 1.f);
    float2 lo[CQ], hi[CQ];
#pragma unroll
    for (int q = 0; q < CQ; ++q) lo[q] = hi[q] = make_float2(0.f, 0.f);
    auto add = [&](float d, const float4 *x) {
#pragma unroll
        for (int q = 0; q < CQ; ++q) {
            if (col0 + 4 * q >= Cp) break;
            const float4 v = __ldg(x + q);
            lo[q] = __ffma2_rn(make_float2(d, d), make_float2(v.x, v.y), lo[q]);
            hi[q] = __ffma2_rn(make_float2(d, d), make_float2(v.z, v.w), hi[q]);
        }
    };
    if (far && f.L >= 2) {
        const float y[3] = {qi.x / a, qi.y / a, qi.z / a};
        float tk[kMaxP];
        for (int d = 0; d < f.dim; ++d) {   // node_weights into shared memory
            tk[0] = 1.f;
            if (f.p > 1) tk[1] = y[d];
            for (int k = 2; k < f.p; ++k) tk[k] = 2.f * y[d] * tk[k - 1] - tk[k - 2];
            const float inv = 1.f / f.p;
            for (int m = 0; m < f.p; ++m) {
                float s = 0.f;
                for (int k = 1; k < f.p; ++k) s = fmaf(f.cheb[m * f.p + k], tk[k], s);
                sW[warp][d][m][lane] = inv + 2.f * inv * s;
            }
        }
        __syncwarp();
        const float *Lb = Lc + (f.leaf0 + b) * (int64_t)f.P * Cp + col0;
        if (f.dim == 2) {
            for (int m0 = 0; m0 < f.p; ++m0) {
                const float w0 = sW[warp][0][m0][lane];
                for (int m1 = 0; m1 < f.p; ++m1, Lb += Cp)
                    add(w0 * sW[warp][1][m1][lane], reinterpret_cast<const float4 *>(Lb));
            }
        } else {
            for (int m0 = 0; m0 < f.p; ++m0)
                for (int m1 = 0; m1 < f.p; ++m1) {
                    const float w01 = sW[warp][0][m0][lane] * sW[warp][1][m1][lane];
                    for (int m2 = 0; m2 < f.p; ++m2, Lb += Cp)
                        add(w01 * sW[warp][2][m2][lane], reinterpret_cast<const float4 *>(Lb));
                }
        }
        __syncwarp();
    }
    const float etai = act ? f.eta[i] : 0.f;
    for (int e = f.near_start[b]; e < f.near_start[b + 1]; ++e) {
        const int nb = f.near_leaf[e];
        const int dc = f.near_delta[e];
        const float ox = ((dc % 3) - 1) * f.h, oy = ((dc / 3) % 3 - 1) * f.h, oz = (dc / 9 - 1) * f.h;
        const int s1 = f.leaf_start[nb + 1];
        for (int c0 = f.leaf_start[nb]; c0 < s1; c0 += 32) {
            // 32 sources at a time: their records through shared memory, their X rows on the way into
            // L1 (one by one each source waited for L2: 1.1 us a source and warp with 32 columns)
            __syncwarp();
            if (c0 + lane < s1) {
                float4 v = __ldg(f.atl + c0 + lane);
                v.x += ox;   // source position in the target leaf's frame
                v.y += oy;
                v.z += oz;
                sS[warp][lane] = v;
                asm volatile("prefetch.global.L1 [%0];" ::"l"(Xs + (int64_t)(c0 + lane) * Cp + col0));
            }
            __syncwarp();
            const int je = min(c0 + 32, s1);
            for (int j = c0; j < je; ++j) {
                const float4 sj = sS[warp][j - c0];
                float4 xv[CQ];   // on their way while D_ij is computed
#pragma unroll
                for (int q = 0; q < CQ; ++q)
                    xv[q] = col0 + 4 * q < Cp ? __ldg(reinterpret_cast<const float4 *>(Xs + (int64_t)j * Cp + col0) + q)
                                              : make_float4(0.f, 0.f, 0.f, 0.f);
                const float dx = qi.x - sj.x, dy = qi.y - sj.y, dz = qi.z - sj.z;
                const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
                const float s2 = fmaf(qi.w, qi.w, sj.w * sj.w);
                const float rinv = rsqrtf(r2);
                float d = rinv;                   // erf(r / s) rounds to 1 in FP32 from r = 4 s on
                if (r2 < 16.f * s2) {
                    const float sinv = rsqrtf(s2);
                    // r -> 0 limit of erf(r / s) / r: 2 / (sqrt(pi) s)
                    d = r2 > 1e-24f ? erff(r2 * rinv * sinv) * rinv : 1.1283791670955126f * sinv;
                }
                if (j == i) d = etai;
#pragma unroll
                for (int q = 0; q < CQ; ++q) {
                    lo[q] = __ffma2_rn(make_float2(d, d), make_float2(xv[q].x, xv[q].y), lo[q]);
                    hi[q] = __ffma2_rn(make_float2(d, d), make_float2(xv[q].z, xv[q].w), hi[q]);
                }
            }
        }
    }
    if (act) {
        float *Ui = U + (int64_t)f.perm[i] * C + col0;
#pragma unroll
        for (int q = 0; q < CQ; ++q) {
            const float v[4] = {lo[q].x, lo[q].y, hi[q].x, hi[q].y};
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (col0 + 4 * q + j < C) Ui[4 * q + j] = v[j];
        }
    }
}

FmmDev dev_view(const Fmm *f) {
    FmmDev d{};
    d.dim = f->dim;
    d.p = f->p;
    d.P = f->P;
    d.L = f->L;
    d.h = (float)f->h;
    d.perm = f->perm;
    d.leaf_start = f->leaf_start;
    d.parent = f->parent;
    d.child_lo = f->child_lo;
    d.child_hi = f->child_hi;
    d.nslots = f->nslots;
    d.m2l_box = f->m2l_box;
    d.m2l_level = f->m2l_level;
    d.m2l_src = f->m2l_src;
    d.slot_off = f->slot_off;
    d.near_start = f->near_start;
    d.near_leaf = f->near_leaf;
    d.tgt_leaf = f->tgt_leaf;
    d.tgt_first = f->tgt_first;
    d.octant = f->octant;
    d.near_delta = f->near_delta;
    d.atl = f->atl;
    d.eta = f->eta;
    d.Tm = f->Tm;
    d.Tl = f->Tl;
    d.K = f->K;
    d.cheb = f->cheb;
    d.leaf0 = f->lvl0[f->L];
    return d;
}

}  // namespace

void fmm_free(Fmm *f) {
    if (!f) return;
    void *ptrs[] = {f->perm, f->leaf_start, f->atl, f->eta, f->parent, f->child_lo, f->child_hi, f->octant,
                    f->m2l_box, f->m2l_level, f->m2l_src, f->slot_off, f->near_start, f->near_leaf, f->near_delta,
                    f->tgt_leaf, f->tgt_first,
                    f->Tm, f->Tl, f->K, f->cheb};
    for (void *p : ptrs)
        if (p) cudaFree(p);
    delete f;
}

size_t fmm_bytes(const Fmm *f) { return f ? f->bytes : 0; }

void fmm_info(const Fmm *f, int64_t *out) {
    out[0] = f->dim;
    out[1] = f->L;
    out[2] = f->p;
    out[3] = f->nleaf;
    out[4] = f->nbox;
    out[5] = f->nil;
    out[6] = f->nnear;
}

int fmm_build(wfq_geom *g, int order, Fmm **out) {
    *out = nullptr;
    const int64_t n = g->n;
    std::vector<double> xyz((size_t)n * 3), eta((size_t)n);
    WFQ_CUDA(cudaMemcpy(xyz.data(), g->xyz, sizeof(double) * 3 * n, cudaMemcpyDeviceToHost));
    WFQ_CUDA(cudaMemcpy(eta.data(), g->eta, sizeof(double) * n, cudaMemcpyDeviceToHost));
    auto *f = new Fmm;
    std::unique_ptr<Fmm, void (*)(Fmm *)> guard(f, fmm_free);
    f->p = order;
    // tree: bounding cube (square when all z are equal), depth = the largest L with
    // side / 2^L >= r_far
    double mn[3], mx[3];
    for (int d = 0; d < 3; ++d) {
        mn[d] = mx[d] = xyz[d];
        for (int64_t i = 1; i < n; ++i) {
            mn[d] = std::min(mn[d], xyz[3 * i + d]);
            mx[d] = std::max(mx[d], xyz[3 * i + d]);
        }
    }
    const int dim = (mx[2] == mn[2]) ? 2 : 3;
    f->dim = dim;
    // nodes per box the tables and kernels are sized for
    if ((dim == 2 && order > 16) || (dim == 3 && order > 6))
        return fail(WFQ_EINVAL, "FMM order must be <= 16 for a flat structure and <= 6 for a 3D one");
    double wmax = 0.0;
    for (int64_t i = 0; i < n; ++i) wmax = std::max(wmax, std::sqrt(2.0 / kPi) / eta[i]);
    f->r_far = 6.0 * std::sqrt(2.0) * wmax;
    double ext = 0.0;
    for (int d = 0; d < dim; ++d) ext = std::max(ext, mx[d] - mn[d]);
    f->side = ext * (1.0 + std::ldexp(1.0, -20)) + 1e-300;
    double origin[3];
    for (int d = 0; d < 3; ++d) origin[d] = 0.5 * (mn[d] + mx[d]);
    for (int d = 0; d < dim; ++d) origin[d] -= 0.5 * f->side;
    int L = 0;
    while (f->side / std::ldexp(1.0, L + 1) >= f->r_far && L < 20) ++L;
    f->L = L;
    f->h = f->side / std::ldexp(1.0, L);
    f->P = 1;
    for (int d = 0; d < dim; ++d) f->P *= order;
    const int64_t nside = (int64_t)1 << L;

    // leaves: integer coordinates, Morton keys, atoms sorted by key
    std::vector<uint64_t> key((size_t)n);
    for (int64_t i = 0; i < n; ++i) {
        int64_t c[3] = {0, 0, 0};
        for (int d = 0; d < dim; ++d) {
            int64_t v = (int64_t)std::floor((xyz[3 * i + d] - origin[d]) / f->h);
            c[d] = std::min(std::max(v, (int64_t)0), nside - 1);
        }
        key[i] = morton(dim, c);
    }
    std::vector<int32_t> perm((size_t)n);
    std::iota(perm.begin(), perm.end(), 0);
    std::stable_sort(perm.begin(), perm.end(), [&](int32_t a, int32_t b) { return key[a] < key[b]; });

    // boxes of every level, sorted by key; global index = level offset + position
    std::vector<std::vector<uint64_t>> keys(L + 1);
    std::vector<int32_t> leaf_start;
    for (int64_t k = 0; k < n; ++k) {
        const uint64_t kk = key[perm[k]];
        if (keys[L].empty() || keys[L].back() != kk) {
            keys[L].push_back(kk);
            leaf_start.push_back((int32_t)k);
        }
    }
    leaf_start.push_back((int32_t)n);
    for (int l = L - 1; l >= 0; --l)
        for (uint64_t kk : keys[l + 1]) {
            const uint64_t pk = kk >> dim;
            if (keys[l].empty() || keys[l].back() != pk) keys[l].push_back(pk);
        }
    f->lvl0.assign(L + 2, 0);
    for (int l = 0; l <= L; ++l) f->lvl0[l + 1] = f->lvl0[l] + (int64_t)keys[l].size();
    f->nbox = f->lvl0[L + 1];
    f->nleaf = (int64_t)keys[L].size();
    std::vector<std::unordered_map<uint64_t, int32_t>> index(L + 1);
    for (int l = 0; l <= L; ++l)
        for (size_t q = 0; q < keys[l].size(); ++q) index[l][keys[l][q]] = (int32_t)(f->lvl0[l] + q);
    std::vector<int32_t> parent(f->nbox, -1), child_lo(f->nbox, 0), child_hi(f->nbox, 0);
    std::vector<int8_t> octant(f->nbox, 0);
    for (int l = 1; l <= L; ++l)
        for (size_t q = 0; q < keys[l].size(); ++q) {
            const int32_t gi = (int32_t)(f->lvl0[l] + q);
            const int32_t pg = index[l - 1].at(keys[l][q] >> dim);
            parent[gi] = pg;
            int64_t c[3] = {0, 0, 0};
            unmorton(dim, keys[l][q], c);
            int o = 0;
            for (int d = 0; d < dim; ++d) o |= (int)(c[d] & 1) << d;
            octant[gi] = (int8_t)o;
            if (child_hi[pg] == 0) child_lo[pg] = gi;
            child_hi[pg] = gi + 1;
        }

    // interaction lists (levels >= 2) and near lists (leaves).  A box's candidates are the children
    // (o) of its parent's neighbours (u); for boxes of one octant the same (u, o) are adjacent, so
    // the others, in order, are the octant's slots.
    const int noct = 1 << dim, nu = dim == 2 ? 9 : 27;
    f->nslots = dim == 2 ? 27 : 189;
    std::vector<int16_t> slot_off((size_t)noct * f->nslots);
    std::vector<int> slot_of((size_t)noct * nu * noct, -1);
    for (int t = 0; t < noct; ++t) {
        int sl = 0;
        for (int u = 0; u < nu; ++u)
            for (int o = 0; o < noct; ++o) {
                int far = 0, code = 0, mul = 1;
                for (int d = 0; d < dim; ++d, mul *= 7) {
                    const int pn = (d == 0 ? u % 3 : d == 1 ? (u / 3) % 3 : u / 9) - 1;
                    const int off = 2 * pn + ((o >> d) & 1) - ((t >> d) & 1);
                    far = std::max(far, std::abs(off));
                    code += (off + 3) * mul;
                }
                if (far <= 1) continue;
                slot_off[(size_t)t * f->nslots + sl] = (int16_t)code;
                slot_of[((size_t)t * nu + u) * noct + o] = sl++;
            }
    }
    std::vector<int32_t> m2l_box;
    std::vector<int8_t> m2l_level;
    for (int t = 0; t < noct; ++t) {
        f->oct_first[t] = (int32_t)m2l_box.size();
        for (int l = 2; l <= L; ++l)
            for (int64_t gi = f->lvl0[l]; gi < f->lvl0[l + 1]; ++gi)
                if (octant[gi] == t) {
                    m2l_box.push_back((int32_t)gi);
                    m2l_level.push_back((int8_t)l);
                }
    }
    f->oct_first[noct] = (int32_t)m2l_box.size();
    f->nm2l = (int64_t)m2l_box.size();
    std::vector<int32_t> m2l_src((size_t)f->nslots * f->nm2l, -1);
    for (int64_t q = 0; q < f->nm2l; ++q) {
        const int l = m2l_level[q], t = octant[m2l_box[q]];
        int64_t ct[3] = {0, 0, 0};
        unmorton(dim, keys[l][m2l_box[q] - f->lvl0[l]], ct);
        const int64_t lim = (int64_t)1 << (l - 1);
        for (int u = 0; u < nu; ++u) {
            int64_t pn[3] = {ct[0] / 2 + (u % 3) - 1, ct[1] / 2 + (u / 3) % 3 - 1, dim == 3 ? ct[2] / 2 + u / 9 - 1 : 0};
            bool ok = true;
            for (int d = 0; d < dim; ++d) ok = ok && pn[d] >= 0 && pn[d] < lim;
            if (!ok) continue;
            for (int o = 0; o < noct; ++o) {
                const int sl = slot_of[((size_t)t * nu + u) * noct + o];
                if (sl < 0) continue;
                int64_t cc[3] = {0, 0, 0};
                for (int d = 0; d < dim; ++d) cc[d] = 2 * pn[d] + ((o >> d) & 1);
                auto it = index[l].find(morton(dim, cc));
                if (it == index[l].end()) continue;
                m2l_src[(size_t)sl * f->nm2l + q] = it->second;
                ++f->nil;
            }
        }
    }
    std::vector<int32_t> near_start(f->nleaf + 1, 0), near_leaf;
    std::vector<int8_t> near_delta;
    for (int64_t q = 0; q < f->nleaf; ++q) {
        int64_t ct[3] = {0, 0, 0};
        unmorton(dim, keys[L][q], ct);
        const int nd = dim == 2 ? 9 : 27;
        for (int u = 0; u < nd; ++u) {
            const int64_t dv[3] = {(u % 3) - 1, (u / 3) % 3 - 1, dim == 3 ? u / 9 - 1 : 0};
            int64_t cc[3] = {ct[0] + dv[0], ct[1] + dv[1], ct[2] + dv[2]};
            bool ok = true;
            for (int d = 0; d < dim; ++d) ok = ok && cc[d] >= 0 && cc[d] < nside;
            if (!ok) continue;
            auto it = index[L].find(morton(dim, cc));
            if (it == index[L].end()) continue;
            near_leaf.push_back((int32_t)(it->second - f->lvl0[L]));
            near_delta.push_back((int8_t)((dv[0] + 1) + 3 * (dv[1] + 1) + 9 * (dv[2] + 1)));
        }
        near_start[q + 1] = (int32_t)near_leaf.size();
    }
    f->nnear = (int64_t)near_leaf.size();

    // atoms relative to their leaf's centre (sorted order)
    std::vector<float4> atl((size_t)n);
    std::vector<float> etas((size_t)n);
    for (int64_t q = 0; q < f->nleaf; ++q) {
        int64_t c[3] = {0, 0, 0};
        unmorton(dim, keys[L][q], c);
        double ctr[3];
        for (int d = 0; d < 3; ++d) ctr[d] = d < dim ? origin[d] + (c[d] + 0.5) * f->h : mn[2];
        for (int32_t k = leaf_start[q]; k < leaf_start[q + 1]; ++k) {
            const int32_t i = perm[k];
            atl[k] = make_float4((float)(xyz[3 * i] - ctr[0]), (float)(xyz[3 * i + 1] - ctr[1]),
                                 (float)(xyz[3 * i + 2] - ctr[2]), (float)(std::sqrt(2.0 / kPi) / eta[i]));
            etas[k] = (float)eta[i];
        }
    }

    // operators (FP64, stored as FP32)
    const int p = order, P = f->P;
    std::vector<double> xm(p);
    for (int m = 0; m < p; ++m) xm[m] = std::cos((2.0 * m + 1.0) * kPi / (2.0 * p));
    std::vector<float> cheb((size_t)p * p);
    for (int m = 0; m < p; ++m)
        for (int k = 0; k < p; ++k) cheb[m * p + k] = (float)std::cos(k * std::acos(xm[m]));
    auto node = [&](int m, int d) {   // per-dimension node index of node m
        return dim == 2 ? (d == 0 ? m / p : m % p) : (d == 0 ? m / (p * p) : d == 1 ? (m / p) % p : m % p);
    };
    const int Pp = (P + 7) / 8 * 8;   // rows of the node tables, in groups of 8
    std::vector<float> Tm((size_t)(1 << dim) * P * Pp, 0.f), Tl((size_t)(1 << dim) * P * Pp, 0.f);
    {
        std::vector<double> S1((size_t)2 * p * p);   // [bit][parent node][child node]
        std::vector<double> w(p);
        for (int bit = 0; bit < 2; ++bit)
            for (int mc = 0; mc < p; ++mc) {
                cheb_weights(p, (bit - 0.5) + 0.5 * xm[mc], w.data());
                for (int mp = 0; mp < p; ++mp) S1[((size_t)bit * p + mp) * p + mc] = w[mp];
            }
        for (int o = 0; o < (1 << dim); ++o)
            for (int m = 0; m < P; ++m)
                for (int mc = 0; mc < P; ++mc) {
                    double v = 1.0;
                    for (int d = 0; d < dim; ++d) v *= S1[((size_t)((o >> d) & 1) * p + node(m, d)) * p + node(mc, d)];
                    Tm[((size_t)o * P + mc) * Pp + m] = (float)v;
                    Tl[((size_t)o * P + m) * Pp + mc] = (float)v;
                }
    }
    const int noff = dim == 2 ? 49 : 343;
    std::vector<float> K((size_t)noff * P * P, 0.f);
    for (int code = 0; code < noff; ++code) {
        const int dl[3] = {code % 7 - 3, (code / 7) % 7 - 3, dim == 3 ? code / 49 - 3 : 0};
        if (std::max(std::abs(dl[0]), std::max(std::abs(dl[1]), std::abs(dl[2]))) <= 1) continue;
        for (int m = 0; m < P; ++m)
            for (int ms = 0; ms < P; ++ms) {
                double r2 = 0.0;
                for (int d = 0; d < dim; ++d) {
                    const double v = xm[node(m, d)] - xm[node(ms, d)] - 2.0 * dl[d];
                    r2 += v * v;
                }
                K[((size_t)code * P + m) * P + ms] = (float)(1.0 / std::sqrt(r2));
            }
    }

    wfq_ctx *ctx = g->ctx;
    WFQ_TRY(upload(ctx, f, &f->perm, perm));
    WFQ_TRY(upload(ctx, f, &f->leaf_start, leaf_start));
    WFQ_TRY(upload(ctx, f, &f->atl, atl));
    WFQ_TRY(upload(ctx, f, &f->eta, etas));
    WFQ_TRY(upload(ctx, f, &f->parent, parent));
    WFQ_TRY(upload(ctx, f, &f->child_lo, child_lo));
    WFQ_TRY(upload(ctx, f, &f->child_hi, child_hi));
    WFQ_TRY(upload(ctx, f, &f->octant, octant));
    WFQ_TRY(upload(ctx, f, &f->m2l_box, m2l_box));
    WFQ_TRY(upload(ctx, f, &f->m2l_level, m2l_level));
    WFQ_TRY(upload(ctx, f, &f->m2l_src, m2l_src));
    WFQ_TRY(upload(ctx, f, &f->slot_off, slot_off));
    WFQ_TRY(upload(ctx, f, &f->near_start, near_start));
    WFQ_TRY(upload(ctx, f, &f->near_leaf, near_leaf));
    WFQ_TRY(upload(ctx, f, &f->near_delta, near_delta));
    std::vector<int32_t> tgt_leaf, tgt_first;
    for (int64_t b = 0; b < f->nleaf; ++b)
        for (int32_t i = leaf_start[b]; i < leaf_start[b + 1]; i += 32) {
            tgt_leaf.push_back((int32_t)b);
            tgt_first.push_back(i);
        }
    f->ngroups = (int64_t)tgt_leaf.size();
    WFQ_TRY(upload(ctx, f, &f->tgt_leaf, tgt_leaf));
    WFQ_TRY(upload(ctx, f, &f->tgt_first, tgt_first));
    WFQ_TRY(upload(ctx, f, &f->Tm, Tm));
    WFQ_TRY(upload(ctx, f, &f->Tl, Tl));
    WFQ_TRY(upload(ctx, f, &f->K, K));
    WFQ_TRY(upload(ctx, f, &f->cheb, cheb));
    *out = guard.release();
    return WFQ_OK;
}

int d_apply_fmm(const wfq_geom *g, int64_t cc, const float2 *X, float2 *U, cudaStream_t s) {
    const Fmm *f = g->fmm;
    if (!f) return fail(WFQ_EUNSUPPORTED, "WFQ_PREC_FMM needs wfq_fmm_build on this geometry first");
    const int64_t C = 2 * cc, Cp = round_up(C, 4), n = g->n;   // internal rows are padded to 16 bytes
    const FmmDev fd = dev_view(f);
    KScope ks(g->ctx, WFQ_KT_FMM, s, (double)n * (double)n);
    DevBuf<float> M, Lc, Xs;
    const int L = f->L, P = f->P, Pp = (P + 7) / 8 * 8;
    const unsigned cols32 = (unsigned)((Cp + 31) / 32);
    const unsigned node_threads = 32u * (unsigned)std::min(8, (P + 7) / 8);   // M2M, L2L: a warp per 8 nodes
    WFQ_TRY(Xs.alloc(g->ctx, (size_t)n * Cp, s));
    k_fmm_sort_x<<<(unsigned)((n * Cp + 255) / 256), 256, 0, s>>>(n, C, Cp, fd.perm, reinterpret_cast<const float *>(X), Xs.ptr);
    note_launch();
    WFQ_CUDA(cudaGetLastError());
    if (L >= 2) {
        const size_t per = (size_t)f->nbox * P * Cp;
        WFQ_TRY(M.alloc(g->ctx, per, s));
        WFQ_TRY(Lc.alloc(g->ctx, per, s));
        const size_t p2m_smem = sizeof(float) * (32 * 3 * kMaxP + 32 * Cp);
        if (p2m_smem > 48 * 1024)
            WFQ_CUDA(cudaFuncSetAttribute(k_fmm_p2m, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)p2m_smem));
        k_fmm_p2m<<<(unsigned)f->nleaf, 128, p2m_smem, s>>>(fd, Cp, Xs.ptr, M.ptr);
        note_launch();
        WFQ_CUDA(cudaGetLastError());
        for (int l = L - 1; l >= 2; --l) {
            k_fmm_m2m<<<dim3((unsigned)(f->lvl0[l + 1] - f->lvl0[l]), cols32), node_threads, 0, s>>>(fd, Pp, Cp, f->lvl0[l], M.ptr);
            note_launch();
        }
        // lanes per box: the columns of a block rounded up to a power of two
        int lpb = 4;
        while (lpb < Cp && lpb < 32) lpb *= 2;
        const int noct = 1 << f->dim, bpb = M2L_WARPS * M2L_NB * (32 / lpb);
        M2lGrid gr{};
        int tiles = 0;
        for (int t = 0; t < noct; ++t) {
            gr.first[t] = f->oct_first[t];
            gr.tile[t] = tiles;
            tiles += (f->oct_first[t + 1] - f->oct_first[t] + bpb - 1) / bpb;
        }
        gr.first[noct] = f->oct_first[noct];
        for (int l = 0; l <= L && l < 24; ++l) gr.inv_a[l] = (float)(2.0 * std::ldexp(1.0, l) / f->side);
        // target nodes per block: the choice with the fewest padded nodes, wider first
        int best = 18;
        for (int rp : {16, 13, 8})
            if (round_up(P, 2 * rp) < round_up(P, 2 * best)) best = rp;
        const dim3 grid((unsigned)tiles, cols32, (unsigned)((P + 2 * best - 1) / (2 * best)));
        const size_t sm = sizeof(float) * (size_t)P * 2 * best;   // at most 256 x 36 floats
        const unsigned th = 32 * M2L_WARPS;
        const int nodes = 64 * (32 / lpb), rows = (int)std::min<int64_t>(nodes, round_up(P, 8));
        const dim3 gbox((unsigned)f->nm2l, cols32, (unsigned)((P + rows - 1) / rows));
        // A slot takes a block of boxes of one octant about 0.1 us per source node (2 blocks an SM at a
        // time); box by box the interactions take about 1 / 70 us per 64 x 64 nodes and 32 columns.
        // us, octant / box: 15k-atom sphere 1277 / 199, 30k 1549 / 552 (1682 / 972 with 32 columns), 20000-atom
        // tube 664 / 173; a 74k-atom disk's apply 474 / 691.
        const double waves = std::ceil((double)grid.x * grid.y * grid.z / (2.0 * g->ctx->num_sms));
        const bool by_box = (double)f->nil * cols32 * P * P / 4096.0 / 70.0 < 0.1 * f->nslots * P * waves;
        if (by_box) {
            const size_t smb = sizeof(float) * 2 * MB_KC * (size_t)(rows + lpb);
            if (smb > 48 * 1024)   // at most 67 KiB (256 nodes); the limit is the process's, never one launch's
                WFQ_CUDA(cudaFuncSetAttribute(k_fmm_m2l_box, cudaFuncAttributeMaxDynamicSharedMemorySize, 72 * 1024));
            k_fmm_m2l_box<<<gbox, 256, smb, s>>>(fd, Cp, f->nm2l, noct, gr, lpb, rows, M.ptr, Lc.ptr);
        } else switch (best) {
            case 18: k_fmm_m2l<18><<<grid, th, sm, s>>>(fd, Cp, f->nm2l, noct, gr, lpb, M.ptr, Lc.ptr); break;
            case 16: k_fmm_m2l<16><<<grid, th, sm, s>>>(fd, Cp, f->nm2l, noct, gr, lpb, M.ptr, Lc.ptr); break;
            case 13: k_fmm_m2l<13><<<grid, th, sm, s>>>(fd, Cp, f->nm2l, noct, gr, lpb, M.ptr, Lc.ptr); break;
            default: k_fmm_m2l<8><<<grid, th, sm, s>>>(fd, Cp, f->nm2l, noct, gr, lpb, M.ptr, Lc.ptr); break;
        }
        note_launch();
        WFQ_CUDA(cudaGetLastError());
        for (int l = 3; l <= L; ++l) {
            k_fmm_l2l<<<dim3((unsigned)(f->lvl0[l + 1] - f->lvl0[l]), cols32), node_threads, 0, s>>>(fd, Pp, Cp, f->lvl0[l], Lc.ptr);
            note_launch();
        }
        WFQ_CUDA(cudaGetLastError());
    }
    // columns per thread: the fewest multiple of 4 (4, 8, 16, 32) that holds them, but fewer, with D_ij
    // computed again for the others, while that leaves under 16 warps an SM (a warp's sources are a chain)
    int cq = Cp > 16 ? 8 : Cp > 8 ? 4 : Cp > 4 ? 2 : 1;
    auto warps = [&](int q) { return f->ngroups * ((Cp + 4 * q - 1) / (4 * q)); };
    while (cq > 2 && warps(cq) < 16 * (int64_t)g->ctx->num_sms) cq /= 2;
    const dim3 gnear((unsigned)((f->ngroups + 3) / 4), (unsigned)((Cp + 4 * cq - 1) / (4 * cq)));
    const int far = L >= 2 ? 1 : 0;
    float *Uf = reinterpret_cast<float *>(U);
    switch (cq) {
        case 8: k_fmm_l2p_near<8><<<gnear, 128, 0, s>>>(fd, f->ngroups, C, Cp, far, Xs.ptr, Lc.ptr, Uf); break;
        case 4: k_fmm_l2p_near<4><<<gnear, 128, 0, s>>>(fd, f->ngroups, C, Cp, far, Xs.ptr, Lc.ptr, Uf); break;
        case 2: k_fmm_l2p_near<2><<<gnear, 128, 0, s>>>(fd, f->ngroups, C, Cp, far, Xs.ptr, Lc.ptr, Uf); break;
        default: k_fmm_l2p_near<1><<<gnear, 128, 0, s>>>(fd, f->ngroups, C, Cp, far, Xs.ptr, Lc.ptr, Uf); break;
    }
    note_launch();
    WFQ_CUDA(cudaGetLastError());
    return WFQ_OK;
}

}  // namespace wfq
