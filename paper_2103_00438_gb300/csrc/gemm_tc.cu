// libwfq entry to the tcgen05 GEMMs of gemm_tc.cuh and gemm_mf.cuh (the dense product of
// the mixed operator, U = D X with three bf16 products), with their autotuner: the first
// product of a shape on a context times the pipeline depths below on the real operands and
// keeps the fastest for later products of that shape.  The depth changes only how far the
// loads run ahead of the tensor cores, never which products are summed in which order, so
// the choice cannot change a result.
#include <vector>

#include "common.h"
#include "gemm_mf.cuh"
#include "gemm_tc.cuh"

namespace wfq {

namespace {

// pipeline depths tried (0: as deep as shared memory allows, at most the kernels' maximum)
constexpr int kStageChoices[] = {0, 4, 3, 2};

template <class Launch>
int tuned_stages(const wfq_geom *g, int64_t key, cudaStream_t s, Launch launch) {
    {
        std::lock_guard<std::mutex> lk(g->ctx->tune_mu);
        auto it = g->ctx->tuned.find(key);
        if (it != g->ctx->tuned.end()) return it->second;
    }
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) {
        cudaGetLastError();
        if (e0) cudaEventDestroy(e0);
        return 0;
    }
    int best = 0;
    float best_ms = 1e30f;
    for (int st : kStageChoices) {
        float ms = 0.f;
        bool ok = true;
        for (int rep = 0; rep < 3 && ok; ++rep) {   // the first of the three warms up
            if (rep == 1) cudaEventRecord(e0, s);
            ok = launch(st) == cudaSuccess;
        }
        cudaEventRecord(e1, s);
        if (!ok || cudaEventSynchronize(e1) != cudaSuccess || cudaEventElapsedTime(&ms, e0, e1) != cudaSuccess) {
            cudaGetLastError();
            continue;
        }
        if (ms < best_ms) {
            best_ms = ms;
            best = st;
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    std::lock_guard<std::mutex> lk(g->ctx->tune_mu);
    g->ctx->tuned[key] = best;
    return best;
}

// The bounded waits run out on purpose (wfq_selftest_wait): warp 0 waits for a barrier that nothing
// completes until its lane 0, whose limit is the shortest, has given up; warp 1 then completes it, so that
// the lanes see different things.  out: lanes of warp 0 whose wait succeeded, by mbar_wait (round 0) and
// by mbar_wait_warp (round 1), and the code recorded.  Every loop here ends by its limit.
__global__ void __launch_bounds__(64) k_selftest_wait(unsigned long long limit_ns, int *err, int *out) {
    __shared__ __align__(8) uint64_t bar[2];
    __shared__ int abort_flag[2];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int r = 0; r < 2; ++r) {
            tc::mbar_init(tc::smem_u32(bar + r), 1);
            abort_flag[r] = 0;
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    tc::Params p{};
    p.err = err;
    p.timeout_ns = lane == 0 ? limit_ns : 50 * limit_ns;
    for (int r = 0; r < 2; ++r) {
        volatile int *flag = abort_flag + r;
        if (warp == 0) {
            const bool ok = r == 0 ? tc::mbar_wait(tc::smem_u32(bar + r), 0u, p, 9, flag)
                                   : tc::mbar_wait_warp(tc::smem_u32(bar + r), 0u, p, 9, flag);
            const unsigned lanes = __ballot_sync(0xffffffffu, ok);
            if (lane == 0) out[r] = __popc(lanes);
        } else if (lane == 0) {
            const uint64_t t0 = tc::global_ns();
            while (!*flag && tc::global_ns() - t0 < 100 * limit_ns) {
            }
            tc::mbar_arrive(tc::smem_u32(bar + r));
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) out[2] = *err;
}

// autotuner keys of the GEMMs: bit 60 set (the GEMV keys stay below 2^40), kernel id, shape
inline int64_t gemm_key(int kernel, int64_t npad, int64_t cpad) {
    return ((int64_t)1 << 60) | ((int64_t)kernel << 56) | (npad << 20) | cpad;
}

}  // namespace

int gemm_3xbf16_mf(const wfq_geom *g, int64_t cpad, const __nv_bfloat16 *Xhi, const __nv_bfloat16 *Xlo, float *U,
                   int64_t ldu, cudaStream_t s, int *err) {
    if (!err) err = g->ctx->dev_err;
    std::string msg;
    int launches = 0;
    // timing twelve launches costs seconds at a million atoms (1.4 s per launch): large
    // shapes take the deepest pipeline without a trial
    const int st = g->npad > 262144 ? 0 : tuned_stages(g, gemm_key(2, g->npad, cpad), s, [&](int stg) {
        int l = 0;
        const cudaError_t e = tc::gemm3_mf(g->atom32, g->atom32p, g->n, g->npad, Xhi, Xlo, cpad, U, ldu, g->ctx->num_sms,
                                           err, s, &l, nullptr, stg);
        for (int i = 0; i < l; ++i) note_launch();
        return e;
    });
    KScope ks(g->ctx, WFQ_KT_GEMM_MIXED, s, 6.0 * (double)g->n * (double)g->n * (double)ldu);
    cudaError_t e = tc::gemm3_mf(g->atom32, g->atom32p, g->n, g->npad, Xhi, Xlo, cpad, U, ldu, g->ctx->num_sms, err,
                                 s, &launches, &msg, st);
    for (int i = 0; i < launches; ++i) note_launch();
    if (e != cudaSuccess) {
        cudaGetLastError();
        return fail(WFQ_ECUDA, "matrix-free tensor-core GEMM: " + (msg.empty() ? std::string(cudaGetErrorString(e)) : msg));
    }
    return WFQ_OK;
}

int gemm_3xbf16(const wfq_geom *g, int64_t cpad, const __nv_bfloat16 *Xhi, const __nv_bfloat16 *Xlo, float *U,
                int64_t ldu, cudaStream_t s, int *err) {
    if (!err) err = g->ctx->dev_err;
    std::string msg;
    int launches = 0;
    const int st = tuned_stages(g, gemm_key(1, g->npad, cpad), s, [&](int stg) {
        int l = 0;
        const cudaError_t e = tc::gemm3_tc(g->Dhi, g->Dlo, g->n, g->npad, Xhi, Xlo, cpad, U, ldu, g->ctx->num_sms,
                                           err, s, &l, nullptr, stg);
        for (int i = 0; i < l; ++i) note_launch();
        return e;
    });
    KScope ks(g->ctx, WFQ_KT_GEMM_MIXED, s, 6.0 * (double)g->n * (double)g->n * (double)ldu);
    cudaError_t e = tc::gemm3_tc(g->Dhi, g->Dlo, g->n, g->npad, Xhi, Xlo, cpad, U, ldu, g->ctx->num_sms,
                                 err, s, &launches, &msg, st);
    for (int i = 0; i < launches; ++i) note_launch();
    if (e != cudaSuccess) {
        cudaGetLastError();
        return fail(WFQ_ECUDA, "tensor-core GEMM: " + (msg.empty() ? std::string(cudaGetErrorString(e)) : msg));
    }
    return WFQ_OK;
}

int selftest_wait(wfq_ctx *ctx, int limit_us, int *out, cudaStream_t s) {
    DevBuf<int> buf;
    WFQ_TRY(buf.alloc(ctx, 4, s));
    WFQ_CUDA(cudaMemsetAsync(buf.ptr, 0, 4 * sizeof(int), s));
    k_selftest_wait<<<1, 64, 0, s>>>(1000ull * (unsigned long long)limit_us, buf.ptr + 3, buf.ptr);
    note_launch();
    WFQ_CUDA(cudaGetLastError());
    WFQ_CUDA(cudaMemcpyAsync(out, buf.ptr, 3 * sizeof(int), cudaMemcpyDeviceToHost, s));
    WFQ_CUDA(cudaStreamSynchronize(s));
    return WFQ_OK;
}

}  // namespace wfq
