// numeric_launch_f32.cuh -- the launches of the pair geometry + quadrature kernels with float
// quadrature, templated on the statistics switch STS (0: the assembly's kernels, without the
// record hashes; 1: nl_interactions' kernels, with them).  Included by numeric_f32.cu (STS = 0)
// and numeric_f32_stats.cu (STS = 1), so that the two sets of kernels compile side by side.
#pragma once

#include "numeric.cuh"

namespace nlf32 {


// the deferred items of a launch, then the sums of each pair's items
template <int BALL, bool INV>
nl_status launch_deferred(nl_ctx *ctx, const nlq::NumArgs &A, unsigned threads)
{
    int blocks = 0;
    nl_status s = nl_deferred_blocks(ctx, &blocks);
    if (s != NL_OK) return s;
    nlq::k_deferred<BALL, INV><<<blocks, threads, 0, ctx->stream>>>(A); ++ctx->launches;
    nlq::k_defer_merge<float><<<blocks, 256, 0, ctx->stream>>>(A); ++ctx->launches;
    NL_CK(cudaGetLastError());
    return NL_OK;
}

// singular kernel.  stage 0: the boundary kernel (and its queue counters' reset); stage 1: the
// near-field and deferred items
template <int BALL, int STS>
nl_status launch_boundary(nl_ctx *ctx, const nlq::NumArgs &A, unsigned grid, unsigned threads, int stage)
{
    if (stage == 0) {
        if (A.defer) NL_CK(cudaMemsetAsync(A.defer_n, 0, sizeof(int), ctx->stream));
        if (A.nearq) NL_CK(cudaMemsetAsync(A.near_n, 0, sizeof(int), ctx->stream));
        const size_t smem = sizeof(nlq::BoundaryShared<float>) * nlq::kWarpsPerBlock;
        // with its near-field queue: a kernel without the near rule's code
        if (A.nearq) {
            NL_CK(cudaFuncSetAttribute(nlq::k_boundary<BALL, float, true, STS>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
            nlq::k_boundary<BALL, float, true, STS><<<grid, threads, smem, ctx->stream>>>(A); ++ctx->launches;
        } else {
            NL_CK(cudaFuncSetAttribute(nlq::k_boundary<BALL, float, false, STS>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
            nlq::k_boundary<BALL, float, false, STS><<<grid, threads, smem, ctx->stream>>>(A); ++ctx->launches;
        }
        NL_CK(cudaGetLastError());
        return NL_OK;
    }
    if (A.nearq) {   // the near-field whole items the boundary kernel queued
        // one resident wave: every warp strides over the queue, so a second wave of blocks
        // would only idle while the first finishes
        int nsm = 0, per_sm = 0;
        NL_CK(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, ctx->device));
        NL_CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, nlq::k_near<BALL>, threads, 0));
        const int blocks = (nsm > 0 ? nsm : 1) * (per_sm > 0 ? per_sm : 1);
        nlq::k_near<BALL><<<blocks, threads, 0, ctx->stream>>>(A); ++ctx->launches;
        NL_CK(cudaGetLastError());
    }
    return A.defer ? launch_deferred<BALL, true>(ctx, A, threads) : NL_OK;
}

template <int STS>
nl_status launch_ball(nl_ctx *ctx, const nlq::NumArgs &A, int ball, unsigned grid, unsigned threads, int stage)
{
    switch (ball) {
    case NL_BALL_BARYCENTER: return launch_boundary<NL_BALL_BARYCENTER, STS>(ctx, A, grid, threads, stage);
    case NL_BALL_NOCAPS: return launch_boundary<NL_BALL_NOCAPS, STS>(ctx, A, grid, threads, stage);
    case NL_BALL_APPROXCAPS: return launch_boundary<NL_BALL_APPROXCAPS, STS>(ctx, A, grid, threads, stage);
    case NL_BALL_EXACTCAPS: return launch_boundary<NL_BALL_EXACTCAPS, STS>(ctx, A, grid, threads, stage);
    case NL_BALL_NGON: return launch_boundary<NL_BALL_NGON, STS>(ctx, A, grid, threads, stage);
    case NL_BALL_OVERLAP: return launch_boundary<NL_BALL_OVERLAP, STS>(ctx, A, grid, threads, stage);
    default: return nl_fail(ctx, NL_EINVAL, "unknown ball mode");
    }
}

// constant kernel: one kernel for all candidates, then the deferred items
template <int BALL, int STS>
nl_status launch_const_k(nl_ctx *ctx, const nlq::NumArgs &A, unsigned grid, unsigned threads)
{
    if (A.defer_n) NL_CK(cudaMemsetAsync(A.defer_n, 0, sizeof(int), ctx->stream));
    const size_t smem = sizeof(nlq::ConstShared<BALL, float>) * nlq::kWarpsPerBlock;
    NL_CK(cudaFuncSetAttribute(nlq::k_const<BALL, float, STS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)smem));
    nlq::k_const<BALL, float, STS><<<grid, threads, smem, ctx->stream>>>(A); ++ctx->launches;
    NL_CK(cudaGetLastError());
    if constexpr (nlq::kConstQueue<BALL, float>)
        if (A.defer) return launch_deferred<nlq::kGeoBall<BALL>, false>(ctx, A, threads);
    return NL_OK;
}

template <int STS>
nl_status launch_const(nl_ctx *ctx, const nlq::NumArgs &A, int ball, unsigned grid, unsigned threads)
{
    switch (ball) {
    case NL_BALL_BARYCENTER: return launch_const_k<NL_BALL_BARYCENTER, STS>(ctx, A, grid, threads);
    case NL_BALL_NOCAPS: return launch_const_k<NL_BALL_NOCAPS, STS>(ctx, A, grid, threads);
    case NL_BALL_APPROXCAPS: return launch_const_k<NL_BALL_APPROXCAPS, STS>(ctx, A, grid, threads);
    case NL_BALL_EXACTCAPS: return launch_const_k<NL_BALL_EXACTCAPS, STS>(ctx, A, grid, threads);
    case NL_BALL_NGON: return launch_const_k<NL_BALL_NGON, STS>(ctx, A, grid, threads);
    case nlq::kBallNgonAny: return launch_const_k<nlq::kBallNgonAny, STS>(ctx, A, grid, threads);
    case NL_BALL_OVERLAP: return launch_const_k<NL_BALL_OVERLAP, STS>(ctx, A, grid, threads);
    case NL_BALL_BARY_NOCAPS: return launch_const_k<NL_BALL_BARY_NOCAPS, STS>(ctx, A, grid, threads);
    case NL_BALL_BARY_APPROXCAPS: return launch_const_k<NL_BALL_BARY_APPROXCAPS, STS>(ctx, A, grid, threads);
    default: return nl_fail(ctx, NL_EINVAL, "unknown ball mode");
    }
}

template <int STS>
nl_status launch_numeric_f32_sts(nl_ctx *ctx, const nlq::NumArgs &A, int ball, bool one_stream)
{
    const unsigned grid = (unsigned)((A.K + nlq::kWarpsPerBlock - 1) / nlq::kWarpsPerBlock);
    const unsigned threads = nlq::kWarpsPerBlock * 32;
    if (A.kernel == NL_KERNEL_CONST) {
        NL_CK(cudaMemsetAsync(A.mbb, 0, sizeof(double) * 6 * (size_t)A.K, ctx->stream));
        return launch_const<STS>(ctx, A, ball, grid, threads);
    }
    nl_status s = one_stream ? nl_numeric_zero(ctx, A) : nl_numeric_fork(ctx, A);
    if (s != NL_OK) return s;
    // the boundary kernel first, so that its blocks are dispatched before the interior kernel's
    s = launch_ball<STS>(ctx, A, ball, grid, threads, 0);
    s = one_stream ? nl_numeric_interior_same<float, STS>(ctx, A, grid, threads, s)
                   : nl_numeric_interior_join<float, STS>(ctx, A, grid, threads, s);
    if (s != NL_OK) return s;
    return launch_ball<STS>(ctx, A, ball, grid, threads, 1);
}

}  // namespace nlf32
