// numeric_batch_f32.cu -- instantiation of the persistent batched numeric kernels with float
// quadrature: one interior launch for every problem of a batch with this value type, one
// boundary launch per ball mode x kernel type present.
#include "numeric.cuh"

namespace {

// one launch of a persistent kernel; SH: its per-warp shared memory
template <typename SH, typename K>
nl_status launch(nl_ctx *ctx, K kernel, const nlq::NumArgs *dA, const nlq::BatchItem *items, int n_items, int *counter,
                 int blocks, bool set_attr, int *per_sm)
{
    const size_t smem = sizeof(SH) * nlq::kWarpsPerBlock;
    if (per_sm || set_attr)
        NL_CK(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    if (per_sm) {
        NL_CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, kernel, nlq::kWarpsPerBlock * 32, smem));
        return NL_OK;
    }
    kernel<<<blocks, nlq::kWarpsPerBlock * 32, smem, ctx->stream>>>(dA, items, n_items, counter);
    ++ctx->launches;
    NL_CK(cudaGetLastError());
    return NL_OK;
}

template <int BALL>
nl_status boundary(nl_ctx *ctx, bool inv, const nlq::NumArgs *dA, const nlq::BatchItem *items, int n_items,
                   int *counter, int blocks, bool set_attr, int *per_sm)
{
    if constexpr (BALL != nlq::kBallNgonAny && !nlq::kSupportBall<BALL>)
        if (inv)
            return launch<nlq::BoundaryShared<float>>(ctx, nlq::k_boundary_batch<BALL, float>, dA, items, n_items, counter,
                                                   blocks, set_attr, per_sm);
    if (inv) return nl_fail(ctx, NL_EINVAL, "unknown ball mode");
    return launch<nlq::ConstShared<BALL, float>>(ctx, nlq::k_const_batch<BALL, float>, dA, items, n_items, counter, blocks,
                                              set_attr, per_sm);
}

nl_status boundary_ball(nl_ctx *ctx, int ball, bool inv, const nlq::NumArgs *dA, const nlq::BatchItem *items,
                        int n_items, int *counter, int blocks, bool set_attr, int *per_sm)
{
#define NL_CASE(B) \
    case B: return boundary<B>(ctx, inv, dA, items, n_items, counter, blocks, set_attr, per_sm)
    switch (ball) {
        NL_CASE(NL_BALL_BARYCENTER);
        NL_CASE(NL_BALL_NOCAPS);
        NL_CASE(NL_BALL_APPROXCAPS);
        NL_CASE(NL_BALL_EXACTCAPS);
        NL_CASE(NL_BALL_NGON);
        NL_CASE(nlq::kBallNgonAny);
        NL_CASE(NL_BALL_OVERLAP);
        NL_CASE(NL_BALL_BARY_NOCAPS);
        NL_CASE(NL_BALL_BARY_APPROXCAPS);
    default: return nl_fail(ctx, NL_EINVAL, "unknown ball mode");
    }
#undef NL_CASE
}

}  // namespace

nl_status nl_launch_interior_batch_f32(nl_ctx *ctx, const nlq::NumArgs *dA, const nlq::BatchItem *items,
                                       int n_items, int *counter, int blocks)
{
    nlq::k_interior_batch<float><<<blocks, nlq::kWarpsPerBlock * 32, 0, ctx->stream>>>(dA, items, n_items, counter);
    ++ctx->launches;
    NL_CK(cudaGetLastError());
    return NL_OK;
}

nl_status nl_launch_boundary_batch_f32(nl_ctx *ctx, int ball, bool inv, const nlq::NumArgs *dA,
                                       const nlq::BatchItem *items, int n_items, int *counter, int blocks,
                                       bool set_attr)
{
    return boundary_ball(ctx, ball, inv, dA, items, n_items, counter, blocks, set_attr, nullptr);
}

nl_status nl_launch_deferred_batch_f32(nl_ctx *ctx, int ball, bool inv, const nlq::NumArgs *dA,
                                       const nlq::DeferItem *items, const int *count, int cap)
{
    int blocks = 0;
    nl_status s = nl_deferred_blocks(ctx, &blocks);
    if (s != NL_OK) return s;
    const unsigned threads = nlq::kWarpsPerBlock * 32;
    if (!inv) {   // the constant kernel queues the N-gon's items only
        nlq::k_deferred_batch<NL_BALL_NGON, false><<<blocks, threads, 0, ctx->stream>>>(dA, items, count, cap);
    } else {
#define NL_CASE(B) \
    case B: nlq::k_deferred_batch<B, true><<<blocks, threads, 0, ctx->stream>>>(dA, items, count, cap); break
        switch (ball) {
            NL_CASE(NL_BALL_BARYCENTER);
            NL_CASE(NL_BALL_NOCAPS);
            NL_CASE(NL_BALL_APPROXCAPS);
            NL_CASE(NL_BALL_EXACTCAPS);
            NL_CASE(NL_BALL_NGON);
            NL_CASE(NL_BALL_OVERLAP);
        default: return nl_fail(ctx, NL_EINVAL, "no deferred items for this ball mode");
        }
#undef NL_CASE
    }
    ++ctx->launches;
    nlq::k_defer_merge_batch<float><<<blocks, 256, 0, ctx->stream>>>(dA, items, count, cap); ++ctx->launches;
    NL_CK(cudaGetLastError());
    return NL_OK;
}

nl_status nl_batch_occupancy_f32(nl_ctx *ctx, int ball, bool inv, int *per_sm)
{
    if (ball < 0) {
        NL_CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, nlq::k_interior_batch<float>,
                                                            nlq::kWarpsPerBlock * 32, 0));
        return NL_OK;
    }
    return boundary_ball(ctx, ball, inv, nullptr, nullptr, 0, nullptr, 0, false, per_sm);
}
