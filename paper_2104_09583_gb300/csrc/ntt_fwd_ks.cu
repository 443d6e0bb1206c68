// Forward transforms fused with the key switch's base conversions (ModUp, ModDown).
#include "ntt_launch.cuh"

copse_status ntt_forward_moddown(copse_ctx *ctx, const MdFuse &f, int njobs, cudaStream_t s, bool *done) {
    if (njobs > MD_JOBS) { set_error("internal: too many ModDown jobs"); return COPSE_EINVAL; }
    NttBatch b{nullptr, 0, 2 * njobs, 0, f.ell, f.ell, -1};
    return launch_fused(ctx, b, MdIO{f, ctx->d_prime, ctx->ks, ctx->L, ctx->alpha, ctx->logN}, s, done);
}

copse_status ntt_forward_modup(copse_ctx *ctx, const u64 *xc, const u64 *x_ntt, size_t xs, u64 *y, int n_items,
                               int ell, cudaStream_t s, bool *done) {
    const int A = ctx->alpha, nd = (ell + A - 1) / A;
    NttBatch b{nullptr, 0, n_items * nd, 0, ell + A, ell, -1};
    b.skip_alpha = A;
    b.skip_period = nd;
    return launch_fused(ctx, b, MuIO{xc, x_ntt, xs, y, ell, A, nd, ctx->L, ctx->NP, ctx->logN, ctx->d_prime, ctx->ks},
                        s, done);
}

copse_status ntt_forward_moddown_drop(copse_ctx *ctx, const MddFuse &f, int npoly, cudaStream_t s, bool *done) {
    NttBatch b{nullptr, 0, npoly, 0, f.ell - 1, f.ell - 1, -1};
    return launch_fused(ctx, b, MddIO{f, ctx->d_prime, ctx->ks, ctx->L, ctx->alpha, ctx->logN}, s, done);
}
