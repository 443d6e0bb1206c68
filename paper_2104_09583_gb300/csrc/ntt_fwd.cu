// Forward transforms: plain, and fused with a modulus switch.
#include "ntt_launch.cuh"

copse_status ntt_forward(copse_ctx *ctx, const NttBatch &b, cudaStream_t s) { return launch_plain<false>(ctx, b, s); }

copse_status ntt_forward_modswitch(copse_ctx *ctx, const MsFuse &f, int nc, cudaStream_t s, bool *done) {
    NttBatch b{nullptr, 0, nc, 0, f.ell - 1, f.ell - 1, -1};
    return launch_fused(ctx, b, MsIO{f, ctx->d_prime, ctx->ks, ctx->L, ctx->logN}, s, done);
}
