// Inverse transforms: in place, out of place, and gathered from separate addresses.
#include "ntt_launch.cuh"

namespace {
__global__ void k_gather_res(const GatherSrc src, int npoly, u64 *dst, int logN) {
    const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= ((size_t)npoly << logN)) return;
    dst[e] = src.p[e >> logN][e & ((1ull << logN) - 1)];
}

}  // namespace

copse_status ntt_inverse(copse_ctx *ctx, const NttBatch &b, cudaStream_t s) { return launch_plain<true>(ctx, b, s); }

copse_status ntt_inverse_copy(copse_ctx *ctx, const u64 *src, size_t sstride, u64 *dst, size_t dstride, int npoly,
                              int nr, int fixed, cudaStream_t s, bool *done, const Shoup *scale) {
    NttBatch b{nullptr, 0, npoly, 0, nr, nr, fixed};
    b.scale = scale;
    b.digits = true;
    return launch_fused<true>(ctx, b, CopyIO{src, sstride, dst, dstride, ctx->logN}, s, done);
}

copse_status ntt_inverse_gather(copse_ctx *ctx, const GatherSrc &src, int npoly, u64 *dst, int fixed, cudaStream_t s,
                                bool *done, const Shoup *scale) {
    if (npoly > MS_POLYS) { set_error("internal: too many polynomials in one gathered transform"); return COPSE_EINVAL; }
    NttBatch b{nullptr, 0, npoly, 0, 1, 1, fixed};
    b.scale = scale;
    b.digits = true;
    STATUS_TRY(launch_fused<true>(ctx, b, GatherIO{src, dst, ctx->logN}, s, done));
    if (*done) return COPSE_OK;
    // a gather, then the in-place transform
    const size_t n = (size_t)npoly * ctx->N;
    k_gather_res<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(src, npoly, dst, ctx->logN);
    if (cudaGetLastError() != cudaSuccess) { set_error("gather kernel failed to launch"); return COPSE_ECUDA; }
    NttBatch bi{dst, (size_t)ctx->N, npoly, 0, 1, 1, fixed};
    bi.scale = scale;
    STATUS_TRY(ntt_inverse(ctx, bi, s));
    *done = true;
    return COPSE_OK;
}
