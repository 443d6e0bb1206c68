// Launching the transforms: which form a batch takes, and the timing families.
#pragma once

#include <atomic>

#include "ntt_core.cuh"

// one block per residue polynomial, in place, a stage per barrier (N <= 2^7; ntt.cu)
copse_status ntt_small(copse_ctx *ctx, const NttBatch &b, cudaStream_t s, bool inverse);

namespace {

// kernel-timer family of each transform variant
template <class IO> constexpr const char *io_family(bool inv) { return inv ? "ntt_inv" : "ntt_fwd"; }
template <> constexpr const char *io_family<CopyIO>(bool) { return "ntt_inv_copy"; }
template <> constexpr const char *io_family<GatherIO>(bool) { return "ntt_inv_copy"; }
template <> constexpr const char *io_family<MsIO>(bool) { return "ntt_fwd_ms"; }
template <> constexpr const char *io_family<MdIO>(bool) { return "ntt_fwd_md"; }
template <> constexpr const char *io_family<MuIO>(bool) { return "ntt_fwd_mu"; }
template <> constexpr const char *io_family<MddIO>(bool) { return "ntt_fwd_mdd"; }

// butterflies of a batch (N/2 log2 N per transformed residue polynomial): the integer
// roof's unit for the transforms
inline double butterflies(const copse_ctx *ctx, const NttBatch &b) {
    return (double)b.npoly * b.nr * (ctx->N / 2) * ctx->logN;
}

template <bool INV>
NttTables tables(const copse_ctx *c) {
    return NttTables{c->d_prime, (const ulonglong2 *)(INV ? c->d_tw_i : c->d_tw_f),
                     (const uint2 *)(INV ? c->d_twq_i : c->d_twq_f), (const ulonglong2 *)(INV ? c->d_low_i : c->d_low_f),
                     (const uint2 *)(INV ? c->d_lowq_i : c->d_lowq_f), c->L};
}

// A cluster kernel's shared memory, and the opt-in to 16-block clusters (N = 2^15, above the
// portable size): function attributes, raised once per kernel and device.  Threads that race
// here raise them twice, which is harmless.
template <int LOGN, class K>
copse_status cluster_attr(K kernel, int device, std::atomic<uint64_t> &done) {
    if (device >= 0 && device < 64 && (done.load(std::memory_order_acquire) & (1ull << device))) return COPSE_OK;
    CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(ClusterSmem<LOGN>)));
    if (LOGN == 15) CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    if (device >= 0 && device < 64) done.fetch_or(1ull << device, std::memory_order_release);
    return COPSE_OK;
}

template <int LOGN, bool INV, class IO>
copse_status launch_cluster(copse_ctx *ctx, const NttBatch &b, const IO &io, cudaStream_t s) {
    const unsigned grid = (unsigned)b.npoly * (unsigned)b.nr * Shape<LOGN>::TILES;
    const double bytes = (double)b.npoly * b.nr * ctx->N * 16.0;  // one read and one write of each residue polynomial
    const size_t smem = sizeof(ClusterSmem<LOGN>);
    static std::atomic<uint64_t> done{0};
    if constexpr (INV)
        STATUS_TRY(cluster_attr<LOGN>(k_ntt_inv_cluster<LOGN, IO>, ctx->device, done));
    else
        STATUS_TRY(cluster_attr<LOGN>(k_ntt_fwd_cluster<LOGN, IO>, ctx->device, done));
    TIMED_OPS(io_family<IO>(INV), bytes, butterflies(ctx, b), s, {
        if constexpr (INV)
            launch_dep(k_ntt_inv_cluster<LOGN, IO>, grid, NTHR, smem, s, b, tables<true>(ctx), io);
        else
            launch_dep(k_ntt_fwd_cluster<LOGN, IO>, grid, NTHR, smem, s, b, tables<false>(ctx), io);
    });
    LAUNCH_CHECK();
    return COPSE_OK;
}

// two launches; the partial transform in `mid`
template <int LOGN, bool INV, class IO>
copse_status launch_tiled(copse_ctx *ctx, const NttBatch &b, const IO &io, const Mid &mid, cudaStream_t s) {
    const unsigned grid = (unsigned)b.npoly * (unsigned)b.nr * Shape<LOGN>::TILES;
    const double bytes = (double)b.npoly * b.nr * ctx->N * 16.0;
    TIMED_OPS(io_family<IO>(INV), bytes, butterflies(ctx, b), s, {
        if constexpr (INV) {
            launch_dep(k_ntt_inv_rows<LOGN, IO>, grid, NTHR, 0, s, b, tables<true>(ctx), io, mid);
            launch_dep(k_ntt_inv_cols<LOGN, IO>, grid, NTHR, 0, s, b, tables<true>(ctx), io, mid);
        } else {
            launch_dep(k_ntt_fwd_cols<LOGN, IO>, grid, NTHR, 0, s, b, tables<false>(ctx), io, mid);
            launch_dep(k_ntt_fwd_rows<LOGN, IO>, grid, NTHR, 0, s, b, tables<false>(ctx), io, mid);
        }
    });
    LAUNCH_CHECK();
    return COPSE_OK;
}

template <int LOGN, bool INV, class IO>
copse_status launch_one(copse_ctx *ctx, const NttBatch &b, const IO &io, cudaStream_t s) {
    using O = One<LOGN>;
    const unsigned grid = ((unsigned)b.npoly * (unsigned)b.nr + O::PER - 1) / O::PER;
    const double bytes = (double)b.npoly * b.nr * ctx->N * 16.0;
    TIMED_OPS(io_family<IO>(INV), bytes, butterflies(ctx, b), s, {
        if constexpr (INV)
            launch_dep(k_ntt_inv_one<LOGN, IO>, grid, O::NT * O::PER, 0, s, b, tables<true>(ctx), io);
        else
            launch_dep(k_ntt_fwd_one<LOGN, IO>, grid, O::NT * O::PER, 0, s, b, tables<false>(ctx), io);
    });
    LAUNCH_CHECK();
    return COPSE_OK;
}

// A batch of b with this IO: clusters up to max_cluster residue polynomials (N = 2^15 only where
// 16-block clusters are opted in), else two launches through `data` (in place) or, when it is
// null, through scratch; where the device does not hold that scratch, clusters, which need none.
template <int LOGN, bool INV, class IO>
copse_status launch_ring(copse_ctx *ctx, const NttBatch &b, const IO &io, u64 *data, long max_cluster, cudaStream_t s) {
    const bool clusters = ctx->ntt_clusters && (LOGN < 15 || ctx->ntt_cluster16);
    if (clusters && (long)b.npoly * b.nr <= max_cluster) return launch_cluster<LOGN, INV, IO>(ctx, b, io, s);
    if (data) return launch_tiled<LOGN, INV, IO>(ctx, b, io, Mid{data, b.stride, 0}, s);
    u64 *scratch = nullptr;
    copse_status st = dev_alloc(ctx, (void **)&scratch, ((size_t)b.npoly * b.nr << LOGN) * sizeof(u64), s);
    if (st == COPSE_ENOMEM && clusters) return launch_cluster<LOGN, INV, IO>(ctx, b, io, s);
    STATUS_TRY(st);
    st = launch_tiled<LOGN, INV, IO>(ctx, b, io, Mid{scratch, (size_t)b.nr << LOGN, b.r0}, s);
    dev_free(scratch, s);
    return st;
}
template <bool INV, class IO>
copse_status launch_io(copse_ctx *ctx, const NttBatch &b, const IO &io, u64 *data, long max_cluster, cudaStream_t s) {
    switch (ctx->logN) {
        case 8: return launch_one<8, INV, IO>(ctx, b, io, s);
        case 9: return launch_one<9, INV, IO>(ctx, b, io, s);
        case 10: return launch_one<10, INV, IO>(ctx, b, io, s);
        case 11: return launch_one<11, INV, IO>(ctx, b, io, s);
        case 12: return launch_ring<12, INV, IO>(ctx, b, io, data, max_cluster, s);
        case 13: return launch_ring<13, INV, IO>(ctx, b, io, data, max_cluster, s);
        case 14: return launch_ring<14, INV, IO>(ctx, b, io, data, max_cluster, s);
        default: return launch_ring<15, INV, IO>(ctx, b, io, data, max_cluster, s);
    }
}

// in place
template <bool INV>
copse_status launch_plain(copse_ctx *ctx, const NttBatch &b, cudaStream_t s) {
    if (b.npoly <= 0 || b.nr <= 0) return COPSE_OK;
    if (ctx->logN < 8) return ntt_small(ctx, b, s, INV);
    return launch_io<INV>(ctx, b, PlainIO{b.data, b.stride, ctx->logN}, b.data, ctx->ntt_cluster_max, s);
}

// fused with the IO (*done = false, nothing launched, below 2^8 and with the fused forms off)
template <bool INV = false, class IO>
copse_status launch_fused(copse_ctx *ctx, const NttBatch &b, const IO &io, cudaStream_t s, bool *done) {
    *done = b.npoly <= 0 || b.nr <= 0;
    if (*done || !ntt_fuses(ctx)) return COPSE_OK;
    STATUS_TRY((launch_io<INV>(ctx, b, io, (u64 *)nullptr, ctx->ntt_fused_max, s)));
    *done = true;
    return COPSE_OK;
}

}  // namespace
