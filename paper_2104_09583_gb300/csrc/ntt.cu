// Negacyclic NTT over Z_q[X]/(X^N+1), batched over (polynomial, residue).
//
// Forward: Cooley-Tukey, natural coefficient order in, bit-reversed
// evaluation order out: position k holds a(psi^(2*brev(k)+1)).  Inverse:
// Gentleman-Sande back to coefficients, then N^-1.  Twiddles are psi^brev(k)
// (forward) and psi^-brev(k) (inverse) with Shoup quotients (the layout of
// Longa and Naehrig, "Speeding up the Number Theoretic Transform for Faster
// Ideal Lattice-Based Cryptography", CANS 2016).  Butterflies are lazy (Harvey
// 2014): no correction inside a pass, one reduction at its end, and outputs are
// exact residues in [0, q).
//
// Rings of N >= 2^12 run as N = N1 x N2, N1 rows of N2 contiguous coefficients: the first
// log2(N1) forward stages pair coefficients of one column, the others of one row
// (ntt_core.cuh; the launches in ntt_launch.cuh, ntt_fwd.cu, ntt_fwd_ks.cu and ntt_inv.cu).
// Smaller rings use one block per polynomial (below 2^8: here).
#include <cstdlib>

#include "ntt_launch.cuh"

namespace {

// inverse butterfly, values in [0, 2q)
__device__ __forceinline__ void bf_inv_small(u64 &x, u64 &y, u64 w, u64 wp, u64 q, u64 q2) {
    const u64 U = x, V = y;
    u64 s = U + V;
    if (s >= q2) s -= q2;
    x = s;
    y = mul_shoup_lazy(U - V + q2, w, wp, q);
}

// ---------------------------------------------------------------- one CTA per polynomial
__global__ void __launch_bounds__(512) k_ntt_fwd(NttBatch b, const PrimeDev *__restrict__ primes,
                                                 const u64 *__restrict__ tw, const u64 *__restrict__ tw_sh,
                                                 int logN, int L) {
    extern __shared__ u64 sm[];
    const int N = 1 << logN, half = N >> 1;
    const int p = blockIdx.x / b.nr, r = b.r0 + blockIdx.x % b.nr;
    if (ntt_skipped(b, p, r)) return;
    const int g = ntt_prime(b, r, L);
    const PrimeDev P = primes[g];
    const u64 q = P.q;
    u64 *data = b.data + (size_t)p * b.stride + (size_t)r * N;
    const u64 *W = tw + (size_t)g * N, *Wp = tw_sh + (size_t)g * N;
    for (int i = threadIdx.x; i < N; i += blockDim.x) sm[i] = data[i];
    __syncthreads();
    for (int m = 1, lt = logN - 1; m < N; m <<= 1, lt--) {
        const int tt = 1 << lt;
        for (int x = threadIdx.x; x < half; x += blockDim.x) {
            const int i = x >> lt, j = x & (tt - 1);
            const int idx = (i << (lt + 1)) + j;
            bf_fwd(sm[idx], sm[idx + tt], make_ulonglong2(W[m + i], Wp[m + i]), q);
        }
        __syncthreads();
    }
    for (int i = threadIdx.x; i < N; i += blockDim.x) {
        u64 v = sm[i];
        data[i] = fwd_reduce(v, P);
    }
}

__global__ void __launch_bounds__(512) k_ntt_inv(NttBatch b, const PrimeDev *__restrict__ primes,
                                                 const u64 *__restrict__ tw, const u64 *__restrict__ tw_sh,
                                                 int logN, int L) {
    extern __shared__ u64 sm[];
    const int N = 1 << logN, half = N >> 1;
    const int p = blockIdx.x / b.nr, r = b.r0 + blockIdx.x % b.nr;
    if (ntt_skipped(b, p, r)) return;
    const int g = ntt_prime(b, r, L);
    const PrimeDev P = primes[g];
    const u64 q = P.q, q2 = 2 * q;
    u64 *data = b.data + (size_t)p * b.stride + (size_t)r * N;
    const u64 *W = tw + (size_t)g * N, *Wp = tw_sh + (size_t)g * N;
    for (int i = threadIdx.x; i < N; i += blockDim.x) sm[i] = data[i];
    __syncthreads();
    for (int m = N, lt = 0; m > 1; m >>= 1, lt++) {
        const int tt = 1 << lt, h = m >> 1;
        for (int x = threadIdx.x; x < half; x += blockDim.x) {
            const int i = x >> lt, j = x & (tt - 1);
            const int idx = (i << (lt + 1)) + j;
            bf_inv_small(sm[idx], sm[idx + tt], W[h + i], Wp[h + i], q, q2);
        }
        __syncthreads();
    }
    const Shoup sc = b.scale ? b.scale[r - b.r0] : Shoup{P.ninv, P.ninv_sh};
    for (int i = threadIdx.x; i < N; i += blockDim.x) data[i] = mul_shoup(sm[i], sc, q);
}

__global__ void k_ms_finish_io(const MsFuse f, const u64 *W, int nc, const PrimeDev *pr, KsTables T, int L,
                               int logN) {
    const size_t per = (size_t)(f.ell - 1) << logN;
    const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (size_t)nc * per) return;
    const int p = (int)(e / per);
    const size_t rem = e - p * per;
    ms_store(f, pr, T, L, logN, p, (int)(rem >> logN), rem & ((1ull << logN) - 1), W[e]);
}

__global__ void k_mdd_conv(const MddFuse f, u64 *W, int npoly, const PrimeDev *pr, KsTables T, int L, int alpha,
                           int logN) {
    const size_t per = (size_t)(f.ell - 1) << logN;
    const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (size_t)npoly * per) return;
    const int p = (int)(e / per);
    const size_t rem = e - p * per;
    W[e] = mdd_load(f, pr, T, L, alpha, logN, p, (int)(rem >> logN), rem & ((1ull << logN) - 1));
}

__global__ void k_mdd_finish(const MddFuse f, const u64 *W, int npoly, const PrimeDev *pr, KsTables T, int L,
                             int logN) {
    const size_t per = (size_t)(f.ell - 1) << logN;
    const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (size_t)npoly * per) return;
    const int p = (int)(e / per);
    const size_t rem = e - p * per;
    mdd_store(f, pr, T, L, logN, p, (int)(rem >> logN), rem & ((1ull << logN) - 1), W[e]);
}

__global__ void k_md_finish_io(const MdFuse f, const u64 *W, int njobs, const PrimeDev *pr, KsTables T, int logN) {
    const size_t per = (size_t)f.ell << logN;
    const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (size_t)2 * njobs * per) return;
    const int p = (int)(e / per);
    const size_t rem = e - p * per;
    md_store(f, pr, T, logN, p, (int)(rem >> logN), rem & ((1ull << logN) - 1), W[e]);
}


// The tables of ntt_core.cuh: (w, w') pairs in natural order, or the split twiddles (2^31 w mod q
// and the two quotients follow from the Shoup quotient w' = floor(w 2^64 / q): floor(w 2^31 / q) is
// its upper 31 bits and floor((2^31 w mod q) 2^32 / q) the 32 below), and the low row stages'
// twiddles (pairs of modulus 2q, or split) in thread order: forward stage s of thread t takes 16 >> (K - s) pairs of
// transform stage A + 4 + s from coefficient 16 t of its tile on, inverse stage s takes 8 >> s
// pairs of distance 2^s (K = LB - 4 low stages).
constexpr long CLUSTER_BLOCKS = 400;
__global__ void k_pairs(const u64 *W, const u64 *Wp, ulonglong2 *out, size_t n) {
    const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e < n) out[e] = make_ulonglong2(W[e], Wp[e]);
}
__device__ __forceinline__ void split_tw(u64 w, u64 wp, u64 q, ulonglong2 *out, uint2 *outq) {
    *out = make_ulonglong2(w, 2 * mul_shoup(1ull << 31, w, wp, q));
    *outq = make_uint2((uint32_t)(wp >> 33), (uint32_t)(wp >> 1));
}
__global__ void k_split_tw(const u64 *W, const u64 *Wp, ulonglong2 *out, uint2 *outq, size_t n, int logN,
                           const PrimeDev *pr) {
    const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e < n) split_tw(W[e], Wp[e], pr[e >> logN].q, out + e, outq + e);
}
__global__ void k_low_tw(const u64 *W, const u64 *Wp, ulonglong2 *out, uint2 *outq, int np, int logN, int pairs, int inverse,
                         const PrimeDev *pr) {
    const int tiles = 1 << (logN - 11), K = logN - logN / 2 - 4;
    const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (size_t)np * tiles * pairs * NTHR) return;
    const int t = (int)(e % NTHR);
    int k = (int)(e / NTHR % pairs);
    const int tile = (int)(e / NTHR / pairs % tiles), g = (int)(e / NTHR / pairs / tiles);
    const int pos = tile * TILE + 16 * t;
    int s = 0;
    for (; k >= (inverse ? 8 >> s : 16 >> (K - s)); s++) k -= inverse ? 8 >> s : 16 >> (K - s);
    const int U = inverse ? logN - 1 - s : logN - K + s;  // transform stage: 2^U groups
    const size_t at = ((size_t)g << logN) + (1 << U) + (pos >> (logN - U)) + k;
    if (outq) split_tw(W[at], Wp[at], pr[g].q, out + e, outq + e);
    else out[e] = make_ulonglong2(W[at], Wp[at] >> 1);
}

}  // namespace

copse_status ntt_small(copse_ctx *ctx, const NttBatch &b, cudaStream_t s, bool inverse) {
    const int N = ctx->N, logN = ctx->logN;
    const double bytes = (double)b.npoly * b.nr * N * 16.0;
    const double bfly = butterflies(ctx, b);
    const size_t smem = (size_t)N * sizeof(u64);
    const int threads = N / 2 < 512 ? N / 2 : 512;
    const unsigned grid = (unsigned)b.npoly * (unsigned)b.nr;
    if (inverse)
        TIMED_OPS("ntt_inv", bytes, bfly, s,
              k_ntt_inv<<<grid, threads, smem, s>>>(b, ctx->d_prime, ctx->d_ipsi, ctx->d_ipsi_sh, logN, ctx->L));
    else
        TIMED_OPS("ntt_fwd", bytes, bfly, s,
              k_ntt_fwd<<<grid, threads, smem, s>>>(b, ctx->d_prime, ctx->d_psi, ctx->d_psi_sh, logN, ctx->L));
    LAUNCH_CHECK();
    return COPSE_OK;
}

copse_status ntt_stage_tables(copse_ctx *ctx) {
    if (ctx->logN < 8) return COPSE_OK;
    if (ctx->logN == 15) {
        // 16-block clusters are above the portable size: an option (COPSE_NTT_CLUSTER16=1) where
        // the device can place at least one
        std::atomic<uint64_t> none{0};
        STATUS_TRY(cluster_attr<15>(k_ntt_fwd_cluster<15, PlainIO>, -1, none));
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3(16);
        cfg.blockDim = dim3(NTHR);
        cfg.dynamicSmemBytes = sizeof(ClusterSmem<15>);
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = 16;
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        int nclusters = 0;
        const cudaError_t e = cudaOccupancyMaxActiveClusters(&nclusters, k_ntt_fwd_cluster<15, PlainIO>, &cfg);
        const char *opt = getenv("COPSE_NTT_CLUSTER16");
        ctx->ntt_cluster16 = e == cudaSuccess && nclusters > 0 && opt && opt[0] == '1';
        cudaGetLastError();
    }
    // Clusters up to about the blocks that fit the GPU at once (three of a cluster kernel's blocks
    // per SM), two launches above; the tuner or the caller may set other crossovers.  Measured at
    // N = 2^14 (us a forward transform in a graph, clusters / tiled): 16 residue polynomials
    // 8.7 / 8.0, 32: 9.2 / 9.6, 48: 11.6 / 11.6, 64: 20.2 / 14.3, 128: 29.8 / 21.8; whole
    // inferences are flat between 300 and 400 blocks.
    if (ctx->logN >= 12 && ctx->logN < 15) ctx->ntt_cluster_max = ctx->ntt_fused_max = CLUSTER_BLOCKS >> (ctx->logN - 11);
    // one block per transform below 2^12: no low row stages
    const int lb = ctx->logN - ctx->logN / 2, pairs = lb == 8 ? 15 : (lb == 7 ? 14 : 12);
    const size_t n = (size_t)ctx->NP * ctx->N;
    const size_t nl = ctx->logN < 12 ? 0 : (size_t)ctx->NP * (ctx->N / TILE) * pairs * NTHR;
    for (int inv = 0; inv < 2; inv++) {
        void *p = nullptr, *l = nullptr;
        CUDA_TRY(cudaMalloc(&p, n * sizeof(ulonglong2)));
        ctx->owned.push_back(p);
        const u64 *W = inv ? ctx->d_ipsi : ctx->d_psi, *Wp = inv ? ctx->d_ipsi_sh : ctx->d_psi_sh;
        (inv ? ctx->d_tw_i : ctx->d_tw_f) = (u64 *)p;
        if (!nl) {
            k_pairs<<<(unsigned)((n + 255) / 256), 256>>>(W, Wp, (ulonglong2 *)p, n);
            CUDA_TRY(cudaGetLastError());
            continue;
        }
        void *pq = nullptr;
        CUDA_TRY(cudaMalloc(&pq, n * sizeof(uint2)));
        ctx->owned.push_back(pq);
        (inv ? ctx->d_twq_i : ctx->d_twq_f) = (u64 *)pq;
        k_split_tw<<<(unsigned)((n + 255) / 256), 256>>>(W, Wp, (ulonglong2 *)p, (uint2 *)pq, n, ctx->logN, ctx->d_prime);
        CUDA_TRY(cudaGetLastError());
        CUDA_TRY(cudaMalloc(&l, nl * sizeof(ulonglong2)));
        ctx->owned.push_back(l);
        void *lq = nullptr;
        if (lb == 8) {
            CUDA_TRY(cudaMalloc(&lq, nl * sizeof(uint2)));
            ctx->owned.push_back(lq);
        }
        k_low_tw<<<(unsigned)((nl + 255) / 256), 256>>>(W, Wp, (ulonglong2 *)l, (uint2 *)lq, ctx->NP, ctx->logN, pairs,
                                                        inv, ctx->d_prime);
        CUDA_TRY(cudaGetLastError());
        (inv ? ctx->d_low_i : ctx->d_low_f) = (u64 *)l;
        (inv ? ctx->d_lowq_i : ctx->d_lowq_f) = (u64 *)lq;
    }
    CUDA_TRY(cudaDeviceSynchronize());
    return COPSE_OK;
}

copse_status moddown_drop_unfused(copse_ctx *ctx, const MddFuse &f, int npoly, cudaStream_t s) {
    const size_t n = (size_t)npoly * (f.ell - 1) * ctx->N;
    u64 *W = nullptr;
    STATUS_TRY(dev_alloc(ctx, (void **)&W, n * sizeof(u64), s));
    const unsigned g = (unsigned)((n + 255) / 256);
    TIMED("moddown_conv", 8.0 * (double)n * (ctx->alpha + 2), s,
          k_mdd_conv<<<g, 256, 0, s>>>(f, W, npoly, ctx->d_prime, ctx->ks, ctx->L, ctx->alpha, ctx->logN));
    copse_status st = cudaGetLastError() == cudaSuccess ? COPSE_OK : COPSE_ECUDA;
    if (st == COPSE_OK) st = ntt_forward(ctx, NttBatch{W, (size_t)(f.ell - 1) * ctx->N, npoly, 0, f.ell - 1, f.ell - 1, -1}, s);
    if (st == COPSE_OK) {
        TIMED("ks_finish", 8.0 * 3.0 * (double)n, s,
              k_mdd_finish<<<g, 256, 0, s>>>(f, W, npoly, ctx->d_prime, ctx->ks, ctx->L, ctx->logN));
        if (cudaGetLastError() != cudaSuccess) st = COPSE_ECUDA;
    }
    dev_free(W, s);
    if (st != COPSE_OK && st != COPSE_ECUDA) return st;
    if (st == COPSE_ECUDA) set_error("moddown-drop kernels failed to launch");
    return st;
}

copse_status modswitch_finish(copse_ctx *ctx, const MsFuse &f, const u64 *W, int nc, cudaStream_t s) {
    const size_t n = (size_t)nc * (f.ell - 1) * ctx->N;
    TIMED("ms_finish", 8.0 * 3.0 * (double)n, s,
          k_ms_finish_io<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(f, W, nc, ctx->d_prime, ctx->ks, ctx->L,
                                                                      ctx->logN));
    LAUNCH_CHECK();
    return COPSE_OK;
}

copse_status moddown_finish(copse_ctx *ctx, const MdFuse &f, const u64 *W, int njobs, cudaStream_t s) {
    if (njobs > MD_JOBS) { set_error("internal: too many ModDown jobs"); return COPSE_EINVAL; }
    const size_t n = (size_t)2 * njobs * f.ell * ctx->N;
    TIMED("ks_finish", 8.0 * 4.0 * (double)n, s,
          k_md_finish_io<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(f, W, njobs, ctx->d_prime, ctx->ks, ctx->logN));
    LAUNCH_CHECK();
    return COPSE_OK;
}
