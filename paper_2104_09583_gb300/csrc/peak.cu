// Measured integer peaks of the modular arithmetic the kernels are built from:
// register-only microbenchmarks, timed with CUDA events, that give the
// denominators of the integer roofline (no spec-sheet rates).
//
//   kind 0  exact products in a lazily reduced sum: x y added to split-28 partial
//           sums (three 32 x 32 -> 64-bit multiply-adds per product), the form of
//           the key-switching, diagonal and encrypted-model dot products
//   kind 1  the forward butterfly of the transforms of N >= 2^12, by a constant
//           split twiddle (eight multiply instructions)
//   kind 2  Barrett products of two data residues (Handbook of Applied
//           Cryptography, Alg. 14.42), fully reduced
//   kind 3  the forward butterfly of the smaller transforms, by a constant exact
//           Shoup twiddle (Harvey 2014; ten multiply instructions)
//
// The butterflies are the kernels' own (bf_fwd), without a correction between
// them; their values wrap in these long chains, which the rate does not see.
// Every thread runs independent dependency chains so that issue, not latency,
// bounds the rate; the results are folded into one word per thread and stored,
// so nothing is dead code.  How many chains a kind takes is measured, the
// fastest of 2 to 16 (T/s): split butterflies 1.23 with two, 1.22 with four,
// 1.12 to 1.19 with more, where registers are allocated less well; exact ones
// 1.04 with two to eight; sums 2.15 with two, 2.52 with four, 2.71 with twelve
// (another card: 1.28, 1.08 and 2.85).
#include <algorithm>

#include "ntt_core.cuh"

namespace {

constexpr int MAC_CHAINS = 12, BF_CHAINS = 2, BARRETT_CHAINS = 8;
constexpr int PEAK_TPB = 256;

__global__ void __launch_bounds__(PEAK_TPB) k_peak_mac(int iters, u64 seed, u64 *sink) {
    const u64 t = (u64)blockIdx.x * blockDim.x + threadIdx.x;
    uint2 x[MAC_CHAINS];
    AccK a[MAC_CHAINS];
#pragma unroll
    for (int c = 0; c < MAC_CHAINS; c++) {
        x[c] = split_k((seed * (t + 1) + 0x9E3779B97F4A7C15ull * (c + 1)) & ((1ull << 55) - 1));
        a[c] = AccK{0, 0, 0};
    }
    u64 v = (seed ^ t) & ((1ull << 55) - 1);
    for (int i = 0; i < iters; i++) {
        v = (v + 0x00A3C59AC2F1ull) & ((1ull << 55) - 1);
        const uint2 y = split_k(v);
        const uint32_t ys = y.x + y.y;
#pragma unroll
        for (int c = 0; c < MAC_CHAINS; c++) mac_k(a[c], x[c], x[c].x + x[c].y, y, ys);
        // the partial sums hold 64 products exactly; lower them before that bound
        if ((i & 31) == 31) {
#pragma unroll
            for (int c = 0; c < MAC_CHAINS; c++) a[c] = AccK{a[c].lo >> 8, a[c].hi >> 8, a[c].s >> 8};
        }
    }
    u64 r = 0;
#pragma unroll
    for (int c = 0; c < MAC_CHAINS; c++) r ^= a[c].lo + a[c].hi + a[c].s;
    sink[t] = r;
}

// m: the twiddle's modulus (2q for split ones)
template <class TW>
__global__ void __launch_bounds__(PEAK_TPB) k_peak_butterfly(int iters, u64 m, TW w, u64 *sink) {
    const u64 t = (u64)blockIdx.x * blockDim.x + threadIdx.x;
    u64 x[BF_CHAINS], y[BF_CHAINS];
#pragma unroll
    for (int c = 0; c < BF_CHAINS; c++) {
        x[c] = (t + c + 1) * 0x9E3779B97F4A7C15ull >> 9;
        y[c] = (t + 3 * c) * 0xBF58476D1CE4E5B9ull >> 9;
    }
    for (int i = 0; i < iters; i++) {
#pragma unroll
        for (int c = 0; c < BF_CHAINS; c++) bf_fwd(x[c], y[c], w, m);
    }
    u64 r = 0;
#pragma unroll
    for (int c = 0; c < BF_CHAINS; c++) r ^= x[c] + y[c];
    sink[t] = r;
}

__global__ void __launch_bounds__(PEAK_TPB) k_peak_barrett(int iters, PrimeDev P, u64 *sink) {
    const u64 t = (u64)blockIdx.x * blockDim.x + threadIdx.x;
    u64 z[BARRETT_CHAINS], w[BARRETT_CHAINS];
#pragma unroll
    for (int c = 0; c < BARRETT_CHAINS; c++) {
        z[c] = (t * 0x9E3779B97F4A7C15ull + c + 1) % P.q;
        w[c] = (t * 0x94D049BB133111EBull + 7 * c + 2) % P.q;
    }
    for (int i = 0; i < iters; i++) {
#pragma unroll
        for (int c = 0; c < BARRETT_CHAINS; c++) z[c] = mul_mod(z[c], w[c], P);
    }
    u64 r = 0;
#pragma unroll
    for (int c = 0; c < BARRETT_CHAINS; c++) r ^= z[c];
    sink[t] = r;
}

}  // namespace

extern "C" copse_status copse_measure_int_peak(copse_ctx *c, int kind, int reps, double *ops_per_s, float *best_ms) {
    if (!c || !ops_per_s || kind < 0 || kind > 3 || reps < 1) { set_error("bad argument"); return COPSE_EINVAL; }
    int sms = 0;
    CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device));
    // eight resident CTAs of 256 threads per SM: enough warps to cover every pipe's latency
    const unsigned blocks = (unsigned)sms * 8;
    const size_t threads = (size_t)blocks * PEAK_TPB;
    const int chains = kind == 0 ? MAC_CHAINS : kind == 2 ? BARRETT_CHAINS : BF_CHAINS;
    const int iters = kind == 0 ? 4096 : (kind == 2 ? 1024 : 8192);
    u64 *sink = nullptr;
    CUDA_TRY(cudaMalloc(&sink, threads * sizeof(u64)));
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    const PrimeDev P = c->hprime[0];
    // a fixed twiddle modulo the first prime, as an exact pair and split (k_split_tw)
    const auto quot = [&](u64 v, int sh) { return (u64)(((unsigned __int128)v << sh) / P.q); };
    const u64 w = (P.q / 3) | 1, v = (u64)(((unsigned __int128)w << 31) % P.q);
    const ulonglong2 exact = make_ulonglong2(w, quot(w, 64));
    const Tw3 split{w, 2 * v, (uint32_t)quot(w, 31), (uint32_t)quot(v, 32)};
    float best = 1e30f;
    copse_status st = COPSE_OK;
    for (int r = 0; r <= reps && st == COPSE_OK; r++) {  // the first run warms up
        cudaEventRecord(e0, 0);
        if (kind == 0) k_peak_mac<<<blocks, PEAK_TPB>>>(iters, 0x1234567ull + r, sink);
        else if (kind == 1) k_peak_butterfly<<<blocks, PEAK_TPB>>>(iters, 2 * P.q, split, sink);
        else if (kind == 3) k_peak_butterfly<<<blocks, PEAK_TPB>>>(iters, P.q, exact, sink);
        else k_peak_barrett<<<blocks, PEAK_TPB>>>(iters, P, sink);
        cudaEventRecord(e1, 0);
        if (cudaEventSynchronize(e1) != cudaSuccess || cudaGetLastError() != cudaSuccess) {
            set_error("peak microbenchmark launch failed");
            st = COPSE_ECUDA;
            break;
        }
        float ms = 0;
        cudaEventElapsedTime(&ms, e0, e1);
        if (r > 0) best = std::min(best, ms);
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    cudaFree(sink);
    if (st != COPSE_OK) return st;
    *ops_per_s = (double)threads * iters * chains / (best * 1e-3);
    if (best_ms) *best_ms = best;
    return COPSE_OK;
}
