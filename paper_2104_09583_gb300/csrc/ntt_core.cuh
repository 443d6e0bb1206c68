// The transform kernels.  For 2^12 <= N <= 2^15: N = 2^A rows of 2^LB coefficients, the first A
// forward stages over columns, the last LB over rows, the inverse the other way round (the
// stage order, twiddle order and lazy ranges are stated in ntt.cu).
//
// A tile is 2048 coefficients (columns x all rows, or rows x all columns) and a block of 128
// threads holds one in registers, 16 coefficients a thread: four stages in registers, one
// exchange through shared memory, the remaining two to four stages in registers.  What bounds a
// large batch is the integer multiplier (a butterfly is a 64-bit Shoup product), so the layout
// spends as little else as it can: an 8-stage pass has one exchange instead of one per two or
// three stages, and no index arithmetic between the stages.  Twiddles are read as (w, w') pairs
// straight from global memory: those of a tile's top stages are shared by the threads of a
// sequence, those of the low stages, one per butterfly, are stored in thread order
// ([tile][pair][thread]), so that every load of a warp is contiguous.
//
// Two forms share this code.  Tiled: a column launch and a row launch with the partial transform
// in global memory between them, any batch size.  Cluster: N / 2048 blocks of a thread-block
// cluster own one residue polynomial and hand the tiles over through distributed shared memory,
// each thread writing its 16 outputs of the first half into the blocks that take them on: one
// launch, for batches too small to fill the GPU (one residue polynomial at N = 2^14: 7.1 us in a
// graph, 7.9 with 512 threads and four coefficients a thread).
//
// Measured (us, forward / inverse; before = a radix-4 / radix-8 pass per two or three stages with
// 512 / 256 threads and every twiddle staged through shared memory): N = 2^15, 1024 residue
// polynomials 616 / 644 before, 331 / 359 now (0.76 / 0.70 T butterflies/s of the 0.95 that the
// multiplier alone reaches), 64: 43 / 47 before, 29 / 31 now; N = 2^14, 1024 in clusters
// 269 / 313 before, 163 / 178 tiled now.
#pragma once

#include <cooperative_groups.h>

#include "ntt_io.cuh"

namespace {

namespace cg = cooperative_groups;

constexpr int TILE = 2048;      // coefficients per block
constexpr int NTHR = TILE / 16; // threads per block

template <int LOGN>
struct Shape {
    static constexpr int A = LOGN / 2, LB = LOGN - A;         // stages over columns, over rows
    static constexpr int LC = 11 - A, C = 1 << LC;            // columns of a column tile
    static constexpr int LR = 11 - LB, R = 1 << LR;           // rows of a row tile
    static constexpr int TILES = 1 << (LOGN - 11);
    static constexpr int SA = 1 << (A - 4), SB = 1 << (LB - 4);  // threads per column, per row
    static constexpr int PAIRS = LB == 8 ? 15 : (LB == 7 ? 14 : 12);  // low row twiddles of a thread
};

__device__ __forceinline__ int ntt_prime(const NttBatch &b, int r, int L) {
    return b.fixed >= 0 ? b.fixed : (r < b.ell ? r : L + (r - b.ell));
}

// residue r of poly p is excluded from this batch (a ModUp digit's own primes)
__device__ __forceinline__ bool ntt_skipped(const NttBatch &b, int p, int r) {
    const int j = b.skip_period > 0 ? p % b.skip_period : p;
    return b.skip_alpha > 0 && r >= j * b.skip_alpha && r < min((j + 1) * b.skip_alpha, b.ell);
}

// Forward butterfly without a correction step: the Shoup product V is below 2q for any
// 64-bit input, so x' = U + V and y' = U - V + 2q only grow by 2q per stage.  From inputs
// below 2q, values stay below (2 log2 N + 2) q <= 32 q <= 2^60 for primes below 2^55 (the
// context's limit); the final store reduces them once.
__device__ __forceinline__ void bf_fwd(u64 &x, u64 &y, ulonglong2 w, u64 q, u64 q2) {
    const u64 U = x;
    const u64 V = mul_shoup_lazy(y, w.x, w.y, q);
    x = U + V;
    y = U - V + q2;
}

// Inverse butterfly without a correction step, for a stage whose inputs are below c (a
// multiple of q): U - V + c is positive and below 2c, so the product is the same residue,
// x' = U + V < 2c and y' < 2q.  From inputs below c0 (q or 2q), stage u of a pass takes
// c = 2^u c0; a pass of at most 8 stages from q, or 7 from 2q, stays below 2^63 for primes below
// 2^55 (the context's limit) and is reduced once before the next pass or the scaling.
__device__ __forceinline__ void bf_inv(u64 &x, u64 &y, ulonglong2 w, u64 q, u64 c) {
    const u64 U = x, V = y;
    x = U + V;
    y = mul_shoup_lazy(U - V + c, w.x, w.y, q);
}

// a transform's lazy value reduced to [0, q)
__device__ __forceinline__ u64 fwd_reduce(u64 v, const PrimeDev &P) {
    const u64 r = reduce64_lazy(v, P);
    return r >= P.q ? r - P.q : r;
}

// K forward stages (distances 2^(K-1), .., 1 within groups of 2^K) on 16 registers;
// tw(s, il): the pair of stage s, group il < 16 >> (K - s)
template <int K, class TW>
__device__ __forceinline__ void stages_fwd(u64 (&v)[16], u64 q, u64 q2, TW tw) {
#pragma unroll
    for (int s = 0; s < K; s++) {
        const int ld = K - 1 - s, d = 1 << ld;
        ulonglong2 w;
#pragma unroll
        for (int x = 0; x < 8; x++) {
            const int il = x >> ld, j = x & (d - 1);
            if (j == 0) w = tw(s, il);
            bf_fwd(v[2 * d * il + j], v[2 * d * il + d + j], w, q, q2);
        }
    }
}
// K inverse stages (distances 1, .., 2^(K-1)); inputs below c0; tw(s, il): il < 8 >> s
template <int K, class TW>
__device__ __forceinline__ void stages_inv(u64 (&v)[16], u64 q, u64 c0, TW tw) {
#pragma unroll
    for (int s = 0; s < K; s++) {
        const int d = 1 << s;
        ulonglong2 w;
#pragma unroll
        for (int x = 0; x < 8; x++) {
            const int il = x >> s, j = x & (d - 1);
            if (j == 0) w = tw(s, il);
            bf_inv(v[2 * d * il + j], v[2 * d * il + d + j], w, q, c0 << s);
        }
    }
}

// a twiddle pair from global memory, or (SH) from the block's copy in shared memory
template <bool SH>
__device__ __forceinline__ ulonglong2 pair_at(const ulonglong2 *p) {
    if constexpr (SH) return *p;
    else return __ldg(p);
}
// Row tiles keep coefficient f of the tile at word f + f / 16 of shared memory: 16 threads that
// read 16 consecutive coefficients each hit different banks, as do 16 that read a run.
constexpr int PTILE = TILE + TILE / 16;
__device__ __forceinline__ int pad(int f) { return f + (f >> 4); }

// twiddles of the passes (T: the prime's pairs in natural order, low: this tile's low row pairs
// of this thread, [pair][thread]); the column stages use the first 2^A pairs only
//
// forward column stages 0..3: the whole transform's first 15 twiddles
template <bool SH>
struct TwColTop {
    const ulonglong2 *T;
    __device__ __forceinline__ ulonglong2 operator()(int s, int il) const { return pair_at<SH>(T + (1 << s) + il); }
};
// forward column stages 4..A-1 of rows 16 b ..
template <int A, bool SH>
struct TwColLow {
    const ulonglong2 *T;
    int b;
    __device__ __forceinline__ ulonglong2 operator()(int s, int il) const {
        return pair_at<SH>(T + (1 << (4 + s)) + ((16 * b) >> (A - 4 - s)) + il);
    }
};
// forward row stages 0..3 of one row
template <int A>
struct TwRowTop {
    const ulonglong2 *T;
    int row;
    __device__ __forceinline__ ulonglong2 operator()(int s, int il) const {
        return pair_at<false>(T + (1 << (A + s)) + (row << s) + il);
    }
};
// the same, and the last four inverse row stages, from a copy of the 15 pairs of each of a tile's
// R rows, those of 2^u groups per row at R (2^u - 1) (gr: the row within the tile)
template <int R, bool INV>
struct TwRowTopSh {
    const ulonglong2 *W;
    int gr;
    __device__ __forceinline__ ulonglong2 operator()(int s, int il) const {
        const int u = INV ? 3 - s : s;
        return W[R * ((1 << u) - 1) + (gr << u) + il];
    }
};
// low row stages in thread order: the pairs of stage s follow those of the stages before
template <int K, bool INV, bool SH>
struct TwRowLow {
    const ulonglong2 *low;
    __device__ __forceinline__ ulonglong2 operator()(int s, int il) const {
        const int off = INV ? 16 - (16 >> s) : (16 >> (K - s)) - (16 >> K);
        return pair_at<SH>(low + (off + il) * NTHR);
    }
};
// inverse column stages of distance 2^s rows, rows 16 b ..
template <int A, bool SH>
struct TwInvColLow {
    const ulonglong2 *T;
    int b;
    __device__ __forceinline__ ulonglong2 operator()(int s, int il) const {
        return pair_at<SH>(T + (1 << (A - 1 - s)) + ((16 * b) >> (s + 1)) + il);
    }
};
// the last four inverse column stages
template <bool SH>
struct TwInvColTop {
    const ulonglong2 *T;
    __device__ __forceinline__ ulonglong2 operator()(int s, int il) const { return pair_at<SH>(T + (1 << (3 - s)) + il); }
};
// the last four inverse row stages of one row
template <int A>
struct TwInvRowTop {
    const ulonglong2 *T;
    int row;
    __device__ __forceinline__ ulonglong2 operator()(int s, int il) const {
        return pair_at<false>(T + (1 << (A + 3 - s)) + (row << (3 - s)) + il);
    }
};

// ---------------------------------------------------------------- the halves of a transform
// Forward column half: the tile's coefficients through io (KL at a time), all A column stages;
// the thread ends with rows 16 b .. 16 b + 15 of its column.  SH: the first 2^A pairs at T are
// the block's copy, complete after `arrived`.
template <int LOGN, int KL, bool SH, class IO, class ARR>
__device__ __forceinline__ void fwd_cols(const IO &io, int p, int r, int g, int tile, const ulonglong2 *T, u64 q,
                                         u64 *sm, u64 (&v)[16], ARR arrived) {
    using S = Shape<LOGN>;
    const int t = threadIdx.x, c = t & (S::C - 1), i = t >> S::LC;
    const size_t n0 = ((size_t)i << S::LB) + (tile << S::LC) + c, dn = (size_t)S::SA << S::LB;
#pragma unroll
    for (int h = 0; h < 16 / KL; h++) {
        u64 x[KL];
        load_n(io, p, r, g, n0 + KL * h * dn, dn, x);
#pragma unroll
        for (int m = 0; m < KL; m++) v[KL * h + m] = x[m];
    }
    arrived();
    stages_fwd<4>(v, q, 2 * q, TwColTop<SH>{T});
#pragma unroll
    for (int m = 0; m < 16; m++) sm[((i + m * S::SA) << S::LC) + c] = v[m];
    __syncthreads();
#pragma unroll
    for (int m = 0; m < 16; m++) v[m] = sm[((16 * i + m) << S::LC) + c];
    stages_fwd<S::A - 4>(v, q, 2 * q, TwColLow<S::A, SH>{T, i});
}

// Forward row half: v holds coefficients i + m SB of the thread's row (i = t mod SB); all LB row
// stages, the values stored through io (reduced unless it takes them raw).  u: the finishes'
// operands where they are loaded ahead (EARLY), in the order of the stores.
template <int LOGN, bool EARLY, class IO, class TOP, class LOW>
__device__ __forceinline__ void fwd_rows(const IO &io, int p, int r, int g, int tile, TOP top, LOW low,
                                         const PrimeDev &P, u64 *sm, u64 (&v)[16]) {
    using S = Shape<LOGN>;
    const int t = threadIdx.x, i = t & (S::SB - 1), gr = t / S::SB;
    const u64 q = P.q;
    const int f0 = (t & ~31) * 16 + (t & 31);
    const size_t k0 = ((size_t)tile << 11) + f0;
    u64 u[4][4];
    if (EARLY) {
#pragma unroll
        for (int h = 0; h < 4; h++) operand_n(io, p, r, k0 + 128 * h, 32, u[h]);
    }
    stages_fwd<4>(v, q, 2 * q, top);
#pragma unroll
    for (int m = 0; m < 16; m++) sm[pad((gr << S::LB) + i + m * S::SB)] = v[m];
    __syncthreads();
#pragma unroll
    for (int m = 0; m < 16; m++) v[m] = sm[pad(16 * t + m)];
    stages_fwd<S::LB - 4>(v, q, 2 * q, low);
    // to runs of 32 coefficients per warp access, within the warp's 512
#pragma unroll
    for (int m = 0; m < 16; m++) sm[pad(16 * t + m)] = v[m];
    __syncwarp();
#pragma unroll
    for (int h = 0; h < 4; h++) {
        u64 x[4];
        if (!EARLY) operand_n(io, p, r, k0 + 128 * h, 32, u[h]);
#pragma unroll
        for (int m = 0; m < 4; m++) {
            x[m] = sm[pad(f0 + 32 * (4 * h + m))];
            if (!IO::RAW) x[m] = fwd_reduce(x[m], P);
        }
        store_n(io, p, r, g, k0 + 128 * h, 32, x, u[h]);
    }
}

// Inverse row half: the tile through io.load, all LB row stages; the thread ends with
// coefficients i + m SB of its row, reduced below 2q.  `arrived`: the twiddles' copies complete.
template <int LOGN, class IO, class TOP, class LOW, class ARR>
__device__ __forceinline__ void inv_rows(const IO &io, int p, int r, int g, int tile, TOP top, LOW low,
                                         const PrimeDev &P, u64 *sm, u64 (&v)[16], ARR arrived) {
    using S = Shape<LOGN>;
    const int t = threadIdx.x, i = t & (S::SB - 1), gr = t / S::SB;
    const u64 q = P.q;
    const int f0 = (t & ~31) * 16 + (t & 31);
#pragma unroll
    for (int m = 0; m < 16; m++) v[m] = io.load(p, r, g, ((size_t)tile << 11) + f0 + 32 * m);
#pragma unroll
    for (int m = 0; m < 16; m++) sm[pad(f0 + 32 * m)] = v[m];
    arrived();
    __syncwarp();
#pragma unroll
    for (int m = 0; m < 16; m++) v[m] = sm[pad(16 * t + m)];
    stages_inv<S::LB - 4>(v, q, q, low);
#pragma unroll
    for (int m = 0; m < 16; m++) sm[pad(16 * t + m)] = v[m];
    __syncthreads();
#pragma unroll
    for (int m = 0; m < 16; m++) v[m] = sm[pad((gr << S::LB) + i + m * S::SB)];
    stages_inv<4>(v, q, q << (S::LB - 4), top);
#pragma unroll
    for (int m = 0; m < 16; m++) v[m] = reduce64_lazy(v[m], P);
}

// an inverse transform's result: scaled, and stored as a conversion's digit where asked (centred,
// offset by (q - 1) / 2, split at 28 bits)
__device__ __forceinline__ u64 inv_result(u64 v, Shoup sc, bool digits, u64 q) {
    u64 x = mul_shoup(v, sc, q);
    if (digits) {
        x = add_mod(x, (q - 1) / 2, q);
        x = ((x >> 28) << 32) | (x & 0x0FFFFFFFu);
    }
    return x;
}

// Inverse column half: v holds rows 16 b .. 16 b + 15 of the thread's column (below 2q); all A
// column stages, scaled and stored through io.
template <int LOGN, bool SH, class IO>
__device__ __forceinline__ void inv_cols(const IO &io, int p, int r, int g, int tile, const ulonglong2 *T, Shoup sc,
                                         bool digits, u64 q, u64 *sm, u64 (&v)[16]) {
    using S = Shape<LOGN>;
    const int t = threadIdx.x, c = t & (S::C - 1), i = t >> S::LC;
    stages_inv<S::A - 4>(v, q, 2 * q, TwInvColLow<S::A, SH>{T, i});
#pragma unroll
    for (int m = 0; m < 16; m++) sm[((16 * i + m) << S::LC) + c] = v[m];
    __syncthreads();
#pragma unroll
    for (int m = 0; m < 16; m++) v[m] = sm[((i + m * S::SA) << S::LC) + c];
    stages_inv<4>(v, q, (2 * q) << (S::A - 4), TwInvColTop<SH>{T});
#pragma unroll
    for (int m = 0; m < 16; m++)
        io.store(p, r, g, ((size_t)(i + m * S::SA) << S::LB) + (tile << S::LC) + c, inv_result(v[m], sc, digits, q));
}

// ---------------------------------------------------------------- tiled: two launches
// The partial transform between the launches: residue r of polynomial p at
// base + p ps + (r - r0) N (the data itself for an in-place transform, else scratch).
struct Mid {
    u64 *base;
    size_t ps;
    int r0;
};
// the block's polynomial, residue, prime and tile
struct TileAt {
    int p, r, g, tile;
};
__device__ __forceinline__ TileAt tile_at(const NttBatch &b, int L, int tiles) {
    TileAt t;
    const int pr = blockIdx.x / tiles;
    t.tile = blockIdx.x % tiles;
    t.p = pr / b.nr;
    t.r = b.r0 + pr % b.nr;
    t.g = ntt_prime(b, t.r, L);
    return t;
}
// the low row pairs of a tile within their table
template <int LOGN>
__device__ __forceinline__ size_t low_at(const TileAt &t) {
    return ((size_t)t.g * Shape<LOGN>::TILES + t.tile) * Shape<LOGN>::PAIRS * NTHR;
}
// constant tables of a launch
struct NttTables {
    const PrimeDev *pr;
    const ulonglong2 *tw;   // [NP][N] pairs in natural order
    const ulonglong2 *low;  // [NP][N / 2048][PAIRS][128] low row pairs
    int L;
};
constexpr int FWD_BLOCKS = 6, INV_BLOCKS = 6;  // blocks per SM that the register count allows for (5: 2% slower, 4: 4%)

template <int LOGN, class IO>
__global__ void __launch_bounds__(NTHR, FWD_BLOCKS) k_ntt_fwd_cols(const __grid_constant__ NttBatch b, NttTables tb,
                                                                   const __grid_constant__ IO io, Mid mid) {
    using S = Shape<LOGN>;
    dep_trigger();
    dep_wait();
    __shared__ u64 sm[TILE];
    const TileAt t = tile_at(b, tb.L, S::TILES);
    if (ntt_skipped(b, t.p, t.r)) {
        io.skip(t.p, t.r, t.tile, S::TILES);
        return;
    }
    u64 v[16];
    fwd_cols<LOGN, 4, false>(io, t.p, t.r, t.g, t.tile, tb.tw + ((size_t)t.g << LOGN), tb.pr[t.g].q, sm, v, [] {});
    const int c = threadIdx.x & (S::C - 1), i = threadIdx.x >> S::LC;
    u64 *o = mid.base + t.p * mid.ps + ((size_t)(t.r - mid.r0) << LOGN) + ((size_t)t.tile << S::LC) + c;
#pragma unroll
    for (int m = 0; m < 16; m++) o[(size_t)(16 * i + m) << S::LB] = v[m];
}

template <int LOGN, class IO>
__global__ void __launch_bounds__(NTHR, FWD_BLOCKS) k_ntt_fwd_rows(const __grid_constant__ NttBatch b, NttTables tb,
                                                                   const __grid_constant__ IO io, Mid mid) {
    using S = Shape<LOGN>;
    dep_trigger();
    dep_wait();
    __shared__ u64 sm[PTILE];
    const TileAt t = tile_at(b, tb.L, S::TILES);
    if (ntt_skipped(b, t.p, t.r)) return;
    const int th = threadIdx.x, i = th & (S::SB - 1), gr = th / S::SB;
    const u64 *in = mid.base + t.p * mid.ps + ((size_t)(t.r - mid.r0) << LOGN) + ((size_t)t.tile << 11) +
                    (gr << S::LB) + i;
    u64 v[16];
#pragma unroll
    for (int m = 0; m < 16; m++) v[m] = in[m * S::SB];
    fwd_rows<LOGN, false>(io, t.p, t.r, t.g, t.tile,
                          TwRowTop<S::A>{tb.tw + ((size_t)t.g << LOGN), (t.tile << S::LR) + gr},
                          TwRowLow<S::LB - 4, false, false>{tb.low + low_at<LOGN>(t) + th}, tb.pr[t.g], sm, v);
}

template <int LOGN, class IO>
__global__ void __launch_bounds__(NTHR, INV_BLOCKS) k_ntt_inv_rows(const __grid_constant__ NttBatch b, NttTables tb,
                                                                   const __grid_constant__ IO io, Mid mid) {
    using S = Shape<LOGN>;
    dep_trigger();
    dep_wait();
    __shared__ u64 sm[PTILE];
    const TileAt t = tile_at(b, tb.L, S::TILES);
    if (ntt_skipped(b, t.p, t.r)) return;
    const int th = threadIdx.x, i = th & (S::SB - 1), gr = th / S::SB;
    u64 v[16];
    inv_rows<LOGN>(io, t.p, t.r, t.g, t.tile,
                   TwInvRowTop<S::A>{tb.tw + ((size_t)t.g << LOGN), (t.tile << S::LR) + gr},
                   TwRowLow<S::LB - 4, true, false>{tb.low + low_at<LOGN>(t) + th}, tb.pr[t.g], sm, v, [] {});
    u64 *o = mid.base + t.p * mid.ps + ((size_t)(t.r - mid.r0) << LOGN) + ((size_t)t.tile << 11) + (gr << S::LB) + i;
#pragma unroll
    for (int m = 0; m < 16; m++) o[m * S::SB] = v[m];
}

template <int LOGN, class IO>
__global__ void __launch_bounds__(NTHR, INV_BLOCKS) k_ntt_inv_cols(const __grid_constant__ NttBatch b, NttTables tb,
                                                                   const __grid_constant__ IO io, Mid mid) {
    using S = Shape<LOGN>;
    dep_trigger();
    dep_wait();
    __shared__ u64 sm[TILE];
    const TileAt t = tile_at(b, tb.L, S::TILES);
    if (ntt_skipped(b, t.p, t.r)) return;
    const int c = threadIdx.x & (S::C - 1), i = threadIdx.x >> S::LC;
    const u64 *in = mid.base + t.p * mid.ps + ((size_t)(t.r - mid.r0) << LOGN) + ((size_t)t.tile << S::LC) + c;
    u64 v[16];
#pragma unroll
    for (int m = 0; m < 16; m++) v[m] = in[(size_t)(16 * i + m) << S::LB];
    const PrimeDev P = tb.pr[t.g];
    const Shoup sc = b.scale ? b.scale[t.r - b.r0] : Shoup{P.ninv, P.ninv_sh};
    inv_cols<LOGN, false>(io, t.p, t.r, t.g, t.tile, tb.tw + ((size_t)t.g << LOGN), sc, b.digits, P.q, sm, v);
}

// ---------------------------------------------------------------- clusters: one launch
// A batch this small waits for memory more than for the multiplier, so every twiddle of the
// block is copied to shared memory from the start (asynchronous copies, in flight with the
// coefficients), the conversions take all of a thread's coefficients at a time (their digits'
// loads wait for one another half as often as with eight: a query of 47 and of 75 launches
// 284 -> 279 us and 1117 -> 1107 us), and the finishes' operands are loaded before the row stages.
template <int LOGN>
struct ClusterSmem {
    u64 colt[TILE], rowt[PTILE];
    ulonglong2 low[Shape<LOGN>::PAIRS * NTHR];  // [pair][thread]
    ulonglong2 top[15 * Shape<LOGN>::R];        // TwRowTopSh
    ulonglong2 col[1 << Shape<LOGN>::A];        // the prime's first 2^A pairs
};
// each thread copies the low pairs that it uses itself
template <int LOGN>
__device__ __forceinline__ void copy_twiddles(ClusterSmem<LOGN> &S, const NttTables &tb, const TileAt &t) {
    using H = Shape<LOGN>;
    const int th = threadIdx.x;
    const ulonglong2 *T = tb.tw + ((size_t)t.g << LOGN), *low = tb.low + low_at<LOGN>(t);
    for (int e = th; e < (1 << H::A); e += NTHR) cp_async16(&S.col[e], T + e);
    for (int e = th; e < 15 * H::R; e += NTHR) {
        // entry R (2^u - 1) + k: pair 2^(A + u) + (row0 << u) + k
        const int u = 31 - __clz(e / H::R + 1), k = e - H::R * ((1 << u) - 1);
        cp_async16(&S.top[e], T + (1 << (H::A + u)) + ((t.tile << H::LR) << u) + k);
    }
#pragma unroll
    for (int k = 0; k < H::PAIRS; k++) cp_async16(&S.low[k * NTHR + th], low + k * NTHR + th);
    cp_async_commit();
}

template <int LOGN, class IO>
__global__ void __cluster_dims__(Shape<LOGN>::TILES, 1, 1) __launch_bounds__(NTHR)
    k_ntt_fwd_cluster(const __grid_constant__ NttBatch b, NttTables tb, const __grid_constant__ IO io) {
    using S = Shape<LOGN>;
    extern __shared__ __align__(16) unsigned char dyn_smem[];
    ClusterSmem<LOGN> &M = *reinterpret_cast<ClusterSmem<LOGN> *>(dyn_smem);
    cg::cluster_group cl = cg::this_cluster();
    const TileAt t = tile_at(b, tb.L, S::TILES);  // tile = the block's rank
    dep_trigger();
    if (ntt_skipped(b, t.p, t.r)) {  // the same for every block of the cluster
        dep_wait();
        io.skip(t.p, t.r, t.tile, S::TILES);
        return;
    }
    cl.barrier_arrive();  // every block runs: its row tile may be written
    copy_twiddles<LOGN>(M, tb, t);
    dep_wait();
    const PrimeDev P = tb.pr[t.g];
    u64 v[16];
    fwd_cols<LOGN, 16, true>(io, t.p, t.r, t.g, t.tile, M.col, P.q, M.colt, v, [] {
        cp_async_wait<0>();
        __syncthreads();
    });
    cl.barrier_wait();
    const int th = threadIdx.x, c = th & (S::C - 1), ic = th >> S::LC, i = th & (S::SB - 1), gr = th / S::SB;
#pragma unroll
    for (int h = 0; h < 16; h += (S::R < 16 ? S::R : 16)) {
        // rows 16 ic + h .. belong to one block: R rows a block, R a power of two >= 8
        u64 *dst = cl.map_shared_rank(M.rowt, (16 * ic + h) >> S::LR);
#pragma unroll
        for (int m = h; m < h + (S::R < 16 ? S::R : 16); m++)
            dst[pad((((16 * ic + m) & (S::R - 1)) << S::LB) + (t.tile << S::LC) + c)] = v[m];
    }
    cl.sync();
#pragma unroll
    for (int m = 0; m < 16; m++) v[m] = M.rowt[pad((gr << S::LB) + i + m * S::SB)];
    fwd_rows<LOGN, true>(io, t.p, t.r, t.g, t.tile, TwRowTopSh<S::R, false>{M.top, gr},
                         TwRowLow<S::LB - 4, false, true>{M.low + th}, P, M.rowt, v);
}

template <int LOGN, class IO>
__global__ void __cluster_dims__(Shape<LOGN>::TILES, 1, 1) __launch_bounds__(NTHR)
    k_ntt_inv_cluster(const __grid_constant__ NttBatch b, NttTables tb, const __grid_constant__ IO io) {
    using S = Shape<LOGN>;
    extern __shared__ __align__(16) unsigned char dyn_smem[];
    ClusterSmem<LOGN> &M = *reinterpret_cast<ClusterSmem<LOGN> *>(dyn_smem);
    cg::cluster_group cl = cg::this_cluster();
    const TileAt t = tile_at(b, tb.L, S::TILES);
    dep_trigger();
    if (ntt_skipped(b, t.p, t.r)) {
        dep_wait();
        return;
    }
    cl.barrier_arrive();
    copy_twiddles<LOGN>(M, tb, t);
    dep_wait();
    const PrimeDev P = tb.pr[t.g];
    const int th = threadIdx.x, i = th & (S::SB - 1), gr = th / S::SB, c = th & (S::C - 1), ic = th >> S::LC;
    u64 v[16];
    // the low pairs are the thread's own copies; the others' are complete after the exchange's barrier
    inv_rows<LOGN>(io, t.p, t.r, t.g, t.tile, TwRowTopSh<S::R, true>{M.top, gr},
                   TwRowLow<S::LB - 4, true, true>{M.low + th}, P, M.rowt, v, [] { cp_async_wait<0>(); });
    cl.barrier_wait();
    const int row = (t.tile << S::LR) + gr;
#pragma unroll
    for (int m = 0; m < 16; m++) {
        const int col = i + m * S::SB;
        cl.map_shared_rank(M.colt, col >> S::LC)[(row << S::LC) + (col & (S::C - 1))] = v[m];
    }
    cl.sync();
#pragma unroll
    for (int m = 0; m < 16; m++) v[m] = M.colt[((16 * ic + m) << S::LC) + c];
    const Shoup sc = b.scale ? b.scale[t.r - b.r0] : Shoup{P.ninv, P.ninv_sh};
    inv_cols<LOGN, true>(io, t.p, t.r, t.g, t.tile, M.col, sc, b.digits, P.q, M.colt, v);
}

// ---------------------------------------------------------------- 2^8 <= N <= 2^11: one block
// A block of N / 16 threads holds one residue polynomial, 16 coefficients a thread: the first
// four stages, the next four and the remaining LOGN - 8 in registers, with an exchange through
// shared memory between them (a stage per exchange before: 5.6 us at N = 2^10 and 9.6 us at
// N = 2^11 for any batch that fits the GPU).
template <int LOGN>
__device__ __forceinline__ void copy_pairs(ulonglong2 *dst, const ulonglong2 *src) {
#pragma unroll
    for (int k = 0; k < 16; k++) cp_async16(dst + threadIdx.x + (k << (LOGN - 4)), src + threadIdx.x + (k << (LOGN - 4)));
    cp_async_commit();
}
template <int LOGN, class IO>
__global__ void __launch_bounds__(1 << (LOGN - 4)) k_ntt_fwd_one(const __grid_constant__ NttBatch b, NttTables tb,
                                                                 const __grid_constant__ IO io) {
    constexpr int NT = 1 << (LOGN - 4), LS = LOGN - 8, SP = 1 << LS;  // SP: threads per sixteenth
    __shared__ u64 sm[(1 << LOGN) + NT];
    __shared__ ulonglong2 T[1 << LOGN];
    const TileAt t = tile_at(b, tb.L, 1);
    dep_trigger();
    if (ntt_skipped(b, t.p, t.r)) {
        dep_wait();
        io.skip(t.p, t.r, 0, 1);
        return;
    }
    copy_pairs<LOGN>(T, tb.tw + ((size_t)t.g << LOGN));
    dep_wait();
    const PrimeDev P = tb.pr[t.g];
    const int th = threadIdx.x, i = th & (SP - 1), blk = th >> LS, f0 = (blk << (LOGN - 4)) + i;
    u64 v[16], u[4][4];
    load_n(io, t.p, t.r, t.g, (size_t)th, NT, v);
    cp_async_wait<0>();
    __syncthreads();
#pragma unroll
    for (int h = 0; h < 4; h++) operand_n(io, t.p, t.r, (size_t)(th + 4 * h * NT), NT, u[h]);
    stages_fwd<4>(v, P.q, 2 * P.q, TwColTop<true>{T});
#pragma unroll
    for (int m = 0; m < 16; m++) sm[pad(th + m * NT)] = v[m];
    __syncthreads();
#pragma unroll
    for (int m = 0; m < 16; m++) v[m] = sm[pad(f0 + m * SP)];
    stages_fwd<4>(v, P.q, 2 * P.q, [&](int s, int il) { return T[(1 << (4 + s)) + (blk << s) + il]; });
    if (LS > 0) {
#pragma unroll
        for (int m = 0; m < 16; m++) sm[pad(f0 + m * SP)] = v[m];
        __syncthreads();
#pragma unroll
        for (int m = 0; m < 16; m++) v[m] = sm[pad(16 * th + m)];
        stages_fwd<LS>(v, P.q, 2 * P.q, [&](int s, int il) { return T[(1 << (8 + s)) + ((16 * th) >> (LS - s)) + il]; });
    }
#pragma unroll
    for (int m = 0; m < 16; m++) sm[pad(16 * th + m)] = v[m];
    __syncthreads();
#pragma unroll
    for (int h = 0; h < 4; h++) {
        u64 x[4];
#pragma unroll
        for (int m = 0; m < 4; m++) {
            x[m] = sm[pad(th + (4 * h + m) * NT)];
            if (!IO::RAW) x[m] = fwd_reduce(x[m], P);
        }
        store_n(io, t.p, t.r, t.g, (size_t)(th + 4 * h * NT), NT, x, u[h]);
    }
}

template <int LOGN, class IO>
__global__ void __launch_bounds__(1 << (LOGN - 4)) k_ntt_inv_one(const __grid_constant__ NttBatch b, NttTables tb,
                                                                 const __grid_constant__ IO io) {
    constexpr int NT = 1 << (LOGN - 4), LS = LOGN - 8, SP = 1 << LS;
    __shared__ u64 sm[(1 << LOGN) + NT];
    __shared__ ulonglong2 T[1 << LOGN];
    const TileAt t = tile_at(b, tb.L, 1);
    dep_trigger();
    if (ntt_skipped(b, t.p, t.r)) {
        dep_wait();
        return;
    }
    copy_pairs<LOGN>(T, tb.tw + ((size_t)t.g << LOGN));
    dep_wait();
    const PrimeDev P = tb.pr[t.g];
    const u64 q = P.q;
    const int th = threadIdx.x, i = th & (SP - 1), blk = th >> LS, f0 = (blk << (LOGN - 4)) + i;
    u64 v[16];
#pragma unroll
    for (int m = 0; m < 16; m++) v[m] = io.load(t.p, t.r, t.g, (size_t)(th + m * NT));
#pragma unroll
    for (int m = 0; m < 16; m++) sm[pad(th + m * NT)] = v[m];
    cp_async_wait<0>();
    __syncthreads();
    if (LS > 0) {
#pragma unroll
        for (int m = 0; m < 16; m++) v[m] = sm[pad(16 * th + m)];
        stages_inv<LS>(v, q, q, [&](int s, int il) { return T[(1 << (LOGN - 1 - s)) + ((16 * th) >> (s + 1)) + il]; });
#pragma unroll
        for (int m = 0; m < 16; m++) sm[pad(16 * th + m)] = v[m];
        __syncthreads();
    }
#pragma unroll
    for (int m = 0; m < 16; m++) v[m] = sm[pad(f0 + m * SP)];
    stages_inv<4>(v, q, q << LS, [&](int s, int il) { return T[(1 << (7 - s)) + (blk << (3 - s)) + il]; });
#pragma unroll
    for (int m = 0; m < 16; m++) sm[pad(f0 + m * SP)] = reduce64_lazy(v[m], P);
    __syncthreads();
#pragma unroll
    for (int m = 0; m < 16; m++) v[m] = sm[pad(th + m * NT)];
    stages_inv<4>(v, q, 2 * q, TwInvColTop<true>{T});
    const Shoup sc = b.scale ? b.scale[t.r - b.r0] : Shoup{P.ninv, P.ninv_sh};
#pragma unroll
    for (int m = 0; m < 16; m++) io.store(t.p, t.r, t.g, (size_t)(th + m * NT), inv_result(v[m], sc, b.digits, q));
}

}  // namespace
