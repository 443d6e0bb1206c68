// The transform kernels.  For 2^12 <= N <= 2^15: N = 2^A rows of 2^LB coefficients, the first A
// forward stages over columns, the last LB over rows, the inverse the other way round (the
// stage order, twiddle order and lazy ranges are stated in ntt.cu).
//
// A tile is 2048 coefficients (columns x all rows, or rows x all columns) and a block of 128
// threads holds one in registers, 16 coefficients a thread: four stages in registers, one
// exchange through shared memory, the remaining two to four stages in registers.  What bounds a
// large batch is the integer multiplier (a butterfly is a 64-bit modular product), so the layout
// spends as little else as it can: an 8-stage pass has one exchange instead of one per two or
// three stages, and no index arithmetic between the stages.  Twiddles are read with their quotients
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
// polynomials 616 / 644 before, 318 / 355 with exact products, 277 / 325 with split ones (0.91 /
// 0.77 T butterflies/s of the 1.24 that the multiplier alone reaches: the rest is additions,
// exchanges, and 4 TB/s of memory traffic in the column half), 128: 44 / 50 and 39 / 47; N = 2^14,
// 1024 in clusters 269 / 313 before, 153 / 173 tiled, 138 / 161 split.
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
    // What the forward stages add to a value, in units of the modulus m = 2q < 2^56 (bf_fwd): all
    // column and the first four row stages are split, the low row stages exact or (LB = 8) split.
    static constexpr int GROWTH = 4 * (A + 4) + (LB == 8 ? 4 : 2) * (LB - 4);
    static_assert(GROWTH < 64, "a doubled word below 2^62 leaves 2^63");
};

__device__ __forceinline__ int ntt_prime(const NttBatch &b, int r, int L) {
    return b.fixed >= 0 ? b.fixed : (r < b.ell ? r : L + (r - b.ell));
}

// residue r of poly p is excluded from this batch (a ModUp digit's own primes)
__device__ __forceinline__ bool ntt_skipped(const NttBatch &b, int p, int r) {
    const int j = b.skip_period > 0 ? p % b.skip_period : p;
    return b.skip_alpha > 0 && r >= j * b.skip_alpha && r < min((j + 1) * b.skip_alpha, b.ell);
}

// Twiddle factors w of modulus m, in two forms.
//
// Exact: the pair (w, w' = floor(w 2^64 / m)); the Shoup product of any 64-bit value is below 2m.
// Ten multiply instructions.
//
// Split (N >= 2^12): the values carry a factor of two, X = 2x, and the modulus is m = 2q.  With
// x = x1 2^31 + x0, so that X's words are x1 and 2 x0 without any shift, and v = w 2^31 mod q,
//   x w = x1 v + x0 w,   X w = x1 (2v) + (2 x0) w  (mod m),
// and the quotient by q is x1 v / q + x0 w / q, below 2^32 for x < 2^62: from
// vq = floor(v 2^32 / q) and wq = floor(w 2^31 / q) with two high words,
//   h = floor(x1 vq / 2^32) + floor(2 x0 wq / 2^32),
// short by less than x1 / 2^32 + 1 (the truncated constants) + 2 (the floors), so that
// X w - h m is below 2 (3.5 q) < 4m.  Eight multiply instructions: 1.24 T butterflies/s of the
// multiplier alone (152 SMs), 1.04 exact ones.
struct Tw3 {
    u64 w, v;         // w, 2 (w 2^31 mod q)
    uint32_t wq, vq;  // floor(w 2^31 / q), floor((w 2^31 mod q) 2^32 / q)
};
__device__ __forceinline__ u64 tw_mul(u64 x, ulonglong2 w, u64 m) { return mul_shoup_lazy(x, w.x, w.y, m); }
__device__ __forceinline__ u64 tw_mul(u64 x, const Tw3 &w, u64 m) {
    const uint32_t x0 = (uint32_t)x, x1 = (uint32_t)(x >> 32);
    const uint32_t h = __umulhi(x1, w.vq) + __umulhi(x0, w.wq);
    return (u64)x1 * w.v + (u64)x0 * w.w - (u64)h * m;
}
// what a product stays below, in units of m
__device__ __forceinline__ constexpr u64 tw_bound(const ulonglong2 &) { return 2; }
__device__ __forceinline__ constexpr u64 tw_bound(const Tw3 &) { return 4; }

// Forward butterfly without a correction step: the product V is below B m (B = 2 or 4), so
// x' = U + V and y' = U - V + B m only grow by B m per stage.  One-block transforms (N <= 2^11,
// m = q, every stage exact): from inputs below 2q, values stay below (2 log2 N + 2) q <= 24q.  From
// 2^12 on (m = 2q < 2^56 for primes below 2^55, the context's limit; Shape::GROWTH): from doubled
// inputs below 2m, values stay below 46m, 48m, 52m and 62m at N = 2^12 .. 2^15 (halved, below 2^61);
// from doubled words below 2^62, below 2^62 + 60m < 2^63, which is what a split product takes.  The
// final store reduces them once.
template <class TW>
__device__ __forceinline__ void bf_fwd(u64 &x, u64 &y, const TW &w, u64 m) {
    const u64 U = x;
    const u64 V = tw_mul(y, w, m);
    x = U + V;
    y = U - V + tw_bound(w) * m;
}

// Inverse butterfly without a correction step, for a stage whose inputs are below c (a
// multiple of m, at least B m / 2): U - V + c is positive and below 2c, so the product is the
// same residue, x' = U + V < 2c and y' < B m <= 2c.  From inputs below c0, stage u of a pass takes
// c = 2^u c0.  The products' inputs stay below 2^63: passes of more than four stages lower the
// values that four stages from 8m would take past that (inv_cap).
template <class TW>
__device__ __forceinline__ void bf_inv(u64 &x, u64 &y, const TW &w, u64 m, u64 c) {
    const u64 U = x, V = y;
    x = U + V;
    y = tw_mul(U - V + c, w, m);
}

// a doubled value reduced below 2m = 4q (reduce64_lazy of modulus 2q)
__device__ __forceinline__ u64 reduce2_lazy(u64 x, const PrimeDev &P) {
    if (P.one_sh >> 33) return mul_shoup_lazy(x, 1, P.one_sh >> 1, 2 * P.q);
    const uint32_t c = (uint32_t)(P.one_sh >> 1);
    const uint32_t h = (uint32_t)(((x >> 32) * c + __umulhi((uint32_t)x, c)) >> 32);
    return x - (u64)h * (2 * P.q);
}

// a transform's lazy value reduced to [0, q)
__device__ __forceinline__ u64 fwd_reduce(u64 v, const PrimeDev &P) {
    const u64 r = reduce64_lazy(v, P);
    return r >= P.q ? r - P.q : r;
}

// K forward stages (distances 2^(K-1), .., 1 within groups of 2^K) on 16 registers;
// tw(s, il): the pair of stage s, group il < 16 >> (K - s)
template <int K, class TW>
__device__ __forceinline__ void stages_fwd(u64 (&v)[16], u64 m, TW tw) {
#pragma unroll
    for (int s = 0; s < K; s++) {
        const int ld = K - 1 - s, d = 1 << ld;
        decltype(tw(0, 0)) w;
#pragma unroll
        for (int x = 0; x < 8; x++) {
            const int il = x >> ld, j = x & (d - 1);
            if (j == 0) w = tw(s, il);
            bf_fwd(v[2 * d * il + j], v[2 * d * il + d + j], w, m);
        }
    }
}
// K inverse stages (distances 1, .., 2^(K-1)); inputs below c0; tw(s, il): il < 8 >> s
template <int K, class TW>
__device__ __forceinline__ void stages_inv(u64 (&v)[16], u64 m, u64 c0, TW tw) {
#pragma unroll
    for (int s = 0; s < K; s++) {
        const int d = 1 << s;
        decltype(tw(0, 0)) w;
#pragma unroll
        for (int x = 0; x < 8; x++) {
            const int il = x >> s, j = x & (d - 1);
            if (j == 0) w = tw(s, il);
            bf_inv(v[2 * d * il + j], v[2 * d * il + d + j], w, m, c0 << s);
        }
    }
}

// After K inverse stages from inputs below C m with products below B m, value j of a group of 2^K
// is below C 2^K m (j = 0: sums only) or B 2^(K - 1 - b) m (b: its highest bit, the last stage at
// which it was the product).  Those that can pass 8m are reduced below 2m.
template <int K, int C, int B>
__device__ __forceinline__ void inv_cap(u64 (&v)[16], const PrimeDev &P) {
#pragma unroll
    for (int x = 0; x < 16; x++) {
        const int j = x & ((1 << K) - 1);
        const int bound = j == 0 ? C << K : (B << (K - 1)) >> (j >= 8 ? 3 : j >= 4 ? 2 : j >= 2 ? 1 : 0);
        if (bound > 8) v[x] = reduce2_lazy(v[x], P);
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
// pad(f + d) - pad(f) where f mod 16 + d mod 16 < 16
__device__ __forceinline__ constexpr int padc(int d) { return d + (d >> 4); }

// a table of split twiddles: (w, 2v) and (wq, vq)
struct Tab3 {
    const ulonglong2 *w;
    const uint2 *q;
    __device__ __forceinline__ Tab3 operator+(size_t k) const { return Tab3{w + k, q + k}; }
};
template <bool SH>
__device__ __forceinline__ Tw3 tw3_at(const Tab3 &t, int k) {
    ulonglong2 a;
    uint2 b;
    if constexpr (SH) {
        a = t.w[k];
        b = t.q[k];
    } else {
        a = __ldg(t.w + k);
        b = __ldg(t.q + k);
    }
    return Tw3{a.x, a.y, b.x, b.y};
}

// twiddles of the passes (T: the prime's split twiddles in natural order, low: this tile's low
// row twiddles of this thread, [pair][thread]); the column stages use the first 2^A twiddles only.
// The low ones are one per butterfly, so that their bytes count: split ones gain for the four low
// stages of N = 2^15 (1024 residue polynomials forward / inverse 295 / 334 us with exact pairs,
// 288 / 325 split) and lose for the three of N = 2^14 (147 / 162 exact, 145 / 165 split).
//
// forward column stages 0..3: the whole transform's first 15 twiddles
template <bool SH>
struct TwColTop {
    Tab3 T;
    __device__ __forceinline__ Tw3 operator()(int s, int il) const { return tw3_at<SH>(T, (1 << s) + il); }
};
// forward column stages 4..A-1 of rows 16 b ..
template <int A, bool SH>
struct TwColLow {
    Tab3 T;
    int b;
    __device__ __forceinline__ Tw3 operator()(int s, int il) const {
        return tw3_at<SH>(T, (1 << (4 + s)) + ((16 * b) >> (A - 4 - s)) + il);
    }
};
// forward row stages 0..3 of one row
template <int A>
struct TwRowTop {
    Tab3 T;
    int row;
    __device__ __forceinline__ Tw3 operator()(int s, int il) const {
        return tw3_at<false>(T, (1 << (A + s)) + (row << s) + il);
    }
};
// the same, and the last four inverse row stages, from a copy of the 15 pairs of each of a tile's
// R rows, those of 2^u groups per row at R (2^u - 1) (gr: the row within the tile)
template <int R, bool INV>
struct TwRowTopSh {
    Tab3 T;
    int gr;
    __device__ __forceinline__ Tw3 operator()(int s, int il) const {
        const int u = INV ? 3 - s : s;
        return tw3_at<true>(T, R * ((1 << u) - 1) + (gr << u) + il);
    }
};
// low row stages in thread order: the twiddles of stage s follow those of the stages before
template <int K, bool INV, bool SH>
struct TwRowLow {
    static constexpr bool SPLIT = K == 4;  // LB = 8
    static constexpr int B = SPLIT ? 4 : 2;
    Tab3 low;
    __device__ __forceinline__ auto operator()(int s, int il) const {
        const int k = ((INV ? 16 - (16 >> s) : (16 >> (K - s)) - (16 >> K)) + il) * NTHR;
        if constexpr (SPLIT) return tw3_at<SH>(low, k);
        else return pair_at<SH>(low.w + k);
    }
};
// inverse column stages of distance 2^s rows, rows 16 b ..
template <int A, bool SH>
struct TwInvColLow {
    Tab3 T;
    int b;
    __device__ __forceinline__ Tw3 operator()(int s, int il) const {
        return tw3_at<SH>(T, (1 << (A - 1 - s)) + ((16 * b) >> (s + 1)) + il);
    }
};
// the last four inverse column stages
template <bool SH>
struct TwInvColTop {
    Tab3 T;
    __device__ __forceinline__ Tw3 operator()(int s, int il) const { return tw3_at<SH>(T, (1 << (3 - s)) + il); }
};
// the last four inverse row stages of one row
template <int A>
struct TwInvRowTop {
    Tab3 T;
    int row;
    __device__ __forceinline__ Tw3 operator()(int s, int il) const {
        return tw3_at<false>(T, (1 << (A + 3 - s)) + (row << (3 - s)) + il);
    }
};

// ---------------------------------------------------------------- the halves of a transform
// Forward column half: the tile's coefficients through io (KL at a time), all A column stages;
// the thread ends with rows 16 b .. 16 b + 15 of its column.  SH: the first 2^A pairs at T are
// the block's copy, complete after `arrived`.
template <int LOGN, int KL, bool SH, class IO, class ARR>
__device__ __forceinline__ void fwd_cols(const IO &io, int p, int r, int g, int tile, Tab3 T,
                                         const PrimeDev &P, u64 *sm, u64 (&v)[16], ARR arrived) {
    using S = Shape<LOGN>;
    const u64 m2 = 2 * P.q;
    const int t = threadIdx.x, c = t & (S::C - 1), i = t >> S::LC;
    const size_t n0 = ((size_t)i << S::LB) + (tile << S::LC) + c, dn = (size_t)S::SA << S::LB;
#pragma unroll
    for (int h = 0; h < 16 / KL; h++) {
        u64 x[KL];
        load_n(io, p, r, g, n0 + KL * h * dn, dn, x);
#pragma unroll
        for (int m = 0; m < KL; m++) v[KL * h + m] = x[m];
    }
    if constexpr (std::is_same<IO, PlainIO>::value) {
        // a caller's coefficients need not be residues: any 64-bit value, lowered where the bounds
        // of split twiddles (x + 60q < 2^62) need it.  One test for the thread's sixteen, which
        // also puts all loads before the first butterfly: 277 us for 1024 residue polynomials of
        // 2^15 (288 without a test, 313 with one per four)
        uint32_t any = 0;
#pragma unroll
        for (int m = 0; m < 16; m++) any |= (uint32_t)(v[m] >> 32);
        if (any >> 29) {
#pragma unroll
            for (int m = 0; m < 16; m++) v[m] = reduce64_lazy(v[m], P);
        }
    }
#pragma unroll
    for (int m = 0; m < 16; m++) v[m] *= 2;
    arrived();
    stages_fwd<4>(v, m2, TwColTop<SH>{T});
#pragma unroll
    for (int m = 0; m < 16; m++) sm[((i + m * S::SA) << S::LC) + c] = v[m];
    __syncthreads();
#pragma unroll
    for (int m = 0; m < 16; m++) v[m] = sm[((16 * i + m) << S::LC) + c];
    stages_fwd<S::A - 4>(v, m2, TwColLow<S::A, SH>{T, i});
}

// Forward row half: v holds coefficients i + m SB of the thread's row (i = t mod SB); all LB row
// stages, the values stored through io (reduced unless it takes them raw).  u: the finishes'
// operands where they are loaded ahead (EARLY), in the order of the stores.
template <int LOGN, bool EARLY, class IO, class TOP, class LOW>
__device__ __forceinline__ void fwd_rows(const IO &io, int p, int r, int g, int tile, TOP top, LOW low,
                                         const PrimeDev &P, u64 *sm, u64 (&v)[16]) {
    using S = Shape<LOGN>;
    const int t = threadIdx.x, i = t & (S::SB - 1), gr = t / S::SB;
    const u64 m2 = 2 * P.q;
    const int f0 = (t & ~31) * 16 + (t & 31);
    u64 *seq = sm + pad((gr << S::LB) + i), *own = sm + pad(16 * t), *run = sm + pad(f0);
    const size_t k0 = ((size_t)tile << 11) + f0;
    constexpr int H = EARLY ? 4 : 8;  // coefficients stored together
    u64 u[16 / H][H];
    if (EARLY) {
#pragma unroll
        for (int h = 0; h < 16 / H; h++) operand_n(io, p, r, k0 + 32 * H * h, 32, u[h]);
    }
    stages_fwd<4>(v, m2, top);
#pragma unroll
    for (int m = 0; m < 16; m++) seq[padc(m * S::SB)] = v[m];
    __syncthreads();
#pragma unroll
    for (int m = 0; m < 16; m++) v[m] = own[m];
    stages_fwd<S::LB - 4>(v, m2, low);
    // to runs of 32 coefficients per warp access, within the warp's 512
#pragma unroll
    for (int m = 0; m < 16; m++) own[m] = v[m];
    __syncwarp();
#pragma unroll
    for (int h = 0; h < 16 / H; h++) {
        u64 x[H];
        if (!EARLY) operand_n(io, p, r, k0 + 32 * H * h, 32, u[h]);
#pragma unroll
        for (int m = 0; m < H; m++) {
            x[m] = run[padc(32 * (H * h + m))] >> 1;
            if (!IO::RAW) x[m] = fwd_reduce(x[m], P);
        }
        store_n(io, p, r, g, k0 + 32 * H * h, 32, x, u[h]);
    }
}

// Inverse row half: the tile through io.load, all LB row stages; the thread ends with
// coefficients i + m SB of its row, doubled, below 4q.  `arrived`: the twiddles' copies complete.
template <int LOGN, class IO, class TOP, class LOW, class ARR>
__device__ __forceinline__ void inv_rows(const IO &io, int p, int r, int g, int tile, TOP top, LOW low,
                                         const PrimeDev &P, u64 *sm, u64 (&v)[16], ARR arrived) {
    using S = Shape<LOGN>;
    const int t = threadIdx.x, i = t & (S::SB - 1), gr = t / S::SB;
    const u64 m2 = 2 * P.q;
    const int f0 = (t & ~31) * 16 + (t & 31);
    u64 *seq = sm + pad((gr << S::LB) + i), *own = sm + pad(16 * t), *run = sm + pad(f0);
#pragma unroll
    for (int m = 0; m < 16; m++) v[m] = 2 * io.load(p, r, g, ((size_t)tile << 11) + f0 + 32 * m);
#pragma unroll
    for (int m = 0; m < 16; m++) run[padc(32 * m)] = v[m];
    arrived();
    __syncwarp();
#pragma unroll
    for (int m = 0; m < 16; m++) v[m] = own[m];
    stages_inv<S::LB - 4>(v, m2, LOW::B / 2 * m2, low);
    inv_cap<S::LB - 4, LOW::B / 2, LOW::B>(v, P);
#pragma unroll
    for (int m = 0; m < 16; m++) own[m] = v[m];
    __syncthreads();
#pragma unroll
    for (int m = 0; m < 16; m++) v[m] = seq[padc(m * S::SB)];
    stages_inv<4>(v, m2, 8 * m2, top);
#pragma unroll
    for (int m = 0; m < 16; m++) v[m] = reduce2_lazy(v[m], P);
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

// sc w mod q as a Shoup pair: with 2^64 = one_sh q + r64, floor(sw 2^64 / q) is sw one_sh +
// floor(sw r64 / q), the last term by its own quotient and possibly one short, so that a product
// of a value below 2^62 stays below 2q
__device__ __forceinline__ Shoup scaled_twiddle(Shoup sc, const Tw3 &w, const PrimeDev &P) {
    u64 s = tw_mul(2 * sc.w, w, 2 * P.q) >> 1;  // below 4q
    if (s >= 2 * P.q) s -= 2 * P.q;
    if (s >= P.q) s -= P.q;
    return Shoup{s, s * P.one_sh + __umul64hi(s, P.r64_sh)};
}

// Inverse column half: v holds rows 16 b .. 16 b + 15 of the thread's column (doubled, below 4q); all A
// column stages, scaled and stored through io.
template <int LOGN, bool SH, class IO>
__device__ __forceinline__ void inv_cols(const IO &io, int p, int r, int g, int tile, Tab3 T, Shoup sc,
                                         bool digits, const PrimeDev &P, u64 *sm, u64 (&v)[16]) {
    using S = Shape<LOGN>;
    const int t = threadIdx.x, c = t & (S::C - 1), i = t >> S::LC;
    const u64 m2 = 2 * P.q;
    stages_inv<S::A - 4>(v, m2, 2 * m2, TwInvColLow<S::A, SH>{T, i});
    inv_cap<S::A - 4, 2, 4>(v, P);
#pragma unroll
    for (int m = 0; m < 16; m++) sm[((16 * i + m) << S::LC) + c] = v[m];
    __syncthreads();
#pragma unroll
    for (int m = 0; m < 16; m++) v[m] = sm[((i + m * S::SA) << S::LC) + c];
    const TwInvColTop<SH> top{T};
    Shoup sw = sc;
    if constexpr (SH) {
        // the last stage's products are by one twiddle: it takes the scaling with it (queries of 75
        // and 90 launches 1035 -> 1027 us and 1675 -> 1666; tiled, where the eight products saved
        // meet the register limit, 325 us either way)
        stages_inv<3>(v, m2, 8 * m2, top);
        sw = scaled_twiddle(sc, top(3, 0), P);
#pragma unroll
        for (int m = 0; m < 8; m++) {
            const u64 U = v[m], V = v[m + 8];
            v[m] = U + V;
            v[m + 8] = U - V + 64 * m2;
        }
    } else {
        stages_inv<4>(v, m2, 8 * m2, top);
    }
#pragma unroll
    for (int m = 0; m < 16; m++)
        io.store(p, r, g, ((size_t)(i + m * S::SA) << S::LB) + (tile << S::LC) + c, inv_result(v[m] >> 1, m < 8 ? sc : sw, digits, P.q));
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
// constant tables of a launch
struct NttTables {
    const PrimeDev *pr;
    const ulonglong2 *tw;   // [NP][N] in natural order: exact pairs of q, or (N >= 2^12) (w, 2v) of split twiddles
    const uint2 *twq;       // and their (wq, vq)
    const ulonglong2 *low;  // [NP][N / 2048][PAIRS][128] low row twiddles: exact pairs of 2q, or (N = 2^15)
    const uint2 *lowq;      // split
    int L;
    // the low row twiddles of a tile
    template <int LOGN>
    __device__ __forceinline__ Tab3 low_of(const TileAt &t) const {
        return Tab3{low, lowq} + ((size_t)t.g * Shape<LOGN>::TILES + t.tile) * Shape<LOGN>::PAIRS * NTHR;
    }
    __device__ __forceinline__ Tab3 tab(int g, int logN) const { return Tab3{tw, twq} + ((size_t)g << logN); }
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
        io.skip(t.p, t.r, t.tile, S::TILES, threadIdx.x, NTHR);
        return;
    }
    u64 v[16];
    fwd_cols<LOGN, 4, false>(io, t.p, t.r, t.g, t.tile, tb.tab(t.g, LOGN), tb.pr[t.g], sm, v, [] {});
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
                          TwRowTop<S::A>{tb.tab(t.g, LOGN), (t.tile << S::LR) + gr},
                          TwRowLow<S::LB - 4, false, false>{tb.low_of<LOGN>(t) + th}, tb.pr[t.g], sm, v);
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
                   TwInvRowTop<S::A>{tb.tab(t.g, LOGN), (t.tile << S::LR) + gr},
                   TwRowLow<S::LB - 4, true, false>{tb.low_of<LOGN>(t) + th}, tb.pr[t.g], sm, v, [] {});
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
    inv_cols<LOGN, false>(io, t.p, t.r, t.g, t.tile, tb.tab(t.g, LOGN), sc, b.digits, P, sm, v);
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
    uint2 lowq[LOGN == 15 ? Shape<LOGN>::PAIRS * NTHR : 1];
    ulonglong2 top[15 * Shape<LOGN>::R];        // TwRowTopSh
    ulonglong2 col[1 << Shape<LOGN>::A];        // the prime's first 2^A twiddles
    uint2 topq[15 * Shape<LOGN>::R], colq[1 << Shape<LOGN>::A];
};
// each thread copies the low pairs that it uses itself
template <int LOGN>
__device__ __forceinline__ void copy_twiddles(ClusterSmem<LOGN> &S, const NttTables &tb, const TileAt &t) {
    using H = Shape<LOGN>;
    const int th = threadIdx.x;
    const Tab3 T = tb.tab(t.g, LOGN);
    const Tab3 low = tb.low_of<LOGN>(t);
    for (int e = th; e < (1 << H::A); e += NTHR) {
        cp_async16(&S.col[e], T.w + e);
        cp_async8(&S.colq[e], T.q + e);
    }
    for (int e = th; e < 15 * H::R; e += NTHR) {
        // entry R (2^u - 1) + k: pair 2^(A + u) + (row0 << u) + k
        const int u = 31 - __clz(e / H::R + 1), k = e - H::R * ((1 << u) - 1);
        const int at = (1 << (H::A + u)) + ((t.tile << H::LR) << u) + k;
        cp_async16(&S.top[e], T.w + at);
        cp_async8(&S.topq[e], T.q + at);
    }
#pragma unroll
    for (int k = 0; k < H::PAIRS; k++) {
        cp_async16(&S.low[k * NTHR + th], low.w + k * NTHR + th);
        if (LOGN == 15) cp_async8(&S.lowq[k * NTHR + th], low.q + k * NTHR + th);
    }
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
        io.skip(t.p, t.r, t.tile, S::TILES, threadIdx.x, NTHR);
        return;
    }
    cl.barrier_arrive();  // every block runs: its row tile may be written
    copy_twiddles<LOGN>(M, tb, t);
    dep_wait();
    const PrimeDev P = tb.pr[t.g];
    u64 v[16];
    fwd_cols<LOGN, 16, true>(io, t.p, t.r, t.g, t.tile, Tab3{M.col, M.colq}, P, M.colt, v, [] {
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
    fwd_rows<LOGN, true>(io, t.p, t.r, t.g, t.tile, TwRowTopSh<S::R, false>{Tab3{M.top, M.topq}, gr},
                         TwRowLow<S::LB - 4, false, true>{Tab3{M.low, M.lowq} + th}, P, M.rowt, v);
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
    inv_rows<LOGN>(io, t.p, t.r, t.g, t.tile, TwRowTopSh<S::R, true>{Tab3{M.top, M.topq}, gr},
                   TwRowLow<S::LB - 4, true, true>{Tab3{M.low, M.lowq} + th}, P, M.rowt, v, [] { cp_async_wait<0>(); });
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
    inv_cols<LOGN, true>(io, t.p, t.r, t.g, t.tile, Tab3{M.col, M.colq}, sc, b.digits, P, M.colt, v);
}

// ---------------------------------------------------------------- 2^8 <= N <= 2^11: one block
// A block of N / 16 threads holds one residue polynomial, 16 coefficients a thread: the first
// four stages, the next four and the remaining LOGN - 8 in registers, with an exchange through
// shared memory between them (a stage per exchange before: 5.6 us at N = 2^10 and 9.6 us at
// N = 2^11 for any batch that fits the GPU).  The inverse takes words below 2q, as the rings below
// do: its passes of LOGN - 4 <= 7 stages start from c0 = 2q and stay below 2^8 q < 2^63.
// At N = 2^8 a transform is half a warp: two of them share a block, which is then one warp, each half
// synchronised by itself.  With a block of 16 threads each, the inverse of 1024 / 2048 residue
// polynomials took 9.9 / 13.5 us (128 threads a block and a stage per barrier: 8.3 / 12.4), now
// 6.1 / 10.2; four and eight to a block measure the same.
template <int LOGN>
struct One {
    static constexpr int NT = 1 << (LOGN - 4), LS = LOGN - 8, SP = 1 << LS;  // SP: threads per sixteenth
    static constexpr int PER = LOGN == 8 ? 2 : 1;                            // transforms per block
    // the transform's place in its block, the thread's in its transform
    static __device__ __forceinline__ int place() { return PER == 1 ? 0 : threadIdx.x / NT; }
    static __device__ __forceinline__ int thread() { return PER == 1 ? threadIdx.x : threadIdx.x % NT; }
    static __device__ __forceinline__ void sync() {
        if constexpr (PER == 2) __syncwarp(0xffffu << (threadIdx.x & 16));
        else __syncthreads();
    }
    // the transform of this thread; false past the last one
    static __device__ __forceinline__ bool at(const NttBatch &b, int L, TileAt &t) {
        const int pr = (int)blockIdx.x * PER + place();
        t.tile = 0;
        t.p = pr / b.nr;
        t.r = b.r0 + pr % b.nr;
        t.g = ntt_prime(b, t.r, L);
        return PER == 1 || pr < b.npoly * b.nr;
    }
};
template <int LOGN>
__device__ __forceinline__ void copy_pairs(ulonglong2 *dst, const ulonglong2 *src) {
    const int th = One<LOGN>::thread();
#pragma unroll
    for (int k = 0; k < 16; k++) cp_async16(dst + th + (k << (LOGN - 4)), src + th + (k << (LOGN - 4)));
    cp_async_commit();
}
template <int LOGN, class IO>
__global__ void __launch_bounds__(One<LOGN>::NT *One<LOGN>::PER)
    k_ntt_fwd_one(const __grid_constant__ NttBatch b, NttTables tb, const __grid_constant__ IO io) {
    using O = One<LOGN>;
    constexpr int NT = O::NT, LS = O::LS, SP = O::SP;
    __shared__ u64 sms[O::PER][(1 << LOGN) + NT];
    __shared__ ulonglong2 Ts[O::PER][1 << LOGN];
    u64 *sm = sms[O::place()];
    ulonglong2 *T = Ts[O::place()];
    TileAt t;
    const bool some = O::at(b, tb.L, t);
    dep_trigger();
    if (!some || ntt_skipped(b, t.p, t.r)) {
        dep_wait();
        if (some) io.skip(t.p, t.r, 0, 1, O::thread(), NT);
        return;
    }
    copy_pairs<LOGN>(T, tb.tw + ((size_t)t.g << LOGN));
    dep_wait();
    const PrimeDev P = tb.pr[t.g];
    const int th = O::thread(), i = th & (SP - 1), blk = th >> LS, f0 = (blk << (LOGN - 4)) + i;
    u64 v[16], u[4][4];
    load_n(io, t.p, t.r, t.g, (size_t)th, NT, v);
    cp_async_wait<0>();
    O::sync();
#pragma unroll
    for (int h = 0; h < 4; h++) operand_n(io, t.p, t.r, (size_t)(th + 4 * h * NT), NT, u[h]);
    stages_fwd<4>(v, P.q, [&](int s, int il) { return T[(1 << s) + il]; });
#pragma unroll
    for (int m = 0; m < 16; m++) sm[pad(th + m * NT)] = v[m];
    O::sync();
#pragma unroll
    for (int m = 0; m < 16; m++) v[m] = sm[pad(f0 + m * SP)];
    stages_fwd<4>(v, P.q, [&](int s, int il) { return T[(1 << (4 + s)) + (blk << s) + il]; });
    if (LS > 0) {
#pragma unroll
        for (int m = 0; m < 16; m++) sm[pad(f0 + m * SP)] = v[m];
        O::sync();
#pragma unroll
        for (int m = 0; m < 16; m++) v[m] = sm[pad(16 * th + m)];
        stages_fwd<LS>(v, P.q, [&](int s, int il) { return T[(1 << (8 + s)) + ((16 * th) >> (LS - s)) + il]; });
    }
#pragma unroll
    for (int m = 0; m < 16; m++) sm[pad(16 * th + m)] = v[m];
    O::sync();
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
__global__ void __launch_bounds__(One<LOGN>::NT *One<LOGN>::PER)
    k_ntt_inv_one(const __grid_constant__ NttBatch b, NttTables tb, const __grid_constant__ IO io) {
    using O = One<LOGN>;
    constexpr int NT = O::NT, LS = O::LS, SP = O::SP;
    __shared__ u64 sms[O::PER][(1 << LOGN) + NT];
    __shared__ ulonglong2 Ts[O::PER][1 << LOGN];
    u64 *sm = sms[O::place()];
    ulonglong2 *T = Ts[O::place()];
    TileAt t;
    const bool some = O::at(b, tb.L, t);
    dep_trigger();
    if (!some || ntt_skipped(b, t.p, t.r)) {
        dep_wait();
        return;
    }
    copy_pairs<LOGN>(T, tb.tw + ((size_t)t.g << LOGN));
    dep_wait();
    const PrimeDev P = tb.pr[t.g];
    const u64 q = P.q;
    const int th = O::thread(), i = th & (SP - 1), blk = th >> LS, f0 = (blk << (LOGN - 4)) + i;
    u64 v[16];
#pragma unroll
    for (int m = 0; m < 16; m++) v[m] = io.load(t.p, t.r, t.g, (size_t)(th + m * NT));
#pragma unroll
    for (int m = 0; m < 16; m++) sm[pad(th + m * NT)] = v[m];
    cp_async_wait<0>();
    O::sync();
    if (LS > 0) {
#pragma unroll
        for (int m = 0; m < 16; m++) v[m] = sm[pad(16 * th + m)];
        stages_inv<LS>(v, q, 2 * q, [&](int s, int il) { return T[(1 << (LOGN - 1 - s)) + ((16 * th) >> (s + 1)) + il]; });
#pragma unroll
        for (int m = 0; m < 16; m++) sm[pad(16 * th + m)] = v[m];
        O::sync();
    }
#pragma unroll
    for (int m = 0; m < 16; m++) v[m] = sm[pad(f0 + m * SP)];
    stages_inv<4>(v, q, (2 * q) << LS, [&](int s, int il) { return T[(1 << (7 - s)) + (blk << (3 - s)) + il]; });
#pragma unroll
    for (int m = 0; m < 16; m++) sm[pad(f0 + m * SP)] = reduce64_lazy(v[m], P);
    O::sync();
#pragma unroll
    for (int m = 0; m < 16; m++) v[m] = sm[pad(th + m * NT)];
    stages_inv<4>(v, q, 2 * q, [&](int s, int il) { return T[(1 << (3 - s)) + il]; });
    const Shoup sc = b.scale ? b.scale[t.r - b.r0] : Shoup{P.ninv, P.ninv_sh};
#pragma unroll
    for (int m = 0; m < 16; m++) io.store(t.p, t.r, t.g, (size_t)(th + m * NT), inv_result(v[m], sc, b.digits, q));
}

}  // namespace
