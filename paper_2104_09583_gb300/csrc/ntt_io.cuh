// What the transforms load and store (see ntt_core.cuh): the plain and out-of-place forms, and
// the base conversions (ModUp, ModDown, relinearise-and-drop, modulus switch) whose conversion
// is the transform's load and whose finish is its store.
#pragma once

#include "internal.cuh"

namespace {

// finishing arithmetic of a modulus switch for value v = NTT(conversion) at (p, r, k)
__device__ __forceinline__ void ms_store(const MsFuse &f, const PrimeDev *pr, const KsTables &T, int L, int logN,
                                         int p, int r, size_t k, u64 v) {
    const PrimeDev P = pr[r];
    const u64 xv = f.xp[0] ? f.xp[p][((size_t)r << logN) + k] : f.x[(((size_t)p * f.ell + r) << logN) + k];
    const u64 d = mul_shoup(v, P.t_mod, P.t_mod_sh, P.q);
    u64 *o = f.outp[0] ? f.outp[p] + ((size_t)r << logN) + k : f.out + (((size_t)p * (f.ell - 1) + r) << logN) + k;
    *o = mul_shoup(sub_mod(xv, d, P.q), T.ms_qinv[(size_t)f.ell * L + r], P.q);
}

// finishing arithmetic of a ModDown for value v = NTT(conversion) at (p = 2 job + c, r, k)
__device__ __forceinline__ void md_store(const MdFuse &f, const PrimeDev *pr, const KsTables &T, int logN, int p,
                                         int r, size_t k, u64 v) {
    const int job = p >> 1, c = p & 1;
    const PrimeDev P = pr[r];
    const u64 uv = f.U[(size_t)p * f.ustride + ((size_t)r << logN) + k];
    u64 res = mul_shoup(sub_mod(uv, mul_shoup(v, P.t_mod, P.t_mod_sh, P.q), P.q), T.md_Pinv[r], P.q);
    if (c < f.add_comps && f.add[job]) {
        const size_t src = (c == 0 && f.gal[job] != 1) ? galois_src((uint32_t)k, f.gal[job], logN) : k;
        res = add_mod(res, f.add[job][(size_t)c * f.acomp + ((size_t)r << logN) + src], P.q);
    }
    f.out[job][(size_t)c * f.ocomp + ((size_t)r << logN) + k] = res;
}

// conversion of polynomial p's residues ell-1 .. ell+alpha-1 (basis of q_{ell-1} P) to q_r
__device__ __forceinline__ u64 mdd_load(const MddFuse &f, const PrimeDev *pr, const KsTables &T, int L, int alpha,
                                        int logN, int p, int r, size_t n) {
    const int nb = alpha + 1, ell = f.ell;
    const u64 *up = f.U + (size_t)p * f.ustride;
    const u64 qi = pr[r].q;
    u64 acc = 0;
    for (int k = 0; k < nb; k++) {
        const u64 bk = k == 0 ? pr[ell - 1].q : pr[L + k - 1].q;
        const u64 y = up[((size_t)(ell - 1 + k) << logN) + n];  // [U_k (B/b_k)^-1 / t]_{b_k}: scaled by the inverse transform
        u64 v = mul_shoup(y, T.mdd_hat[((size_t)ell * nb + k) * L + r], qi);
        if (y > (bk - 1) / 2) v = sub_mod(v, T.mdd_B[(size_t)ell * L + r], qi);
        acc = add_mod(acc, v, qi);
    }
    return acc;
}

__device__ __forceinline__ void mdd_store(const MddFuse &f, const PrimeDev *pr, const KsTables &T, int L, int logN,
                                          int p, int r, size_t k, u64 v) {
    const PrimeDev P = pr[r];
    const u64 uv = f.U[(size_t)p * f.ustride + ((size_t)r << logN) + k];
    u64 res = mul_shoup(sub_mod(uv, mul_shoup(v, P.t_mod, P.t_mod_sh, P.q), P.q), T.mdd_Binv[(size_t)f.ell * L + r], P.q);
    if (!f.outp[0]) {
        f.out[(((size_t)p * (f.ell - 1) + r) << logN) + k] = res;
        return;
    }
    const size_t at = (((size_t)(p & 1) * (f.ell - 1) + r) << logN) + k;
    if (f.addp[p >> 1]) res = add_mod(res, f.addp[p >> 1][at], P.q);
    f.outp[p >> 1][at] = res;
}

// Load / store of the transforms: coefficient n of residue r (global prime g) of batch
// polynomial p in; value v at position k out, in [0, q), or (RAW) unreduced below 62q < 2^61.
struct PlainIO {
    static constexpr bool RAW = false;
    u64 *data;
    size_t stride;
    int logN;
    __device__ __forceinline__ u64 load(int p, int r, int, size_t n) const {
        return data[(size_t)p * stride + ((size_t)r << logN) + n];
    }
    __device__ __forceinline__ void store(int p, int r, int, size_t k, u64 v) const {
        data[(size_t)p * stride + ((size_t)r << logN) + k] = v;
    }
    __device__ __forceinline__ void skip(int, int, int, int, int, int) const {}
};

// out-of-place transform: residue r of polynomial p from src into dst
struct CopyIO {
    static constexpr bool RAW = false;
    const u64 *src;
    size_t sstride;
    u64 *dst;
    size_t dstride;
    int logN;
    __device__ __forceinline__ u64 load(int p, int r, int, size_t n) const {
        return src[(size_t)p * sstride + ((size_t)r << logN) + n];
    }
    __device__ __forceinline__ void store(int p, int r, int, size_t k, u64 v) const {
        dst[(size_t)p * dstride + ((size_t)r << logN) + k] = v;
    }
    __device__ __forceinline__ void skip(int, int, int, int, int, int) const {}
};

// one residue of polynomials at separate addresses in, contiguous residues out
struct GatherIO {
    static constexpr bool RAW = false;
    GatherSrc src;
    u64 *dst;
    int logN;
    __device__ __forceinline__ u64 load(int p, int, int, size_t n) const { return src.p[p][n]; }
    __device__ __forceinline__ void store(int p, int, int, size_t k, u64 v) const {
        dst[((size_t)p << logN) + k] = v;
    }
    __device__ __forceinline__ void skip(int, int, int, int, int, int) const {}
};

// ModUp (polynomial p = item nd + digit j, residue r of the extended basis): load the
// centred conversion of the digit's coefficient-form residues, store into
// y [item][nd][ell+alpha][N]; a digit's own residues (skipped by the transform) are
// copied from the input, which already holds them in NTT form
struct MuIO {
    static constexpr bool RAW = false;
    const u64 *xc;     // [item][ell][N] coefficient form
    const u64 *x_ntt;  // item i at x_ntt + i * xs, [ell][N] NTT domain
    size_t xs;
    u64 *y;
    int ell, alpha, nd, L, NP, logN;
    const PrimeDev *pr;
    KsTables T;
    __device__ __forceinline__ void store(int p, int r, int, size_t k, u64 v) const {
        y[(((size_t)p * (ell + alpha) + r) << logN) + k] = v;
    }
    // part `rank` of `cl`, by thread t of nt
    __device__ __forceinline__ void skip(int p, int r, int rank, int cl, int t, int nt) const {
        const int item = p / nd;
        const size_t n = (size_t)1 << logN, part = n / cl, k0 = (size_t)rank * part;
        const u64 *src = x_ntt + (size_t)item * xs + ((size_t)r << logN) + k0;
        u64 *dst = y + (((size_t)p * (ell + alpha) + r) << logN) + k0;
        for (size_t k = t; k < part / 2; k += nt) ((ulonglong2 *)dst)[k] = ((const ulonglong2 *)src)[k];
    }
};

// modulus switch: load the centred conversion of the last prime's residue, store the finish
struct MsIO {
    static constexpr bool RAW = true;
    MsFuse f;
    const PrimeDev *pr;
    KsTables T;
    int L, logN;
    __device__ __forceinline__ const u64 *operand(int p, int r) const {
        return (f.xp[0] ? f.xp[p] : f.x + (size_t)p * f.ell * ((size_t)1 << logN)) + ((size_t)r << logN);
    }
    __device__ __forceinline__ void skip(int, int, int, int, int, int) const {}
};

// ModDown: load the conversion of the alpha special residues, store the finish
struct MdIO {
    static constexpr bool RAW = true;
    MdFuse f;
    const PrimeDev *pr;
    KsTables T;
    int L, alpha, logN;
    __device__ __forceinline__ const u64 *operand(int p, int r) const {
        return f.U + (size_t)p * f.ustride + ((size_t)r << logN);
    }
    __device__ __forceinline__ void skip(int, int, int, int, int, int) const {}
};

// relinearise-and-drop ModDown: load the conversion from the q_{ell-1} P basis, store the finish
struct MddIO {
    static constexpr bool RAW = true;
    MddFuse f;
    const PrimeDev *pr;
    KsTables T;
    int L, alpha, logN;
    __device__ __forceinline__ const u64 *operand(int p, int r) const {
        return f.U + (size_t)p * f.ustride + ((size_t)r << logN);
    }
    __device__ __forceinline__ void skip(int, int, int, int, int, int) const {}
};

// ---------------------------------------------------------------- a thread's coefficients of a tile
// The forward kernels load K coefficients n0 + i dn (i < K) of one residue polynomial at a
// time and store K results k0 + i dk.  By default each goes through the functor's
// load / store; the fused conversions and finishes below take all K together, their
// per-tile constants loaded once and every global load of a step in flight at once.
template <int K, class IO>
__device__ __forceinline__ void load_n(const IO &io, int p, int r, int g, size_t n0, size_t dn, u64 (&v)[K]) {
#pragma unroll
    for (int i = 0; i < K; i++) v[i] = io.load(p, r, g, n0 + (size_t)i * dn);
}
template <int K, class IO>
__device__ __forceinline__ void store_n(const IO &io, int p, int r, int g, size_t k0, size_t dk, const u64 (&v)[K],
                                        const u64 (&)[K]) {
#pragma unroll
    for (int i = 0; i < K; i++) io.store(p, r, g, k0 + (size_t)i * dk, v[i]);
}
// The operand of a finish (the value whose switched-down remainder the transform makes), loaded
// ahead of its store: u[i] for position k0 + i dk.
template <int K, class IO>
__device__ __forceinline__ void operand_n(const IO &io, int p, int r, size_t k0, size_t dk, u64 (&u)[K]) {
    if constexpr (IO::RAW) {
        const u64 *x = io.operand(p, r);
#pragma unroll
        for (int i = 0; i < K; i++) u[i] = x[k0 + (size_t)i * dk];
    } else {
#pragma unroll
        for (int i = 0; i < K; i++) u[i] = 0;
    }
}

// A base conversion sum_k c_k f_k mod q of centred digits c_k = [y_k] in (-b_k / 2, b_k / 2).
// The inverse transform that makes the digits stores them as y_k + (b_k - 1) / 2 mod b_k
// (NttBatch::digits), so that c_k is that value less (b_k - 1) / 2 and the centring of every
// digit is one constant per target prime: with f_k in Montgomery form F_k = f_k 2^64 mod q and
// C = -sum_k ((b_k - 1) / 2) F_k mod q,
//   S = C + sum_k (y_k + (b_k - 1) / 2 mod b_k) F_k
// is summed exactly (digits and factors are stored split at 28 bits: three multiply-adds a
// product, at most 64 products) and reduced once, S 2^-64 mod q (Montgomery).
// S < m 2^(2 bits) + q < q 2^64 for m < 2^(63 - bits) terms of residues below 2^bits; the result
// stays below 2q, which the transform takes (the bounds are at bf_fwd, ntt_core.cuh).
// The digits of the next factor are loaded while this one's are multiplied.
// Taking the centring out of the sums (a comparison and a count per product before) and the
// factors and digits apart beforehand, with finishes of one combined reduction: ModDown with six
// special primes at N = 2^15 83 -> 66 ms over a batch of 16 encrypted query ciphertexts, ModUp
// 52 -> 44, relinearise-and-drop 17 -> 13; a batch of 16 residue polynomials at N = 2^14 34 -> 28 us.
template <int K, class FAC>
__device__ __forceinline__ void conv_sum(const u64 *y, size_t ystep, size_t dn, int m, u64 C, const PrimeDev &P,
                                         FAC fac, u64 (&v)[K]) {
    AccK s[K];
    uint2 d[K];
#pragma unroll
    for (int i = 0; i < K; i++) {
        s[i] = AccK{C, 0, C};
        d[i] = *(const uint2 *)(y + (size_t)i * dn);
    }
    for (int k = 0; k < m; k++) {
        uint2 nx[K];
        y += k + 1 < m ? ystep : 0;
#pragma unroll
        for (int i = 0; i < K; i++) nx[i] = *(const uint2 *)(y + (size_t)i * dn);
        const u64 F = __ldg(fac(k));
        const uint2 f = make_uint2((uint32_t)F, (uint32_t)(F >> 32));
        const uint32_t fs = f.x + f.y;
#pragma unroll
        for (int i = 0; i < K; i++) {
            mac_k(s[i], d[i], d[i].x + d[i].y, f, fs);
            d[i] = nx[i];
        }
    }
#pragma unroll
    for (int i = 0; i < K; i++) {
        const unsigned __int128 x = acc_value(s[i]);
        const u64 lo = (u64)x, mm = lo * P.qinv_neg;
        v[i] = (u64)(x >> 64) + __umul64hi(mm, P.q) + (lo != 0);
    }
}

template <int K>
__device__ __forceinline__ void load_n(const MuIO &io, int p, int, int g, size_t n0, size_t dn, u64 (&v)[K]) {
    const int item = p / io.nd, j = p - item * io.nd;
    const int lo = j * io.alpha, hi = min(lo + io.alpha, io.ell);
    const size_t N = (size_t)1 << io.logN, t0 = ((size_t)io.ell * io.L + lo) * io.NP + g;
    conv_sum(io.xc + ((size_t)item * io.ell + lo) * N + n0, N, dn, hi - lo, io.T.modup_c[t0], io.pr[g],
             [&](int k) { return io.T.modup_f + t0 + (size_t)k * io.NP; }, v);
}

template <int K>
__device__ __forceinline__ void load_n(const MdIO &io, int p, int r, int, size_t n0, size_t dn, u64 (&v)[K]) {
    const size_t N = (size_t)1 << io.logN;
    conv_sum(io.f.U + (size_t)p * io.f.ustride + (size_t)io.f.ell * N + n0, N, dn, io.alpha, io.T.md_c[r], io.pr[r],
             [&](int k) { return io.T.md_f + (size_t)k * io.L + r; }, v);
}

template <int K>
__device__ __forceinline__ void load_n(const MddIO &io, int p, int r, int, size_t n0, size_t dn, u64 (&v)[K]) {
    const size_t N = (size_t)1 << io.logN, t0 = (size_t)io.f.ell * (io.alpha + 1) * io.L + r;
    conv_sum(io.f.U + (size_t)p * io.f.ustride + (size_t)(io.f.ell - 1) * N + n0, N, dn, io.alpha + 1,
             io.T.mdd_c[(size_t)io.f.ell * io.L + r], io.pr[r],
             [&](int k) { return io.T.mdd_f + t0 + (size_t)k * io.L; }, v);
}

// the one digit of a modulus switch: c = d - (q_{ell-1} - 1) / 2, |c| < q_r as the chain is in
// decreasing order
template <int K>
__device__ __forceinline__ void load_n(const MsIO &io, int p, int r, int, size_t n0, size_t dn, u64 (&v)[K]) {
    const u64 up = io.pr[r].q - (io.pr[io.f.ell - 1].q - 1) / 2;
    const u64 *w = io.f.last + ((size_t)p << io.logN) + n0;  // already times t^-1
#pragma unroll
    for (int i = 0; i < K; i++) {
        const uint2 d = *(const uint2 *)(w + (size_t)i * dn);
        v[i] = ((u64)d.y << 28) + d.x + up;
    }
}

// x a + v b mod q for constants a, b (Shoup pairs), x < q and v < 2^61, in [0, q): the two quotients
// are subtracted together; x's part is below q + q x / 2^64, v's below q + q v / 2^64, the sum below 3q
__device__ __forceinline__ u64 mul2_shoup(u64 x, Shoup a, u64 v, Shoup b, u64 q) {
    const u64 h = __umul64hi(x, a.wp) + __umul64hi(v, b.wp);
    u64 r = x * a.w + v * b.w - h * q;
    if (r >= 2 * q) r -= 2 * q;
    return r >= q ? r - q : r;
}

// the finishes of ms_store, md_store and mdd_store for K positions of one residue, from the
// transform's unreduced values: (U - t v) B^-1 = U B^-1 + v (-t B^-1)
template <int K>
__device__ __forceinline__ void store_n(const MsIO &io, int p, int r, int, size_t k0, size_t dk, const u64 (&v)[K],
                                        const u64 (&u)[K]) {
    const MsFuse &f = io.f;
    const u64 q = io.pr[r].q;
    const Shoup qinv = io.T.ms_qinv[(size_t)f.ell * io.L + r], tq = io.T.ms_ntq[(size_t)f.ell * io.L + r];
    u64 *o = (f.outp[0] ? f.outp[p] : f.out + (size_t)p * (f.ell - 1) * ((size_t)1 << io.logN)) + ((size_t)r << io.logN);
#pragma unroll
    for (int i = 0; i < K; i++) o[k0 + (size_t)i * dk] = mul2_shoup(u[i], qinv, v[i], tq, q);
}

template <int K>
__device__ __forceinline__ void store_n(const MdIO &io, int p, int r, int, size_t k0, size_t dk, const u64 (&v)[K],
                                        const u64 (&u)[K]) {
    const MdFuse &f = io.f;
    const int job = p >> 1, c = p & 1;
    const u64 q = io.pr[r].q;
    const Shoup pinv = io.T.md_Pinv[r], tp = io.T.md_ntP[r];
    u64 res[K];
#pragma unroll
    for (int i = 0; i < K; i++) res[i] = mul2_shoup(u[i], pinv, v[i], tp, q);
    if (c < f.add_comps && f.add[job]) {
        const u64 *a = f.add[job] + (size_t)c * f.acomp + ((size_t)r << io.logN);
        const u64 gal = f.gal[job];
        u64 av[K];
#pragma unroll
        for (int i = 0; i < K; i++) {
            const size_t k = k0 + (size_t)i * dk;
            av[i] = a[(c == 0 && gal != 1) ? (size_t)galois_src((uint32_t)k, gal, io.logN) : k];
        }
#pragma unroll
        for (int i = 0; i < K; i++) res[i] = add_mod(res[i], av[i], q);
    }
    u64 *out = f.out[job] + (size_t)c * f.ocomp + ((size_t)r << io.logN);
#pragma unroll
    for (int i = 0; i < K; i++) out[k0 + (size_t)i * dk] = res[i];
}

template <int K>
__device__ __forceinline__ void store_n(const MddIO &io, int p, int r, int, size_t k0, size_t dk, const u64 (&v)[K],
                                        const u64 (&u)[K]) {
    const MddFuse &f = io.f;
    const u64 q = io.pr[r].q;
    const size_t n = (size_t)1 << io.logN;
    const Shoup binv = io.T.mdd_Binv[(size_t)f.ell * io.L + r], tb = io.T.mdd_ntB[(size_t)f.ell * io.L + r];
    u64 res[K];
#pragma unroll
    for (int i = 0; i < K; i++) res[i] = mul2_shoup(u[i], binv, v[i], tb, q);
    u64 *out;
    if (!f.outp[0]) {
        out = f.out + ((size_t)p * (f.ell - 1) + r) * n;
    } else {
        const size_t at = ((size_t)(p & 1) * (f.ell - 1) + r) * n;
        const u64 *add = f.addp[p >> 1];
        if (add) {
            u64 av[K];
#pragma unroll
            for (int i = 0; i < K; i++) av[i] = add[at + k0 + (size_t)i * dk];
#pragma unroll
            for (int i = 0; i < K; i++) res[i] = add_mod(res[i], av[i], q);
        }
        out = f.outp[p >> 1] + at;
    }
#pragma unroll
    for (int i = 0; i < K; i++) out[k0 + (size_t)i * dk] = res[i];
}


}  // namespace
