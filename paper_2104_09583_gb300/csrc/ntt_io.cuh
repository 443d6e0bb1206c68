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

// Load / store of the forward cluster transform: coefficient n of residue r (global
// prime g) of batch polynomial p in; NTT-domain value v (in [0, q)) at position k out.
struct PlainIO {
    u64 *data;
    size_t stride;
    int logN;
    __device__ __forceinline__ u64 load(int p, int r, int, size_t n) const {
        return data[(size_t)p * stride + ((size_t)r << logN) + n];
    }
    __device__ __forceinline__ void store(int p, int r, int, size_t k, u64 v) const {
        data[(size_t)p * stride + ((size_t)r << logN) + k] = v;
    }
    __device__ __forceinline__ void skip(int, int, int, int) const {}
};

// out-of-place transform: residue r of polynomial p from src into dst
struct CopyIO {
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
    __device__ __forceinline__ void skip(int, int, int, int) const {}
};

// one residue of polynomials at separate addresses in, contiguous residues out
struct GatherIO {
    GatherSrc src;
    u64 *dst;
    int logN;
    __device__ __forceinline__ u64 load(int p, int, int, size_t n) const { return src.p[p][n]; }
    __device__ __forceinline__ void store(int p, int, int, size_t k, u64 v) const {
        dst[((size_t)p << logN) + k] = v;
    }
    __device__ __forceinline__ void skip(int, int, int, int) const {}
};

// ModUp (polynomial p = item nd + digit j, residue r of the extended basis): load the
// centred conversion of the digit's coefficient-form residues, store into
// y [item][nd][ell+alpha][N]; a digit's own residues (skipped by the transform) are
// copied from the input, which already holds them in NTT form
struct MuIO {
    const u64 *xc;     // [item][ell][N] coefficient form
    const u64 *x_ntt;  // item i at x_ntt + i * xs, [ell][N] NTT domain
    size_t xs;
    u64 *y;
    int ell, alpha, nd, L, NP, logN;
    const PrimeDev *pr;
    KsTables T;
    __device__ __forceinline__ u64 load(int p, int, int g, size_t n) const {
        const int item = p / nd, j = p - item * nd;
        const int lo = j * alpha, hi = min(lo + alpha, ell);
        const u64 qg = pr[g].q;
        const u64 *x = xc + (size_t)item * ell * ((size_t)1 << logN);
        u64 acc = 0;
        for (int i = lo; i < hi; i++) {
            const u64 qi = pr[i].q;
            const u64 v = x[((size_t)i << logN) + n];  // already times modup_inv (inverse transform's scale)
            const size_t ti = ((size_t)ell * L + i) * NP + g;
            u64 w = mul_shoup(v, T.modup_hat[ti], qg);
            if (v > (qi - 1) / 2) w = sub_mod(w, T.modup_qhat[ti], qg);
            acc = add_mod(acc, w, qg);
        }
        return acc;
    }
    __device__ __forceinline__ void store(int p, int r, int, size_t k, u64 v) const {
        y[(((size_t)p * (ell + alpha) + r) << logN) + k] = v;
    }
    __device__ __forceinline__ void skip(int p, int r, int rank, int cl) const {
        const int item = p / nd;
        const size_t n = (size_t)1 << logN, part = n / cl, k0 = (size_t)rank * part;
        const u64 *src = x_ntt + (size_t)item * xs + ((size_t)r << logN) + k0;
        u64 *dst = y + (((size_t)p * (ell + alpha) + r) << logN) + k0;
        for (size_t k = threadIdx.x; k < part / 2; k += blockDim.x) ((ulonglong2 *)dst)[k] = ((const ulonglong2 *)src)[k];
    }
};

// modulus switch: load the centred conversion of the last prime's residue, store the finish
struct MsIO {
    MsFuse f;
    const PrimeDev *pr;
    KsTables T;
    int L, logN;
    __device__ __forceinline__ u64 load(int p, int r, int, size_t n) const {
        const u64 ql = pr[f.ell - 1].q;
        const u64 w = f.last[((size_t)p << logN) + n];  // already times t^-1 (inverse transform's scale)
        // |centred w| < q_{ell-1}/2 < q_r: the chain is in decreasing order
        return w > (ql - 1) / 2 ? pr[r].q - (ql - w) : w;
    }
    __device__ __forceinline__ void store(int p, int r, int, size_t k, u64 v) const {
        ms_store(f, pr, T, L, logN, p, r, k, v);
    }
    __device__ __forceinline__ void skip(int, int, int, int) const {}
};

// ModDown: load the conversion of the alpha special residues, store the finish
struct MdIO {
    MdFuse f;
    const PrimeDev *pr;
    KsTables T;
    int L, alpha, logN;
    __device__ __forceinline__ u64 load(int p, int r, int, size_t n) const {
        const u64 *up = f.U + (size_t)p * f.ustride;
        const u64 qi = pr[r].q;
        u64 acc = 0;
        for (int k = 0; k < alpha; k++) {
            const u64 pk = pr[L + k].q;
            const u64 y = up[((size_t)(f.ell + k) << logN) + n];  // already times md_inv[k] (inverse transform's scale)
            u64 v = mul_shoup(y, T.md_hat[(size_t)k * L + r], qi);
            if (y > (pk - 1) / 2) v = sub_mod(v, T.md_P[r], qi);
            acc = add_mod(acc, v, qi);
        }
        return acc;
    }
    __device__ __forceinline__ void store(int p, int r, int, size_t k, u64 v) const {
        md_store(f, pr, T, logN, p, r, k, v);
    }
    __device__ __forceinline__ void skip(int, int, int, int) const {}
};

// relinearise-and-drop ModDown: load the conversion from the q_{ell-1} P basis, store the finish
struct MddIO {
    MddFuse f;
    const PrimeDev *pr;
    KsTables T;
    int L, alpha, logN;
    __device__ __forceinline__ u64 load(int p, int r, int, size_t n) const {
        return mdd_load(f, pr, T, L, alpha, logN, p, r, n);
    }
    __device__ __forceinline__ void store(int p, int r, int, size_t k, u64 v) const {
        mdd_store(f, pr, T, L, logN, p, r, k, v);
    }
    __device__ __forceinline__ void skip(int, int, int, int) const {}
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
__device__ __forceinline__ void store_n(const IO &io, int p, int r, int g, size_t k0, size_t dk, const u64 (&v)[K]) {
#pragma unroll
    for (int i = 0; i < K; i++) io.store(p, r, g, k0 + (size_t)i * dk, v[i]);
}

// A base conversion sum_k [y_k]_centred * f_k mod q as one lazy sum: with f_k in Montgomery form
// F_k = f_k 2^64 mod q and C = (-c) 2^64 mod q for the correction c that every centred negative
// digit takes (the product of the basis, the same for all of them),
// S = sum_k y_k F_k + #{k: y_k > (b_k - 1) / 2} C is summed exactly (the products split at 28 bits,
// three multiply-adds each, at most 64 of them) and reduced once, S 2^-64 mod q (Montgomery).
// S < m 2^(2 bits) + m q < q 2^64 for m < 2^(63 - bits) terms of residues below 2^bits.
struct ConvSum {
    AccK a;
    uint32_t neg;
};
template <int K>
__device__ __forceinline__ void conv_term(ConvSum (&s)[K], const u64 (&y)[K], u64 F, u64 half) {
    const uint2 f = split_k(F);
    const uint32_t fs = f.x + f.y;
#pragma unroll
    for (int i = 0; i < K; i++) {
        const uint2 v = split_k(y[i]);
        mac_k(s[i].a, v, v.x + v.y, f, fs);
        s[i].neg += y[i] > half;
    }
}
template <int K>
__device__ __forceinline__ void conv_reduce(const ConvSum (&s)[K], u64 C, const PrimeDev &P, u64 (&v)[K]) {
#pragma unroll
    for (int i = 0; i < K; i++) {
        const unsigned __int128 x = acc_value(s[i].a) + (u64)s[i].neg * C;
        v[i] = mont_reduce(Acc128{(u64)x, (u64)(x >> 64)}, P);
    }
}

template <int K>
__device__ __forceinline__ void load_n(const MuIO &io, int p, int, int g, size_t n0, size_t dn, u64 (&v)[K]) {
    const int item = p / io.nd, j = p - item * io.nd;
    const int lo = j * io.alpha, hi = min(lo + io.alpha, io.ell);
    const u64 *x = io.xc + (size_t)item * io.ell * ((size_t)1 << io.logN) + n0;
    ConvSum s[K];
#pragma unroll
    for (int i = 0; i < K; i++) s[i] = ConvSum{AccK{0, 0, 0}, 0};
    for (int i = lo; i < hi; i++) {
        const size_t ti = ((size_t)io.ell * io.L + i) * io.NP + g;
        const u64 *xi = x + ((size_t)i << io.logN);
        u64 y[K];
#pragma unroll
        for (int k = 0; k < K; k++) y[k] = xi[(size_t)k * dn];  // already times modup_inv (the inverse transform's scale)
        conv_term(s, y, io.T.modup_hat_m[ti], (io.pr[i].q - 1) / 2);
    }
    conv_reduce(s, io.T.modup_negq_m[((size_t)io.ell * io.L + lo) * io.NP + g], io.pr[g], v);
}

template <int K>
__device__ __forceinline__ void load_n(const MdIO &io, int p, int r, int, size_t n0, size_t dn, u64 (&v)[K]) {
    const u64 *up = io.f.U + (size_t)p * io.f.ustride + ((size_t)io.f.ell << io.logN) + n0;
    const u64 C = io.T.md_negP_m[r];
    ConvSum s[K];
#pragma unroll
    for (int i = 0; i < K; i++) s[i] = ConvSum{AccK{0, 0, 0}, 0};
    for (int k = 0; k < io.alpha; k++) {
        const u64 *yk = up + ((size_t)k << io.logN);
        u64 y[K];
#pragma unroll
        for (int i = 0; i < K; i++) y[i] = yk[(size_t)i * dn];  // already times md_inv[k] (the inverse transform's scale)
        conv_term(s, y, io.T.md_hat_m[(size_t)k * io.L + r], (io.pr[io.L + k].q - 1) / 2);
    }
    conv_reduce(s, C, io.pr[r], v);
}

template <int K>
__device__ __forceinline__ void load_n(const MddIO &io, int p, int r, int, size_t n0, size_t dn, u64 (&v)[K]) {
    const int ell = io.f.ell, nb = io.alpha + 1;
    const u64 *up = io.f.U + (size_t)p * io.f.ustride + ((size_t)(ell - 1) << io.logN) + n0;
    const u64 C = io.T.mdd_negB_m[(size_t)ell * io.L + r];
    ConvSum s[K];
#pragma unroll
    for (int i = 0; i < K; i++) s[i] = ConvSum{AccK{0, 0, 0}, 0};
    for (int k = 0; k < nb; k++) {
        const u64 bk = k == 0 ? io.pr[ell - 1].q : io.pr[io.L + k - 1].q;
        const u64 *yk = up + ((size_t)k << io.logN);
        u64 y[K];
#pragma unroll
        for (int i = 0; i < K; i++) y[i] = yk[(size_t)i * dn];  // scaled by the inverse transform
        conv_term(s, y, io.T.mdd_hat_m[((size_t)ell * nb + k) * io.L + r], (bk - 1) / 2);
    }
    conv_reduce(s, C, io.pr[r], v);
}

template <int K>
__device__ __forceinline__ void load_n(const MsIO &io, int p, int r, int, size_t n0, size_t dn, u64 (&v)[K]) {
    const u64 ql = io.pr[io.f.ell - 1].q, qr = io.pr[r].q, half = (ql - 1) / 2;
    const u64 *w = io.f.last + ((size_t)p << io.logN) + n0;  // already times t^-1
#pragma unroll
    for (int i = 0; i < K; i++) {
        const u64 x = w[(size_t)i * dn];
        v[i] = x > half ? qr - (ql - x) : x;  // |centred x| < q_{ell-1} / 2 < q_r
    }
}

// the finishes of ms_store, md_store and mdd_store for K positions of one residue
template <int K>
__device__ __forceinline__ void store_n(const MsIO &io, int p, int r, int, size_t k0, size_t dk, const u64 (&v)[K]) {
    const MsFuse &f = io.f;
    const u64 q = io.pr[r].q;
    const Shoup tm{io.pr[r].t_mod, io.pr[r].t_mod_sh}, qinv = io.T.ms_qinv[(size_t)f.ell * io.L + r];
    const u64 *x = (f.xp[0] ? f.xp[p] : f.x + (size_t)p * f.ell * ((size_t)1 << io.logN)) + ((size_t)r << io.logN);
    u64 *o = (f.outp[0] ? f.outp[p] : f.out + (size_t)p * (f.ell - 1) * ((size_t)1 << io.logN)) + ((size_t)r << io.logN);
    u64 xv[K];
#pragma unroll
    for (int i = 0; i < K; i++) xv[i] = x[k0 + (size_t)i * dk];
#pragma unroll
    for (int i = 0; i < K; i++) o[k0 + (size_t)i * dk] = mul_shoup(sub_mod(xv[i], mul_shoup(v[i], tm, q), q), qinv, q);
}

template <int K>
__device__ __forceinline__ void store_n(const MdIO &io, int p, int r, int, size_t k0, size_t dk, const u64 (&v)[K]) {
    const MdFuse &f = io.f;
    const int job = p >> 1, c = p & 1;
    const u64 q = io.pr[r].q;
    const Shoup tm{io.pr[r].t_mod, io.pr[r].t_mod_sh}, pinv = io.T.md_Pinv[r];
    const u64 *U = f.U + (size_t)p * f.ustride + ((size_t)r << io.logN);
    u64 res[K];
#pragma unroll
    for (int i = 0; i < K; i++) res[i] = U[k0 + (size_t)i * dk];
#pragma unroll
    for (int i = 0; i < K; i++) res[i] = mul_shoup(sub_mod(res[i], mul_shoup(v[i], tm, q), q), pinv, q);
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
__device__ __forceinline__ void store_n(const MddIO &io, int p, int r, int, size_t k0, size_t dk, const u64 (&v)[K]) {
    const MddFuse &f = io.f;
    const u64 q = io.pr[r].q;
    const size_t n = (size_t)1 << io.logN;
    const Shoup tm{io.pr[r].t_mod, io.pr[r].t_mod_sh}, binv = io.T.mdd_Binv[(size_t)f.ell * io.L + r];
    const u64 *U = f.U + (size_t)p * f.ustride + ((size_t)r << io.logN);
    u64 res[K];
#pragma unroll
    for (int i = 0; i < K; i++) res[i] = U[k0 + (size_t)i * dk];
#pragma unroll
    for (int i = 0; i < K; i++) res[i] = mul_shoup(sub_mod(res[i], mul_shoup(v[i], tm, q), q), binv, q);
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
