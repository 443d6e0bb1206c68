// Encrypted-model multiply-accumulate on the integer pipe, for few query ciphertexts.
//
// The same sums as the tensor-core kernel (encmac.cu), from the same operands: per element,
// query ciphertext b and accumulator x the ciphertext products
//   (d0 R0, d0 R1 + d1 R0, d1 R1) summed over the baby steps j
// (Section 4.3's diagonal method with the diagonals encrypted, Section 8.3).  The tensor-core
// kernel pays per element for the digits of every diagonal, a 128-row operand whether or not it
// has 8 query ciphertexts, and a hand-over between its warps: about 12,000 cycles an element
// however small the matrix.  Here an element costs its masks and its products:
//   - the three sums of a ciphertext product from three residue products, the middle one as
//     (d0 + d1)(R0 + R1) less the outer two (Karatsuba), taken on the finished sums;
//   - a residue product of operands split at 28 bits (x = x1 2^28 + x0) from three 32 x 32 -> 64-bit
//     multiply-adds into 64-bit partial sums (x0 y0, x1 y1 and (x0 + x1)(y0 + y1)), folded into
//     128 bits every 16 baby steps and reduced mod q once per output.
// A block takes E elements, a tile of accumulators and a tile of query ciphertexts, and walks the
// baby steps in chunks of 32: all threads stage the chunk (c0 and R read as contiguous runs, the
// masks regenerated once per block, every operand split once), then thread (element, accumulator,
// pair of query ciphertexts, part of the chunk's baby steps) multiplies out of shared memory.
// Where the tiles are small the baby steps are divided over up to 16 threads, their 128-bit sums
// added by shuffles.  The bound is the integer pipe: mask generation for one query ciphertext,
// the multiply-adds from about four on.
#include <algorithm>

#include "internal.cuh"

namespace {

constexpr int IM_JC = 32;        // baby steps per chunk
// products between folds: with masks below 2^57 the middle product's sums of halves are below
// 2^30.2 and 2^29.6, sixteen of their products below 2^64
constexpr int IM_FOLD = 16;
constexpr int IM_THREADS = 128;  // threads per block at most
constexpr size_t IM_SMEM = 40 * 1024;
constexpr int IM_QT = 16;        // query ciphertexts per tile at most

struct IntMacArgs {
    const u64 *mac;       // [n_el][nm][nb16] diagonals' c0
    const uint32_t *idx;  // [nm][nb] model ciphertext index, ~0u = none
    const u64 *R;         // [n_el][nc][nq][64][2] rotations, split at 28 bits (rot_to_elements)
    u64 *acc;             // [nq][nm][3][n_el]
    size_t a_ct;
    int nm, nb, nb16, nq, ell, logN, nc;
    int logE, JP, mt, qt; // log2 of the elements per block, parts of the baby steps, tile sizes
    u64 seed;
    const PrimeDev *pr;
};

using u128 = unsigned __int128;
__device__ __forceinline__ void fold(u128 &t, AccK &a) {
    t += acc_value(a);
    a = AccK{0, 0, 0};
}
__device__ __forceinline__ u128 shfl_down_u128(u128 v, int d) {
    const u64 lo = __shfl_down_sync(0xffffffffu, (u64)v, d), hi = __shfl_down_sync(0xffffffffu, (u64)(v >> 64), d);
    return ((u128)hi << 64) | lo;
}

// QP query ciphertexts per thread (1 or 2)
template <int QP>
__global__ void __launch_bounds__(IM_THREADS, QP == 1 ? 6 : 4) k_enc_mac_int(const IntMacArgs P) {
    extern __shared__ uint4 sm_int[];
    const int E = 1 << P.logE, JP = P.JP;
    const size_t n_el = (size_t)P.ell << P.logN;
    const size_t e0 = (size_t)blockIdx.x << P.logE;
    const int x0 = blockIdx.y * P.mt, nx = min(P.mt, P.nm - x0);
    const int q0 = blockIdx.z * P.qt, nqt = min(P.qt, P.nq - q0);
    const int nqp = (P.qt + QP - 1) / QP, nqr = nqp * QP;  // threads' groups of query ciphertexts, rows of them
    // A chunk's operands, both components split at 28 bits in one 16-byte word, rows of its baby
    // steps (RS long: the padding spreads the JP-long groups that eight lanes read from different
    // rows over the banks): D [element][accumulator], Y [element][query ciphertext]
    const int RS = IM_JC + (JP & 7);
    uint4 *D = sm_int, *Y = D + (P.mt << P.logE) * RS;
    // the block's elements lie in one residue (E divides N)
    const int r = (int)(e0 >> P.logN);
    const uint32_t pos0 = (uint32_t)(e0 & ((1u << P.logN) - 1));
    const PrimeDev pd = P.pr[r];
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, w0 = tid >> 5, nw = nt >> 5;
    const int jp = tid % JP, slot = (tid / JP) % (P.mt * nqp), te = tid / JP / (P.mt * nqp);
    const int tx = slot % P.mt, tq = slot / P.mt;
    const bool active = te < E && tx < nx && tq * QP < nqt;
    AccK a[QP][3];
    u128 t[QP][3];
#pragma unroll
    for (int i = 0; i < QP; i++)
#pragma unroll
        for (int k = 0; k < 3; k++) {
            a[i][k] = AccK{0, 0, 0};
            t[i][k] = 0;
        }
    for (int j0 = 0; j0 < P.nb; j0 += IM_JC) {
        if (j0) __syncthreads();
        // one row per warp at a time, lane = baby step.  Rotations first (asynchronous copies),
        // the diagonals' masks while they arrive.
        const int jj = j0 + lane;
        {
            const u64 *src = P.R + ((e0 * P.nc + (jj >> 6)) * P.nq + q0 + w0) * 128 + (jj & 63) * 2;
            const size_t wrap = ((size_t)P.nc * P.nq - nqr) * 128;  // from one element's rows to the next's
            uint4 *dst = Y + w0 * RS + lane;
            for (int q = w0, left = (nqr << P.logE) - w0; left > 0; left -= nw, q += nw, src += nw * 128, dst += nw * RS) {
                while (q >= nqr) {
                    q -= nqr;
                    src += wrap;
                }
                if (q < nqt && jj < P.nb)
                    cp_async16(dst, src);
                else
                    *dst = make_uint4(0, 0, 0, 0);
            }
            cp_async_commit();
        }
        {
            const u64 *src = P.mac + (e0 * P.nm + x0 + w0) * P.nb16 + jj;
            const size_t wrap = (size_t)(P.nm - P.mt) * P.nb16;
            const uint32_t *id0 = P.idx + (size_t)x0 * P.nb + jj;
            uint4 *dst = D + w0 * RS + lane;
            uint32_t pos = pos0;
            for (int x = w0, left = (P.mt << P.logE) - w0; left > 0; left -= nw, x += nw, src += nw * P.nb16, dst += nw * RS) {
                while (x >= P.mt) {
                    x -= P.mt;
                    src += wrap;
                    pos++;
                }
                uint4 w = make_uint4(0, 0, 0, 0);
                if (x < nx && jj < P.nb) {
                    const u64 c0 = *src;
                    const uint32_t id = __ldg(id0 + x * P.nb);
                    if (id != ~0u) {
                        const u64 c1 = mask_at_lazy(mask_state(P.seed, r, pos, P.logN), id, pd);  // below 4q < 2^57
                        w = make_uint4((uint32_t)c0 & 0x0FFFFFFFu, (uint32_t)(c0 >> 28), (uint32_t)c1 & 0x0FFFFFFFu,
                                       (uint32_t)(c1 >> 28));
                    }
                }
                *dst = w;
            }
        }
        cp_async_wait<0>();
        __syncthreads();
        if (active) {
            const uint4 *d = D + (te * P.mt + tx) * RS + jp, *y = Y + (te * nqp + tq) * QP * RS + jp;
            // IM_FOLD products at a time (rows hold zeros past the last baby step)
            const int n = min(IM_FOLD, IM_JC / JP);
            for (int jb = 0; jb < IM_JC; jb += IM_FOLD * JP) {
#pragma unroll 2
                for (int i2 = 0; i2 < n; i2++, d += JP, y += JP) {
                    const uint4 dv = *d;
                    const uint32_t x0s = dv.x + dv.y, x1s = dv.z + dv.w;
                    const uint2 xs = make_uint2(dv.x + dv.z, dv.y + dv.w);
#pragma unroll
                    for (int i = 0; i < QP; i++) {
                        const uint4 yv = y[i * RS];
                        const uint32_t y0s = yv.x + yv.y, y1s = yv.z + yv.w;
                        mac_k(a[i][0], make_uint2(dv.x, dv.y), x0s, make_uint2(yv.x, yv.y), y0s);
                        mac_k(a[i][2], make_uint2(dv.z, dv.w), x1s, make_uint2(yv.z, yv.w), y1s);
                        mac_k(a[i][1], xs, x0s + x1s, make_uint2(yv.x + yv.z, yv.y + yv.w), y0s + y1s);
                    }
                }
#pragma unroll
                for (int i = 0; i < QP; i++)
#pragma unroll
                    for (int k = 0; k < 3; k++) fold(t[i][k], a[i][k]);
            }
        }
    }
    // the parts of the baby steps (JP consecutive lanes; every lane of the warp takes part)
    for (int d = JP / 2; d > 0; d >>= 1)
#pragma unroll
        for (int i = 0; i < QP; i++)
#pragma unroll
            for (int k = 0; k < 3; k++) t[i][k] += shfl_down_u128(t[i][k], d);
    // outputs through shared memory: E consecutive elements per (query ciphertext, accumulator, sum)
    __syncthreads();
    u64 *out = (u64 *)sm_int;  // [q][x][3][E]
    if (active && jp == 0)
#pragma unroll
        for (int i = 0; i < QP; i++) {
            const int q = tq * QP + i;
            if (q >= nqt) continue;
            const u128 t0 = t[i][0], t2 = t[i][2], t1 = t[i][1] - t0 - t2;
            u64 *o = out + (((q * P.mt + tx) * 3) << P.logE) + te;
            o[0] = reduce_words((u64)(t0 >> 64), (u64)t0, pd);
            o[E] = reduce_words((u64)(t1 >> 64), (u64)t1, pd);
            o[2 * E] = reduce_words((u64)(t2 >> 64), (u64)t2, pd);
        }
    __syncthreads();
    const int e = tid & (E - 1), nk = 3 * nx, step = nt >> P.logE;
    int k = tid >> P.logE, q = 0;
    while (k >= nk) {
        k -= nk;
        q++;
    }
    u64 *dst = P.acc + (size_t)q0 * P.a_ct + (size_t)x0 * 3 * n_el + e0 + e;
    while (q < nqt) {
        dst[(size_t)q * P.a_ct + (size_t)k * n_el] = out[((q * P.mt * 3 + k) << P.logE) + e];
        k += step;
        while (k >= nk) {
            k -= nk;
            q++;
        }
    }
}

}  // namespace

// Time of one element in SM nanoseconds, fitted to both kernels on a GB300 (the 7 launches of an
// encrypted model's matrices, N = 2^15, 64 to 1536 (accumulator, baby step) products, 1 to 64
// query ciphertexts): here 1.0 a product and tile of query ciphertexts (its mask) and 0.32 a
// product and query ciphertext; the tensor cores 2800 a tile of 16 accumulators and run of 256
// baby steps, 1930 a pass of 8 query ciphertexts and 0.8 a product.  Measured, ms here / there:
// 64 products 1.9 / 74.6 at 1, 6.5 / 74.6 at 8, 11.6 / 98 at 16; 1024-1536 products 23 / 87 at 1,
// 57 / 88 at 8, 100 / 127 at 16 (before the blocks were halved 173 / 155 at 24).
bool enc_mac_use_int(const std::vector<EncModel::MacMat> &mats, int nq) {
    double t_int = 0, t_tc = 0;
    for (const EncModel::MacMat &M : mats) {
        const double prod = (double)M.nm * M.nb;
        t_int += prod * ((nq + IM_QT - 1) / IM_QT + 0.32 * nq);
        t_tc += ((M.nm + 15) / 16) * ((M.nb + 255) / 256) * (2800.0 + 1930.0 * ((nq + 7) / 8)) + 0.8 * prod;
    }
    return t_int <= t_tc;
}

copse_status enc_mac_int(copse_ctx *c, const EncModel::MacMat &M, const u64 *R, int nq, u64 *acc, size_t a_ct,
                         u64 seed, cudaStream_t s) {
    if (nq <= 0 || M.nm <= 0 || M.nb <= 0) return COPSE_OK;
    IntMacArgs P;
    P.mac = M.c0;
    P.idx = M.idx;
    P.R = R;
    P.acc = acc;
    P.a_ct = a_ct;
    P.nm = M.nm;
    P.nb = M.nb;
    P.nb16 = mac_row(M.nb);
    P.nq = nq;
    P.ell = M.ell;
    P.logN = c->logN;
    P.nc = (M.nb + 63) / 64;
    P.seed = seed;
    P.pr = c->d_prime;
    // tiles: at most 16 query ciphertexts and 64 (accumulator, thread's query ciphertexts) slots,
    // evenly divided; then as many elements (up to 16) and parts of the baby steps (up to 16) as
    // fill the block.  Small blocks, so that the staging of some overlaps the products of others:
    // with 256 threads 5 query ciphertexts of a 252-branch model took 22.2 ms, with 128 14.7; 16 of
    // a 1008-branch model 111 and 100
    const int qp = nq > 1 ? 2 : 1;
    const int nqt = (nq + IM_QT - 1) / IM_QT;
    P.qt = (nq + nqt - 1) / nqt;
    const int qs = (P.qt + qp - 1) / qp;
    const int xmax = std::max(1, std::min({16, 64 / qs, 22 - qs * qp}));
    const int nmt = (M.nm + xmax - 1) / xmax;
    P.mt = (M.nm + nmt - 1) / nmt;
    const int slots = P.mt * qs;
    auto bytes = [&](int E, int JP) { return (size_t)E * (P.mt + qs * qp) * (IM_JC + (JP & 7)) * sizeof(uint4); };
    int E = 2;
    P.logE = 1;
    P.JP = 1;
    while (E < 16 && E * 2 * slots <= IM_THREADS && bytes(E * 2, 7) <= IM_SMEM) {
        E *= 2;
        P.logE++;
    }
    while (P.JP < 16 && E * slots * P.JP * 2 <= IM_THREADS && bytes(E, P.JP * 2) <= IM_SMEM) P.JP *= 2;
    const int threads = std::max(64, (E * slots * P.JP + 31) / 32 * 32);
    const size_t smem = std::max(bytes(E, P.JP), (size_t)E * 3 * P.mt * P.qt * sizeof(u64));
    const size_t n_el = (size_t)M.ell << c->logN;
    const dim3 grid((unsigned)(n_el / E), (unsigned)nmt, (unsigned)nqt);
    if (qp == 1)
        k_enc_mac_int<1><<<grid, threads, smem, s>>>(P);
    else
        k_enc_mac_int<2><<<grid, threads, smem, s>>>(P);
    LAUNCH_CHECK();
    return COPSE_OK;
}
