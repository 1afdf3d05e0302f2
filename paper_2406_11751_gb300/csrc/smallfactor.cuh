// Device-side pieces of the n x n steps of Algorithm alg_2 (Section 4) -- the Cholesky factorisation and
// R = R_1 R_s -- shared by their kernels (smallfactor.cu) and the persistent batched kernel (persist.cu).
//
// Cholesky G = R^T R, right-looking over 32 x 32 blocks.  R (np x np row-major) starts as G's upper triangle; step k:
//   chol_diag32   the diagonal block W_kk = R_kk^T R_kk (four warps, rows in registers, one barrier per column);
//   chol_rows8    R_kj = R_kk^{-T} W_kj, eight columns per warp (forward substitution);
//   chol_trail    W_ij -= R_ki^T R_kj, k < i <= j.
// The same row operations applied to the identity give R^{-T}: its blocks take part as further columns
// (stored transposed, so that the array ends as R^{-1}), which costs no further steps of the chain.
// Every element sees the same operations in the same order whatever the launch shape, so one CTA alone gives
// the bits of the many-CTA form.
//
// Bound: the chain of columns; the pivot's root and its reciprocal are formed in 64-bit fixed point (common.cuh).
#pragma once
#include "common.cuh"

namespace rpq {

constexpr int kCb = 32;               // Cholesky block
constexpr int kCbLd = kCb + 1;

// root = sqrt(x) and inv = 1 / sqrt(x) for x > 0: y (1 + h) as well as the root (fixed_root); the plain operations outside
// its range.
__device__ __forceinline__ void root_and_inverse(double x, double& root, double& inv) {
    if (root_in_range(x)) {
        const FixedRoot r = fixed_root(x);
        root = fixed_root_value(r);
        const unsigned long long y = r.Y >> 1;   // Q63
        inv = from_q63(y + static_cast<unsigned long long>(__mul64hi(static_cast<long long>(y), r.h << 3)), -r.k / 2);
    } else {
        root = sqrt(x);
        inv = 1.0 / root;
    }
}

struct CholShared {
    double d[kCb][kCbLd];    // R_kk (upper, its nk rows), rows written as they are finished
    double inv[kCb];         // 1 / diag
    int bad;                 // first pivot that is not > 0, or kCb
};

// The diagonal block (nk x nk, upper, entry (0, 0) at A, ld lda) into sh by the first 128 threads of the CTA.  Warp w
// holds rows w, w + 4, ... (lane = column); the warp that owns row i finishes it and hands it to the others.
// Every thread of the CTA calls this; barrier 3 joins the four warps.
__device__ __forceinline__ void chol_diag32(const double* A, int64_t lda, int nk, CholShared& sh) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) sh.bad = kCb;
    __syncthreads();
    if (warp < 4) {
        double a[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int r = 4 * u + warp;
            a[u] = (r < nk && lane < nk && r <= lane) ? A[static_cast<int64_t>(r) * lda + lane] : (r == lane ? 1.0 : 0.0);
        }
#pragma unroll
        for (int i = 0; i < kCb; ++i) {
            if (i == nk) break;   // (a short block's padding is never read)
            if (warp == (i & 3)) {
                const double piv = __shfl_sync(0xffffffffu, a[i >> 2], i);
                double root = 1.0, inv = 1.0;
                if (piv > 0.0) root_and_inverse(piv, root, inv);
                else if (lane == 0 && i < sh.bad) sh.bad = i;      // (one warp at a time)
                const double v = lane == i ? root : a[i >> 2] * inv;
                if (lane >= i) sh.d[i][lane] = v;
                if (lane == i) sh.inv[i] = inv;
            }
            asm volatile("bar.sync 3, 128;\n" ::: "memory");
            if (i + 1 < kCb) {
                const double x = -sh.d[i][lane];
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    if (4 * u + 3 <= i) continue;                    // (every row of this u is finished)
                    const int r = 4 * u + warp;
                    if (r > i && r <= lane) a[u] = fma(sh.d[i][r], x, a[u]);
                }
            }
        }
    }
    __syncthreads();
}

// One warp: eight columns of R_kk^{-T} B, in place.  Entry (r, c) of B at B[r * sr + c * sc]; nk rows, ncol columns.
// ident: B is the identity's columns c0 .. (its entries are not read).
__device__ __forceinline__ void chol_rows8(double* B, int64_t sr, int64_t sc, int nk, int ncol, bool ident, int c0,
                                           const CholShared& sh) {
    const int lane = threadIdx.x & 31, col = lane >> 2, rr = lane & 3;   // rows rr, rr + 4, ...
    double* Bc = B + col * sc;
    double a[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        const int r = 4 * u + rr;
        a[u] = ident ? (r == c0 + col ? 1.0 : 0.0) : (r < nk && col < ncol) ? Bc[r * sr] : 0.0;
    }
#pragma unroll
    for (int i = 0; i < kCb; ++i) {
        if (i >= nk) break;
        const double x = __shfl_sync(0xffffffffu, a[i >> 2] * sh.inv[i], (lane & ~3) | (i & 3));
        if (rr == (i & 3)) a[i >> 2] = x;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            if (4 * u + 3 <= i) continue;
            const int r = 4 * u + rr;
            if (r > i && r < nk) a[u] = fma(-sh.d[i][r], x, a[u]);
        }
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        const int r = 4 * u + rr;
        if (r < nk && col < ncol) Bc[r * sr] = a[u];
    }
}

// One warp: a 16 x 8 tile of O -= A^T B over nk <= 32 terms.  Entry (p, r) of A at A[p * np + r], (p, q) of B at
// B[p * sp + q * sq], (r, q) of O at O[r * sr + q * sq]; nr, nq valid rows and columns; upper: only r0 + r <= q0 + q.
// Two partial sums (even and odd terms) per entry.
__device__ __forceinline__ void chol_trail_tile(const double* A, int np, const double* B, int64_t sp, double* O, int64_t sr,
                                                int64_t sq, int nk, int nr, int nq, bool upper, int r0, int q0) {
    const int lane = threadIdx.x & 31, q = lane & 7;
#pragma unroll
    for (int h = 0; h < 4; ++h) {
        const int r = (lane >> 3) + 4 * h;
        if (r < nr && q < nq && (!upper || r0 + r <= q0 + q)) {
            const double *ap = A + r, *bp = B + q * sq;
            double s0 = 0.0, s1 = 0.0;
#pragma unroll 8
            for (int p = 0; p + 1 < nk; p += 2) {
                s0 = fma(ap[p * np], bp[p * sp], s0);
                s1 = fma(ap[(p + 1) * np], bp[(p + 1) * sp], s1);
            }
            if (nk & 1) s0 = fma(ap[(nk - 1) * np], bp[(nk - 1) * sp], s0);
            O[r * sr + q * sq] -= s0 + s1;
        }
    }
}

// Entry e of the working array: G's upper triangle, zero below, identity padding.
__device__ __forceinline__ double chol_init_entry(const double* G, int64_t ldg, int n, int np, int64_t e) {
    const int r = static_cast<int>(e / np), c = static_cast<int>(e - static_cast<int64_t>(r) * np);
    return (r >= n || c >= n) ? (r == c ? 1.0 : 0.0) : (r <= c ? G[static_cast<int64_t>(r) * ldg + c] : 0.0);
}

// The factorisation by one CTA of NT threads (a multiple of 128): R (np x np, identity padding) of G (n x n, ld ldg).
// Returns false on NOT_SPD (status set).
template <int NT>
__device__ __forceinline__ bool cholesky_one_cta(const double* G, int64_t ldg, int n, int np, double* R, int32_t* info,
                                                 CholShared& sh) {
    constexpr int NW = NT / 32;
    const int tid = threadIdx.x, warp = tid >> 5;
    for (int e = tid; e < np * np; e += NT) R[e] = chol_init_entry(G, ldg, n, np, e);
    for (int k0 = 0; k0 < n; k0 += kCb) {
        const int nk = n - k0 < kCb ? n - k0 : kCb;
        double* Rk = R + static_cast<int64_t>(k0) * np;
        __syncthreads();
        chol_diag32(Rk + k0, np, nk, sh);
        if (sh.bad < nk) {
            if (tid == 0) set_status(info, RPCHOLQR_ERR_NOT_SPD, k0 + sh.bad);
            return false;
        }
        for (int e = tid; e < kCb * kCb; e += NT) {
            const int i = e / kCb, j = e % kCb;
            if (i <= j && j < nk) Rk[static_cast<int64_t>(i) * np + k0 + j] = sh.d[i][j];
        }
        const int rest = n - k0 - nk;
        for (int c = 8 * warp; c < rest; c += 8 * NW)
            chol_rows8(Rk + k0 + nk + c, np, 1, nk, rest - c, false, 0, sh);
        __syncthreads();
        const int nr = (rest + 15) / 16, nq = (rest + 7) / 8;
        for (int t = warp; t < nr * nq; t += NW) {
            const int r0 = 16 * (t / nq), q0 = 8 * (t % nq);
            if (r0 > q0 + 7) continue;
            chol_trail_tile(Rk + k0 + nk + r0, np, Rk + k0 + nk + q0, np,
                            R + static_cast<int64_t>(k0 + nk + r0) * np + k0 + nk + q0, np, 1, nk, rest - r0, rest - q0, true,
                            r0, q0);
        }
    }
    __syncthreads();
    return true;
}

// Entry (i, j) of R = R1 Rs for upper-triangular R1 (ld ld1) and Rs (ld lds): sum_{k=i..j} R1[i][k] Rs[k][j], four
// partial sums (k = i, i + 1, i + 2, i + 3 mod 4), 0 below the diagonal.
__device__ __forceinline__ double triu_mul_entry(const double* __restrict__ R1, int64_t ld1,
                                                 const double* __restrict__ Rs, int64_t lds, int i, int j) {
    double s[4] = {0.0, 0.0, 0.0, 0.0};
    const double *a = R1 + i * ld1, *b = Rs + j;
    int k = i;
#pragma unroll 2
    for (; k + 3 <= j; k += 4) {
#pragma unroll
        for (int u = 0; u < 4; ++u) s[u] = fma(a[k + u], b[(k + u) * lds], s[u]);
    }
    if (k <= j) s[0] = fma(a[k], b[k * lds], s[0]);
    if (k + 1 <= j) s[1] = fma(a[k + 1], b[(k + 1) * lds], s[1]);
    if (k + 2 <= j) s[2] = fma(a[k + 2], b[(k + 2) * lds], s[2]);
    return (s[0] + s[1]) + (s[2] + s[3]);
}

}  // namespace rpq
