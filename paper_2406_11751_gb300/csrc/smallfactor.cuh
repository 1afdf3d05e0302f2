// Device-side pieces of the n x n steps of Algorithm alg_2 (Section 4) -- the Cholesky factorisation and
// R = R_1 R_s -- shared by their kernels (smallfactor.cu) and the persistent batched kernel (persist.cu).
#pragma once
#include "common.cuh"

namespace rpq {

// Upper Cholesky G = R^T R, row by row:
//   t_l = G[j][l] - sum_{k<j} R[k][j] R[k][l]  (l >= j),  R[j][j] = sqrt(t_j),  R[j][l] = t_l / R[j][j].
// G: n x n (ld ldg), n <= 128.  R: np x np row-major (ld np), padded with the identity; R_user
// (optional, n x n, ld n).  A pivot t_j that is not > 0 sets NOT_SPD with pivot j.
// Thread (part, l) = (tid / 128, tid % 128): each dot product is split over kCholParts threads
// (k = part, part + kCholParts, ...), so that all four schedulers' FP64 units work on it; the partial
// sums are subtracted in part order.  The upper triangle of G is copied into the working matrix first,
// so a step touches shared memory only; the square root is taken once per step.
constexpr int kCholParts = 8;
constexpr int kCholThreads = 128 * kCholParts;
// The factorisation by a CTA of NT threads (NT divides kCholThreads): thread tid plays the virtual
// threads tid, tid + NT, ... of the kCholThreads-thread layout above, so every sum is formed in the same
// order whatever NT.  csm: (np * np + kCholParts * np) doubles of shared memory.  Returns false on
// NOT_SPD (status set) or when info already holds a status.
template <int NT>
__device__ __forceinline__ bool cholesky_small(const double* __restrict__ G, int64_t ldg, int n, int np,
                                               double* __restrict__ R, double* __restrict__ R_user, int32_t* info,
                                               double* csm) {
    static_assert(kCholThreads % NT == 0, "the virtual-thread layout must tile the CTA");
    double* psum = csm + np * np;
    __shared__ double diag_s;
    __shared__ int fail_s;
    const int tid = threadIdx.x;
    for (int e = tid; e < np * np; e += NT) {
        const int r = e / np, c = e - r * np;
        csm[e] = (r <= c && c < n) ? G[static_cast<int64_t>(r) * ldg + c] : 0.0;
    }
    if (tid == 0) fail_s = -1;
    __syncthreads();
    for (int j = 0; j < n; ++j) {
#pragma unroll
        for (int vt = tid; vt < kCholThreads; vt += NT) {
            const int part = vt >> 7, l = vt & 127;
            if (l >= j && l < n) {
                double acc = 0.0;
                for (int k = part; k < j; k += kCholParts) acc += csm[k * np + j] * csm[k * np + l];
                psum[part * np + l] = acc;
            }
        }
        __syncthreads();
#pragma unroll
        for (int vt = tid; vt < kCholThreads; vt += NT) {
            const int part = vt >> 7, l = vt & 127;
            if (part == 0 && l > j && l < n) {
                double tl = csm[j * np + l];
#pragma unroll
                for (int q = 0; q < kCholParts; ++q) tl -= psum[q * np + l];
                csm[j * np + l] = tl;
            } else if (vt == 0) {
                double tj = csm[j * np + j];
#pragma unroll
                for (int q = 0; q < kCholParts; ++q) tj -= psum[q * np + j];
                if (!(tj > 0.0)) {
                    fail_s = j;
                } else {
                    diag_s = sqrt(tj);
                    csm[j * np + j] = diag_s;
                }
            }
        }
        __syncthreads();
        if (fail_s >= 0) break;
#pragma unroll
        for (int vt = tid; vt < kCholThreads; vt += NT) {
            const int part = vt >> 7, l = vt & 127;
            if (part == 0 && l > j && l < n) csm[j * np + l] /= diag_s;
        }
        __syncthreads();
    }
    if (fail_s >= 0) {
        if (tid == 0) set_status(info, RPCHOLQR_ERR_NOT_SPD, fail_s);
        return false;
    }
    for (int e = tid; e < np * np; e += NT) {
        const int r = e / np, c = e - r * np;
        double val = (r < n && c < n) ? csm[e] : (r == c ? 1.0 : 0.0);
        R[e] = val;
        if (R_user && r < n && c < n) R_user[r * n + c] = val;
    }
    return true;
}

// Entry (i, j) of R = R1 Rs for upper-triangular R1 (ld ld1) and Rs (ld lds): sum_{k=i..j} R1[i][k] Rs[k][j]
// in order of k, 0 below the diagonal.
__device__ __forceinline__ double triu_mul_entry(const double* __restrict__ R1, int64_t ld1,
                                                 const double* __restrict__ Rs, int64_t lds, int i, int j) {
    double acc = 0.0;
    for (int k = i; k <= j; ++k) acc += R1[i * ld1 + k] * Rs[k * lds + j];
    return acc;
}

}  // namespace rpq
