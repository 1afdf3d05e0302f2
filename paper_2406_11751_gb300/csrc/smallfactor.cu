// The small dense steps of Algorithm alg_2 (Section 4):
//   'Cholesky' G_1 = R_1^T R_1 -- n x n upper Cholesky, and R_1^{-1} with it where the split second pass wants it;
//   'recover'  R = R_1 R_s     -- product of upper-triangular factors, one CTA per row.
#include "smallfactor.cuh"

namespace rpq {

// ---- blocked Cholesky (algorithm and reasons in smallfactor.cuh), on many SMs --------------------------------
// R (np x np) is the work array; the factored diagonal blocks go to D (32 x 32 each) until k_chol_finish, because
// every CTA of a panel factors the diagonal block W_kk itself from R.  W (np x np, nullable): R^{-1}; the identity's
// columns take part as block columns j <= k, entry (r, c) of R^{-T} at W[c * np + r].
//   k_chol_panel   CTA c: factor W_kk, then block column k + 1 + c of R, or the identity's block column c - (nb - k - 1);
//   k_chol_trail   one warp per 16 x 8 tile of the updated blocks.
// Measured on GB300, Cholesky alone: n = 64 126 -> 81 us, 128 323 -> 198, 512 1.30 -> 0.92 ms, 1000 2.82 -> 2.02 ms; R^{-1}
// takes no further launches where a warp per column took 0.12 ms (n = 128) to 0.95 ms (512) and a blocked row solve of
// the identity 21 ms (1000).
__global__ void k_chol_init(const double* __restrict__ G, int64_t ldg, int n, int np, double* __restrict__ R,
                            double* __restrict__ W, const int32_t* info) {
    if (load_status(info) != 0) return;
    const int64_t e = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (e >= static_cast<int64_t>(np) * np) return;
    R[e] = chol_init_entry(G, ldg, n, np, e);
    if (W) W[e] = e / np == e % np ? 1.0 : 0.0;
}

__global__ void __launch_bounds__(128)
k_chol_panel(double* R, double* W, double* __restrict__ D, int n, int np, int k, int32_t* info) {
    __shared__ CholShared sh;
    if (cta_stopped(info)) return;
    const int tid = threadIdx.x, warp = tid >> 5, nb = (n + kCb - 1) / kCb;
    const int k0 = k * kCb, nk = n - k0 < kCb ? n - k0 : kCb;
    double* Rk = R + static_cast<int64_t>(k0) * np;
    chol_diag32(Rk + k0, np, nk, sh);
    if (blockIdx.x == 0) {
        for (int e = tid; e < kCb * kCb; e += 128) {
            const int i = e / kCb, j = e % kCb;
            D[static_cast<int64_t>(k) * kCb * kCb + e] = i <= j && j < nk ? sh.d[i][j] : 0.0;
        }
        if (tid == 0 && sh.bad < nk) set_status(info, RPCHOLQR_ERR_NOT_SPD, k0 + sh.bad);
    }
    if (sh.bad < nk) return;
    const int c = blockIdx.x, right = nb - k - 1;
    if (c < right) {
        const int j0 = (k + 1 + c) * kCb + 8 * warp;
        if (j0 < n) chol_rows8(Rk + j0, np, 1, nk, n - j0, false, 0, sh);
    } else if (W) {
        const int j = c - right, j0 = j * kCb + 8 * warp;      // (the last block's padding stays the identity)
        if (j0 < n) chol_rows8(W + static_cast<int64_t>(j0) * np + k0, 1, np, nk, n - j0, j == k, 8 * warp, sh);
    }
}

// Tiles of W_ij -= R_ki^T R_kj (k < i <= j) and, with W, of R^{-T}_ij -= R_ki^T R^{-T}_kj (j <= k < i): warp t of the
// launch takes 16-row tile t / nq and 8-column tile t % nq of the rows i > k; columns: R's right of block k, then
// R^{-T}'s up to block k.
__global__ void __launch_bounds__(128)
k_chol_trail(double* R, double* W, int n, int np, int k, const int32_t* info) {
    if (load_status(info) != 0) return;
    const int k0 = k * kCb, s0 = k0 + kCb, rest = n - s0, nr = (rest + 15) / 16, nqr = (rest + 7) / 8;
    const int nq = nqr + (W ? s0 / 8 : 0);
    const int t = blockIdx.x * 4 + (threadIdx.x >> 5);
    if (t >= nr * nq) return;
    const int r0 = 16 * (t / nq), qt = t % nq;
    const double* A = R + static_cast<int64_t>(k0) * np + s0 + r0;
    if (qt < nqr) {
        const int q0 = 8 * qt;
        if (r0 > q0 + 7) return;
        chol_trail_tile(A, np, R + static_cast<int64_t>(k0) * np + s0 + q0, np,
                        R + static_cast<int64_t>(s0 + r0) * np + s0 + q0, np, 1, kCb, rest - r0, rest - q0, true, r0, q0);
    } else {
        double* Wq = W + static_cast<int64_t>(8 * (qt - nqr)) * np;
        chol_trail_tile(A, np, Wq + k0, 1, Wq + s0 + r0, 1, np, kCb, rest - r0, 8, false, 0, 0);
    }
}

// The whole of it for one block, n <= 32: the same steps by one CTA in one launch instead of three (n = 1 14.5 -> 10.3 us, 16 25.0 -> 17.0).
__global__ void __launch_bounds__(128)
k_chol_one(const double* __restrict__ G, int64_t ldg, int n, int np, double* __restrict__ R, double* __restrict__ W,
           double* __restrict__ R_user, int32_t* info) {
    __shared__ CholShared sh;
    if (cta_stopped(info)) return;
    const int tid = threadIdx.x, j0 = 8 * (tid >> 5);
    chol_diag32(G, ldg, n, sh);
    if (sh.bad < n) {
        if (tid == 0) set_status(info, RPCHOLQR_ERR_NOT_SPD, sh.bad);
        return;
    }
    for (int e = tid; e < np * np; e += 128) {
        const int r = e / np, c = e - r * np;
        const bool in = r < n && c < n;
        const double v = in ? (r <= c ? sh.d[r][c] : 0.0) : (r == c ? 1.0 : 0.0);
        R[e] = v;
        if (R_user && in) R_user[r * n + c] = v;
        if (W && !in) W[e] = v;
    }
    if (W && j0 < n) chol_rows8(W + static_cast<int64_t>(j0) * np, 1, np, n, n - j0, true, j0, sh);
}

// The diagonal blocks into R, and (nullable) the n x n factor for the caller.
__global__ void k_chol_finish(double* __restrict__ R, const double* __restrict__ D, int n, int np, double* __restrict__ R_user,
                              const int32_t* info) {
    if (load_status(info) != 0) return;
    const int64_t e = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (e >= static_cast<int64_t>(n) * n) return;
    const int r = static_cast<int>(e / n), c = static_cast<int>(e - static_cast<int64_t>(r) * n);
    double v = R[static_cast<int64_t>(r) * np + c];
    if (r / kCb == c / kCb) {
        v = D[static_cast<int64_t>(r / kCb) * kCb * kCb + (r % kCb) * kCb + c % kCb];
        R[static_cast<int64_t>(r) * np + c] = v;
    }
    if (R_user) R_user[e] = v;
}

// R[i][j] = sum_{k=i..j} R1[i][k] Rs[k][j] for j >= i, 0 below; block i = row i.
__global__ void k_triu_mul(const double* __restrict__ R1, int64_t ld1, const double* __restrict__ Rs,
                           int64_t lds, int n, double* __restrict__ R, int64_t ldr,
                           const int32_t* info) {
    if (info && load_status(info) != 0) return;
    const int i = blockIdx.x;
    for (int j = threadIdx.x; j < n; j += blockDim.x)
        R[static_cast<int64_t>(i) * ldr + j] = triu_mul_entry(R1, ld1, Rs, lds, i, j);
}

// ---- host launchers ------------------------------------------------------------------------------
int cholesky_launches(int n) { return n <= kCb ? 1 : 2 * ((n + kCb - 1) / kCb) + 1; }

// R (np x np) = chol(G), identity padding; W (nullable, np x np): R^{-1}, identity padding; R_user (nullable, n x n).
// D: workspace of np x 32 doubles.
cudaError_t launch_cholesky(const double* G, int64_t ldg, int n, int np, double* R, double* W, double* D, double* R_user,
                            int32_t* info, cudaStream_t st) {
    if (n <= kCb) {
        k_chol_one<<<1, 128, 0, st>>>(G, ldg, n, np, R, W, R_user, info);
        return cudaGetLastError();
    }
    const int64_t tot = static_cast<int64_t>(np) * np;
    k_chol_init<<<static_cast<unsigned>((tot + 255) / 256), 256, 0, st>>>(G, ldg, n, np, R, W, info);
    const int nb = (n + kCb - 1) / kCb;
    for (int k = 0; k < nb; ++k) {
        const int ctas = nb - k - 1 + (W ? k + 1 : 0);
        k_chol_panel<<<ctas > 0 ? ctas : 1, 128, 0, st>>>(R, W, D, n, np, k, info);
        const int rest = n - (k + 1) * kCb;
        if (rest > 0) {
            const int tiles = (rest + 15) / 16 * ((rest + 7) / 8 + (W ? (k + 1) * kCb / 8 : 0));
            k_chol_trail<<<(tiles + 3) / 4, 128, 0, st>>>(R, W, n, np, k, info);
        }
    }
    k_chol_finish<<<static_cast<unsigned>((static_cast<int64_t>(n) * n + 255) / 256), 256, 0, st>>>(R, D, n, np, R_user,
                                                                                                 info);
    return cudaGetLastError();
}

void launch_triu_mul(const double* R1, int64_t ld1, const double* Rs, int64_t lds, int n, double* R,
                     int64_t ldr, const int32_t* info, cudaStream_t st) {
    const int threads = n < 32 ? 32 : (n > 256 ? 256 : (n + 31) / 32 * 32);
    k_triu_mul<<<n, threads, 0, st>>>(R1, ld1, Rs, lds, n, R, ldr, info);
}

}  // namespace rpq

// ---- choice of the split mode's second pass -------------------------------------------------------
// Q = A1 R1^{-1} as a split tensor-core product with the explicit inverse W = R1^{-1} is accurate to
// ~u times the product of the row bounds of A1 and the column bounds of W; its residual ||A - QR||
// grows with kappa(A1), while an FP64 row-wise substitution stays backward stable.  est =
// ||R1||_F ||W||_F / n lies between kappa(A1)/n and kappa(A1) (about 1.2 for well-sampled incoherent
// A).  The kernel writes two gate status words: the branch not taken gets kGateSkip (its kernels
// return at once), the taken one 0, and both carry an earlier error of info.
namespace rpq {

constexpr int kGateSkip = 1000;

// Sums of squares of R1's and W's upper triangles over rows b, b + gridDim.x, ...: CTA b's into part[2 b], part[2 b + 1].
__global__ void __launch_bounds__(256)
k_gate_norms(const double* __restrict__ R1, const double* __restrict__ W, int n, int np, double* __restrict__ part,
             const int32_t* info) {
    __shared__ double red[2][8];
    if (load_status(info) != 0) return;
    double a = 0.0, b = 0.0;
    for (int r = blockIdx.x; r < n; r += gridDim.x)
        for (int c = r + threadIdx.x; c < n; c += 256) {
            const double x = R1[static_cast<int64_t>(r) * np + c], y = W[static_cast<int64_t>(r) * np + c];
            a = fma(x, x, a);
            b = fma(y, y, b);
        }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_xor_sync(0xffffffffu, a, o);
        b += __shfl_xor_sync(0xffffffffu, b, o);
    }
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane == 0) { red[0][warp] = a; red[1][warp] = b; }
    __syncthreads();
    if (threadIdx.x < 2) {
        double s = 0.0;
        for (int w = 0; w < 8; ++w) s += red[threadIdx.x][w];
        part[2 * blockIdx.x + threadIdx.x] = s;
    }
}

// One warp: est <= tau as ||R1||_F^2 ||W||_F^2 <= (n tau)^2 (NaN takes the FP64 branch).
__global__ void __launch_bounds__(32)
k_pass2_gate(const double* __restrict__ part, int nparts, int n, double tau, const int32_t* info, int32_t* gate_split,
             int32_t* gate_fp64, int32_t* used_fp64) {
    const int lane = threadIdx.x, st = load_status(info);
    double a = 0.0, b = 0.0;
    if (st == 0)
        for (int i = lane; i < nparts; i += 32) {
            a += part[2 * i];
            b += part[2 * i + 1];
        }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_xor_sync(0xffffffffu, a, o);
        b += __shfl_xor_sync(0xffffffffu, b, o);
    }
    if (lane == 0) {
        const double lim = n * tau;
        const bool fp = !(a * b <= lim * lim);
        gate_split[0] = st ? st : (fp ? kGateSkip : 0);
        gate_fp64[0] = st ? st : (fp ? 0 : kGateSkip);
        gate_split[1] = gate_fp64[1] = -1;
        *used_fp64 = fp ? 1 : 0;
    }
}

// The first real error of the taken branch into info.
__global__ void k_gate_merge(int32_t* info, const int32_t* gate_split, const int32_t* gate_fp64) {
    if (threadIdx.x != 0 || load_status(info) != 0) return;
    const int32_t* g[2] = {gate_split, gate_fp64};
    for (int k = 0; k < 2; ++k)
        if (g[k][0] != 0 && g[k][0] != kGateSkip) {
            info[1] = g[k][1];
            info[0] = g[k][0];
            return;
        }
}

// part: workspace of 2 x 128 doubles.
void launch_pass2_gate(const double* R1, const double* W, int n, int np, double tau, double* part, const int32_t* info,
                       int32_t* gates, cudaStream_t st) {
    const int g = n < 128 ? (n + 7) / 8 : 128;   // a few rows per CTA
    k_gate_norms<<<g, 256, 0, st>>>(R1, W, n, np, part, info);
    k_pass2_gate<<<1, 32, 0, st>>>(part, g, n, tau, info, gates, gates + 2, gates + 4);
}
void launch_gate_merge(int32_t* info, const int32_t* gates, cudaStream_t st) {
    k_gate_merge<<<1, 32, 0, st>>>(info, gates, gates + 2);
}
}  // namespace rpq

namespace rpq {
// Shifted Cholesky-QR3's first stage (Fukaya et al. 2020, cited in Section 1): G += sigma I with
// sigma = 11 (m n + n (n + 1)) u trace(G), the trace summed in index order by one thread.
__global__ void k_scholqr3_shift(double* G, int64_t ldg, int n, int64_t m, const int32_t* info) {
    __shared__ double sigma;
    if (load_status(info) != 0) return;
    if (threadIdx.x == 0) {
        double tr = 0.0;
        for (int i = 0; i < n; ++i) tr += G[static_cast<int64_t>(i) * ldg + i];
        sigma = 11.0 * (static_cast<double>(m) * static_cast<double>(n) +
                        static_cast<double>(n) * static_cast<double>(n + 1)) * 0x1p-53 * tr;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += blockDim.x) G[static_cast<int64_t>(i) * ldg + i] += sigma;
}

void launch_scholqr3_shift(double* G, int64_t ldg, int n, int64_t m, const int32_t* info, cudaStream_t st) {
    k_scholqr3_shift<<<1, 256, 0, st>>>(G, ldg, n, m, info);
}
}  // namespace rpq
