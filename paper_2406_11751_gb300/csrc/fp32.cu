// FP32 mode: the two passes of Algorithm alg_2 in single precision, for single-precision Krylov /
// LOBPCG users (A, Q, R stored as float).  The sample, the Householder R_s and the Cholesky factor R1
// stay in FP64 (they are small, and their stability needs it: Section 4 keeps R_s^{-1} applied to the
// ill-conditioned A); the m-row work runs on the FP32 FMA pipe (~70 TFLOP/s on GB300, against ~1 for
// FP64):
//
//   k_prep_f32       T32 = float(T) padded with the identity, rinv32 = 1 / diag(T32);
//   k_rowsolve_f32   Y = X T^{-1} row by row (Section 2.1: each row of A_1 is a triangular solve with
//                    R_s), rows in shared memory, left-looking over 32-column blocks: the off-diagonal part of a
//                    block as a register-tiled product, the 32 x 32 diagonal block by forward substitution;
//   k_syrk_f32       per-range partials of G = A_1^T A_1 over 64 x 64 upper tiles, FP32 products summed
//                    in FP32 over 8 rows, those sums added without error into FP32 pairs.
#include "common.cuh"

namespace rpq {

constexpr int kF32Blk = 32;      // column block of the row solves
constexpr int kSyrkRows = 8;     // rows summed in plain FP32
constexpr int kSyrkSpillRows = 256;   // rows between looks at the pairs' size

__host__ __device__ constexpr int pad32(int n) { return (n + 31) / 32 * 32; }

// T32 (np32 x np32 row-major): float(T) on and above the diagonal of the leading n x n block, 0 below,
// identity in the padding.  A diagonal that is not a normal FP32 number sets `fail_status`.
__global__ void k_prep_f32(const double* __restrict__ T, int64_t ldt, int n, int np32, float* __restrict__ T32,
                           float* __restrict__ rinv32, int fail_status, int32_t* info) {
    if (load_status(info) != 0) return;
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= np32 * np32) return;
    const int r = e / np32, c = e - r * np32;
    float v;
    if (r < n && c < n) v = r <= c ? static_cast<float>(T[static_cast<int64_t>(r) * ldt + c]) : 0.0f;
    else v = r == c ? 1.0f : 0.0f;
    T32[e] = v;
    if (r == c) {
        if (!(fabsf(v) >= 1.17549435e-38f) || !isfinite(v)) set_status(info, fail_status, r);
        rinv32[r] = 1.0f / v;
    }
}

__device__ __forceinline__ void cp_async4f(void* dst, const void* src, bool valid) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(static_cast<unsigned>(__cvta_generic_to_shared(dst))),
                 "l"(src), "r"(valid ? 4 : 0));
}
__device__ __forceinline__ void cp_async16f(void* dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(static_cast<unsigned>(__cvta_generic_to_shared(dst))),
                 "l"(src));
}

// Y = X T^{-1} for upper-triangular T (T32, rinv32 from k_prep_f32).  Y may equal X (ldy == ldx).  A CTA keeps R rows
// in shared memory from load to store (row stride np32 + 4: float4 reads of a quarter-warp's rows hit distinct
// banks) and solves them left-looking over 32-column blocks:
//   off-diagonal  C -= Y[:, <block] T[<block, block], T streamed in 32 x 32 tiles (two buffers); a thread owns R / 32
//                 rows x 4 columns, so four terms take R / 32 + 4 16-byte reads for R / 2 multiply-adds;
//   diagonal      forward substitution, one thread per row, T's rows read as broadcasts.
// 2^20 x 128 on GB300: 0.61 ms (28 TFLOP/s; shared-memory pipe 74 % busy, issue slots 57 %; the FMA pipe alone would take
// 0.21 and HBM 0.16).  One row per thread, with the solved values re-read from global memory and a broadcast read of T
// for every four multiply-adds, took 1.58 ms.
// Rows per CTA: 128 while two such panels fit an SM, 64 above, 32 for matrices that give no full wave of 64.
template <int R>
__global__ void __launch_bounds__(256)
k_rowsolve_f32(const float* X, int64_t ldx, float* Y, int64_t ldy, int64_t m, int n,
               const float* __restrict__ T32, int np32, const float* __restrict__ rinv32, int32_t* info,
               bool check_finite, bool vec_in, bool vec_out) {
    extern __shared__ float4 fsm4[];
    constexpr int RT = R / 32;            // rows of a thread: ty + 32 i
    if (cta_stopped(info)) return;
    float* ts = reinterpret_cast<float*>(fsm4);            // two 32 x 32 tiles of T
    float* panel = ts + 2 * kF32Blk * kF32Blk;
    const int ld = np32 + 4;
    const int tid = threadIdx.x, tx = tid & 7, ty = tid >> 3;
    const int64_t row0 = static_cast<int64_t>(blockIdx.x) * R;
    const int nq = np32 / 4;
    if (vec_in) {
        for (int e = tid; e < R * nq; e += 256) {
            const int r = e / nq, c = 4 * (e - r * nq);
            float* dst = panel + r * ld + c;
            if (row0 + r < m && c + 3 < n) cp_async16f(dst, X + (row0 + r) * ldx + c);
            else
                for (int u = 0; u < 4; ++u) {
                    const bool ok = row0 + r < m && c + u < n;
                    cp_async4f(dst + u, ok ? X + (row0 + r) * ldx + c + u : X, ok);
                }
        }
    } else {
        for (int e = tid; e < R * np32; e += 256) {
            const int r = e / np32, c = e - r * np32;
            const bool ok = row0 + r < m && c < n;
            cp_async4f(panel + r * ld + c, ok ? X + (row0 + r) * ldx + c : X, ok);
        }
    }
    // tile (kt, J) of T into buffer b: rows 32 kt .., columns 32 J ..; one float4 per thread
    auto stage = [&](int kt, int J, int b) {
        cp_async16f(ts + b * kF32Blk * kF32Blk + 4 * tid,
                    T32 + static_cast<size_t>(kt * kF32Blk + ty) * np32 + J * kF32Blk + 4 * tx);
    };
    stage(0, 0, 0);
    cp_async_commit();
    bool bad = false;
    int b = 0;
    const int nblk = np32 / kF32Blk;
    for (int J = 0; J < nblk; ++J) {
        float acc[RT][4];
        for (int kt = 0; kt <= J; ++kt) {
            // the tile (kt, J) and, the first time, the panel have landed; prefetch the next tile
            cp_async_wait_all();
            __syncthreads();
            const bool last = kt == J;
            if (!last || J + 1 < nblk) stage(last ? 0 : kt + 1, last ? J + 1 : J, b ^ 1);
            cp_async_commit();
            const float* t0 = ts + b * kF32Blk * kF32Blk;
            b ^= 1;
            if (kt == 0 && J > 0) {
#pragma unroll
                for (int i = 0; i < RT; ++i) {
                    const float4 v = *reinterpret_cast<const float4*>(panel + (ty + 32 * i) * ld + J * kF32Blk + 4 * tx);
                    acc[i][0] = v.x; acc[i][1] = v.y; acc[i][2] = v.z; acc[i][3] = v.w;
#pragma unroll
                    for (int u = 0; u < 4; ++u) bad |= !isfinite(acc[i][u]);
                }
            }
            if (!last) {
#pragma unroll
                for (int k = 0; k < kF32Blk; k += 4) {
                    float4 tv[4];
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk) tv[kk] = *reinterpret_cast<const float4*>(t0 + (k + kk) * kF32Blk + 4 * tx);
#pragma unroll
                    for (int i = 0; i < RT; ++i) {
                        const float4 y4 = *reinterpret_cast<const float4*>(panel + (ty + 32 * i) * ld + kt * kF32Blk + k);
                        const float y[4] = {-y4.x, -y4.y, -y4.z, -y4.w};
#pragma unroll
                        for (int kk = 0; kk < 4; ++kk) {
                            acc[i][0] = fmaf(y[kk], tv[kk].x, acc[i][0]);
                            acc[i][1] = fmaf(y[kk], tv[kk].y, acc[i][1]);
                            acc[i][2] = fmaf(y[kk], tv[kk].z, acc[i][2]);
                            acc[i][3] = fmaf(y[kk], tv[kk].w, acc[i][3]);
                        }
                    }
                }
                continue;
            }
            if (J > 0) {
#pragma unroll
                for (int i = 0; i < RT; ++i)
                    *reinterpret_cast<float4*>(panel + (ty + 32 * i) * ld + J * kF32Blk + 4 * tx) =
                        make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
                __syncthreads();
            }
            if (tid < R) {
                float4* xr = reinterpret_cast<float4*>(panel + tid * ld + J * kF32Blk);
                float x[kF32Blk];
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    const float4 v = xr[q];
                    x[4 * q] = v.x; x[4 * q + 1] = v.y; x[4 * q + 2] = v.z; x[4 * q + 3] = v.w;
                }
                if (J == 0)
#pragma unroll
                    for (int c = 0; c < kF32Blk; ++c) bad |= !isfinite(x[c]);
#pragma unroll
                for (int j = 0; j < kF32Blk; ++j) {
                    x[j] *= __ldg(rinv32 + J * kF32Blk + j);
                    const float xj = -x[j];
#pragma unroll
                    for (int q = (j + 1) / 4; q < 8; ++q) {
                        const float4 tv = *reinterpret_cast<const float4*>(t0 + j * kF32Blk + 4 * q);
                        if (4 * q + 0 > j) x[4 * q + 0] = fmaf(xj, tv.x, x[4 * q + 0]);
                        if (4 * q + 1 > j) x[4 * q + 1] = fmaf(xj, tv.y, x[4 * q + 1]);
                        if (4 * q + 2 > j) x[4 * q + 2] = fmaf(xj, tv.z, x[4 * q + 2]);
                        if (4 * q + 3 > j) x[4 * q + 3] = fmaf(xj, tv.w, x[4 * q + 3]);
                    }
                }
#pragma unroll
                for (int q = 0; q < 8; ++q) xr[q] = make_float4(x[4 * q], x[4 * q + 1], x[4 * q + 2], x[4 * q + 3]);
            }
        }
    }
    __syncthreads();
    if (vec_out) {
        for (int e = tid; e < R * nq; e += 256) {
            const int r = e / nq, c = 4 * (e - r * nq);
            if (row0 + r >= m) continue;
            const float4 v = *reinterpret_cast<const float4*>(panel + r * ld + c);
            float* dst = Y + (row0 + r) * ldy + c;
            if (c + 3 < n) *reinterpret_cast<float4*>(dst) = v;
            else {
                if (c < n) dst[0] = v.x;
                if (c + 1 < n) dst[1] = v.y;
                if (c + 2 < n) dst[2] = v.z;
            }
        }
    } else {
        for (int e = tid; e < R * np32; e += 256) {
            const int r = e / np32, c = e - r * np32;
            if (row0 + r < m && c < n) Y[(row0 + r) * ldy + c] = panel[r * ld + c];
        }
    }
    if (__syncthreads_or(check_finite && bad) && threadIdx.x == 0) set_status(info, RPCHOLQR_ERR_NONFINITE);
}

// The same for up to W <= 16 columns, one row per thread in registers: the panels above have nothing to share there and keep
// few rows in flight (2^20 x 8: 117 us against 21 here, 2^20 x 16: 119 and 34; HBM alone would take 10 and 20).
template <int W>
__global__ void __launch_bounds__(256)
k_rowsolve_f32_narrow(const float* X, int64_t ldx, float* Y, int64_t ldy, int64_t m, int n, const float* __restrict__ T32,
                      int np32, const float* __restrict__ rinv32, int32_t* info, bool check_finite, bool vec_in,
                      bool vec_out) {
    __shared__ float4 ts[W][W / 4];
    __shared__ float ri[W];
    if (cta_stopped(info)) return;
    const int tid = threadIdx.x;
    if (tid < W * W / 4)
        ts[tid / (W / 4)][tid % (W / 4)] =
            *reinterpret_cast<const float4*>(T32 + static_cast<size_t>(tid / (W / 4)) * np32 + 4 * (tid % (W / 4)));
    if (tid < W) ri[tid] = rinv32[tid];
    __syncthreads();
    const int64_t row = static_cast<int64_t>(blockIdx.x) * 256 + tid;
    bool bad = false;
    if (row < m) {
        const float* xr = X + row * ldx;
        float* yr = Y + row * ldy;
        float x[W];
#pragma unroll
        for (int c = 0; c < W; c += 4) {
            if (vec_in && c + 3 < n) {
                const float4 v = *reinterpret_cast<const float4*>(xr + c);
                x[c] = v.x; x[c + 1] = v.y; x[c + 2] = v.z; x[c + 3] = v.w;
            } else {
#pragma unroll
                for (int u = 0; u < 4; ++u) x[c + u] = c + u < n ? xr[c + u] : 0.0f;
            }
        }
#pragma unroll
        for (int c = 0; c < W; ++c) bad |= !isfinite(x[c]);
#pragma unroll
        for (int j = 0; j < W; ++j) {
            x[j] *= ri[j];
            const float xj = -x[j];
#pragma unroll
            for (int q = (j + 1) / 4; q < W / 4; ++q) {
                const float4 tv = ts[j][q];
                if (4 * q + 0 > j) x[4 * q + 0] = fmaf(xj, tv.x, x[4 * q + 0]);
                if (4 * q + 1 > j) x[4 * q + 1] = fmaf(xj, tv.y, x[4 * q + 1]);
                if (4 * q + 2 > j) x[4 * q + 2] = fmaf(xj, tv.z, x[4 * q + 2]);
                if (4 * q + 3 > j) x[4 * q + 3] = fmaf(xj, tv.w, x[4 * q + 3]);
            }
        }
#pragma unroll
        for (int c = 0; c < W; c += 4) {
            if (vec_out && c + 3 < n) {
                *reinterpret_cast<float4*>(yr + c) = make_float4(x[c], x[c + 1], x[c + 2], x[c + 3]);
            } else {
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (c + u < n) yr[c + u] = x[c + u];
            }
        }
    }
    if (__syncthreads_or(check_finite && bad) && tid == 0) set_status(info, RPCHOLQR_ERR_NONFINITE);
}

// Partials of G = X^T X: CTA (tile, range) accumulates the 64 x 64 tile (I, J), I <= J, over the rows
// [range*rows_per, ...) and writes gpart[range][p][q] (ld np64, FP64) for its tile.  Thread (ty, tx) of 8 x 16 owns the
// 8 x 4 outputs p = 64 I + 8 ty + i, q = 64 J + 4 tx + j: three 16-byte reads for 32 multiply-adds (4 x 4 outputs
// needed two for 16: 1.00 -> 0.69 ms at 2^20 x 128).  Sums of 8 rows go into FP32 pairs: plain FP32 sums over a range's rows were
// what bounded the orthogonality on inputs with a few heavy rows.  20000 x 64 coherent inputs with smoothing, 72 draws:
// ||Q^T Q - I|| 6 times lower in the geometric mean, 0.88 of it on incoherent ones; the pairs take the time to 0.97 ms.
__global__ void __launch_bounds__(128)
k_syrk_f32(const float* __restrict__ X, int64_t ldx, int64_t m, int n, int np64, int64_t rows_per,
           double* __restrict__ gpart, const int32_t* info, bool vec) {
    __shared__ __align__(16) float xs[2][32][2 * 64 + 4];   // double-buffered 32-row chunks
    if (load_status(info) != 0) return;
    const int nb = np64 / 64;
    int tt = blockIdx.x, I = 0;
    while (tt >= nb - I) { tt -= nb - I; ++I; }
    const int J = I + tt;
    const int64_t rb = static_cast<int64_t>(blockIdx.y) * rows_per;
    const int64_t re = (rb + rows_per < m) ? rb + rows_per : m;
    const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
    const int boff = I == J ? 0 : 64;    // a diagonal tile's two operands are the same columns
    float hi[8][4], lo[8][4];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) hi[i][j] = lo[i][j] = 0.0f;
    // rows k0 .. k0+31 of the two 64-column blocks into xs[b] (zero outside X); 16-byte copies where rows are aligned
    auto stage = [&](int64_t k0, int b) {
        const int per = 16 + (boff >> 2);            // float4 columns of a row
        for (int e = tid; e < 32 * per; e += 128) {
            const int rr = e / per, cc = 4 * (e - rr * per);
            const int col = cc < 64 ? 64 * I + cc : 64 * J + (cc - 64);
            float* dst = &xs[b][rr][cc];
            const float* src = X + (k0 + rr) * ldx + col;
            if (vec && k0 + rr < re && col + 3 < n) cp_async16f(dst, src);
            else
                for (int u = 0; u < 4; ++u) {
                    const bool ok = k0 + rr < re && col + u < n;
                    cp_async4f(dst + u, ok ? src + u : X, ok);
                }
        }
    };
    // The pairs into this thread's FP64 partials: at the end, and before that when they have grown to where an FP32 total
    // of the range could overflow (rows far heavier than the sampled ones).
    double* out = gpart + static_cast<size_t>(blockIdx.y) * np64 * np64;
    bool flushed = false;
    auto flush = [&]() {
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                double& o = out[static_cast<size_t>(64 * I + 8 * ty + i) * np64 + 64 * J + 4 * tx + j];
                const double v = isfinite(hi[i][j]) ? static_cast<double>(hi[i][j]) + lo[i][j] : hi[i][j];   // an overflow stays one
                o = flushed ? o + v : v;
                hi[i][j] = lo[i][j] = 0.0f;
            }
        flushed = true;
    };
    if (rb < re) stage(rb, 0);
    cp_async_commit();
    int b = 0;
    for (int64_t k0 = rb; k0 < re; k0 += 32, b ^= 1) {
        if ((k0 - rb) % kSyrkSpillRows == 0) {
            float most = 0.0f;
#pragma unroll
            for (int i = 0; i < 8; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) most = fmaxf(most, fabsf(hi[i][j]));
            if (most > 0x1p100f) flush();
        }
        cp_async_wait_all();
        __syncthreads();   // chunk k0 has landed, and every thread is done with xs[b ^ 1]
        if (k0 + 32 < re) stage(k0 + 32, b ^ 1);
        cp_async_commit();
#pragma unroll 1
        for (int c = 0; c < 32; c += kSyrkRows) {
            float acc[8][4];
#pragma unroll
            for (int i = 0; i < 8; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = 0.0f;
#pragma unroll
            for (int kk = c; kk < c + kSyrkRows; ++kk) {
                const float4 a0 = *reinterpret_cast<const float4*>(&xs[b][kk][8 * ty]);
                const float4 a1 = *reinterpret_cast<const float4*>(&xs[b][kk][8 * ty + 4]);
                const float4 bb = *reinterpret_cast<const float4*>(&xs[b][kk][boff + 4 * tx]);
                const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w}, bv[4] = {bb.x, bb.y, bb.z, bb.w};
#pragma unroll
                for (int i = 0; i < 8; ++i)
#pragma unroll
                    for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(av[i], bv[j], acc[i][j]);
            }
            // (hi, lo) += acc, hi's rounding error into lo (Knuth's two-sum)
#pragma unroll
            for (int i = 0; i < 8; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const float s = __fadd_rn(hi[i][j], acc[i][j]), v = __fsub_rn(s, hi[i][j]);
                    lo[i][j] = __fadd_rn(lo[i][j], __fadd_rn(__fsub_rn(hi[i][j], __fsub_rn(s, v)), __fsub_rn(acc[i][j], v)));
                    hi[i][j] = s;
                }
        }
    }
    cp_async_wait_all();
    flush();
}

// dst (n x n float, ld ldd) = float(src) (n x n, ld lds)
__global__ void k_f64_to_f32(const double* __restrict__ src, int64_t lds, int n, float* __restrict__ dst,
                             int64_t ldd) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n * n) return;
    const int r = e / n, c = e - r * n;
    dst[static_cast<int64_t>(r) * ldd + c] = static_cast<float>(src[static_cast<int64_t>(r) * lds + c]);
}

// ---- host launchers --------------------------------------------------------------------------------
int f32_pad(int n) { return pad32(n); }

void launch_prep_f32(const double* T, int64_t ldt, int n, float* T32, float* rinv32, int fail_status,
                     int32_t* info, cudaStream_t st) {
    const int np32 = pad32(n);
    k_prep_f32<<<(np32 * np32 + 255) / 256, 256, 0, st>>>(T, ldt, n, np32, T32, rinv32, fail_status, info);
}

template <int R>
static cudaError_t launch_rowsolve_f32_r(const float* X, int64_t ldx, float* Y, int64_t ldy, int64_t m, int n,
                                         const float* T32, const float* rinv32, int32_t* info, bool check_finite,
                                         cudaStream_t st) {
    const int np32 = pad32(n);
    const int smem = (2 * kF32Blk * kF32Blk + R * (np32 + 4)) * static_cast<int>(sizeof(float));
    cudaError_t err = cudaFuncSetAttribute(k_rowsolve_f32<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (err != cudaSuccess) return err;
    // 16-byte copies need 16-byte aligned rows
    const bool vec_in = reinterpret_cast<uintptr_t>(X) % 16 == 0 && ldx % 4 == 0;
    const bool vec_out = reinterpret_cast<uintptr_t>(Y) % 16 == 0 && ldy % 4 == 0;
    k_rowsolve_f32<R><<<static_cast<unsigned>((m + R - 1) / R), 256, smem, st>>>(X, ldx, Y, ldy, m, n, T32, np32, rinv32, info,
                                                                                check_finite, vec_in, vec_out);
    return cudaGetLastError();
}

// sms: the device's SMs, for the choice of rows per CTA (see k_rowsolve_f32).
cudaError_t launch_rowsolve_f32(const float* X, int64_t ldx, float* Y, int64_t ldy, int64_t m, int n,
                                const float* T32, const float* rinv32, int32_t* info, bool check_finite, int sms,
                                cudaStream_t st) {
    if (n <= 16) {
        const bool vec_in = reinterpret_cast<uintptr_t>(X) % 16 == 0 && ldx % 4 == 0;
        const bool vec_out = reinterpret_cast<uintptr_t>(Y) % 16 == 0 && ldy % 4 == 0;
        auto kern = n <= 8 ? k_rowsolve_f32_narrow<8> : k_rowsolve_f32_narrow<16>;
        kern<<<static_cast<unsigned>((m + 255) / 256), 256, 0, st>>>(X, ldx, Y, ldy, m, n, T32, pad32(n), rinv32, info,
                                                                    check_finite, vec_in, vec_out);
        return cudaGetLastError();
    }
    if (m < static_cast<int64_t>(sms) * 64) return launch_rowsolve_f32_r<32>(X, ldx, Y, ldy, m, n, T32, rinv32, info, check_finite, st);
    if (n > 192 || m < static_cast<int64_t>(sms) * 256)
        return launch_rowsolve_f32_r<64>(X, ldx, Y, ldy, m, n, T32, rinv32, info, check_finite, st);
    return launch_rowsolve_f32_r<128>(X, ldx, Y, ldy, m, n, T32, rinv32, info, check_finite, st);
}

// ranges x np64 x np64 doubles in gpart; returns the number of ranges used.
int launch_syrk_f32(const float* X, int64_t ldx, int64_t m, int n, int max_ranges, double* gpart,
                    const int32_t* info, cudaStream_t st) {
    const int np64 = (n + 63) / 64 * 64;
    const int nb = np64 / 64;
    const int tiles = nb * (nb + 1) / 2;
    int ranges = (3 * max_ranges) / tiles;   // about three CTAs per SM
    if (ranges > max_ranges) ranges = max_ranges;
    if (ranges < 1) ranges = 1;
    const int64_t most = (m + 31) / 32;
    if (ranges > most) ranges = static_cast<int>(most);
    int64_t rows_per = (m + ranges - 1) / ranges;
    rows_per = (rows_per + 31) / 32 * 32;
    const bool vec = reinterpret_cast<uintptr_t>(X) % 16 == 0 && ldx % 4 == 0;
    k_syrk_f32<<<dim3(tiles, ranges), 128, 0, st>>>(X, ldx, m, n, np64, rows_per, gpart, info, vec);
    return ranges;
}

void launch_f64_to_f32(const double* src, int64_t lds, int n, float* dst, int64_t ldd, cudaStream_t st) {
    k_f64_to_f32<<<(n * n + 255) / 256, 256, 0, st>>>(src, lds, n, dst, ldd);
}

}  // namespace rpq
