// Device-side building blocks shared by the rpCholesky-QR kernels (sm_103a).
#pragma once
#include <climits>
#include <cstdint>
#include <cuda_runtime.h>

#include "../../include/rpcholqr.h"

namespace rpq {

// Every matrix dimension is padded to a multiple of this (the k extent of mma m16n8k16).
constexpr int kPad = 16;
constexpr int kMaxNP = 128;             // widest panel the row-pass kernels keep in shared memory

__host__ __device__ constexpr int pad16(int n) { return (n + kPad - 1) / kPad * kPad; }
// Padded width of the n x n factors: a multiple of 16 up to 128 columns, of 64 above (64-column blocks).
__host__ __device__ constexpr int pad_np(int n) { return n <= kMaxNP ? pad16(n) : (n + 63) / 64 * 64; }

// ---- launch shape of the FP64 row passes (rowpass.cu) ----------------------------------------------
// A panel is 256 rows (8 warps x 32) up to 64 columns, 128 rows (8 warps x 16) above: two warps on each of the
// SM's four schedulers, so that one warp's dependent chains and shared-memory loads run under the other's FP64
// work (four warps x 32 rows at 128 columns kept the FP64 pipe 74-83 % busy).  Matrices too short to give every
// SM such a panel take one panel of 64 to 128 rows (4 to 8 warps x 16) per SM.
constexpr int kRowpassWarps = 8, kRowpassMinWarps = 4;
__host__ __device__ constexpr int rowpass_rows_per_warp(int np) { return np <= 64 ? 32 : 16; }
__host__ __device__ constexpr int rowpass_big_rows(int np) { return kRowpassWarps * rowpass_rows_per_warp(np); }
// Warps of the short shape for m rows on sms SMs, 0: the big panels.
__host__ __device__ constexpr int rowpass_short_warps(int np, int64_t m, int sms) {
    const int64_t w = (m + 16 * static_cast<int64_t>(sms) - 1) / (16 * static_cast<int64_t>(sms));
    return w * 16 >= rowpass_big_rows(np) || w > kRowpassWarps ? 0
           : w < kRowpassMinWarps                              ? kRowpassMinWarps
                                                               : static_cast<int>(w);
}
__host__ __device__ constexpr int rowpass_rows(int np, int64_t m, int sms) {
    const int w = rowpass_short_warps(np, m, sms);
    return w ? 16 * w : rowpass_big_rows(np);
}
// CTAs of the fused Gram pass, each leaving one partial: one per panel, at most one per SM.
__host__ __device__ constexpr int rowpass_parts(int np, int64_t m, int sms) {
    const int64_t rows = rowpass_rows(np, m, sms), panels = (m + rows - 1) / rows;
    return static_cast<int>(panels < sms ? panels : sms);
}
// The most of those partials any width and any row count up to m leave: short panels have 64 rows or more.
__host__ __device__ constexpr int rowpass_max_parts(int64_t m, int sms) {
    const int64_t panels = (m + 16 * kRowpassMinWarps - 1) / (16 * kRowpassMinWarps);
    return static_cast<int>(panels < sms ? panels : sms);
}
// The plain solve up to 48 columns runs two CTAs per SM (128 registers a thread, two panels fit the
// shared memory): one CTA's panel load overlaps the other's FP64 work and each scheduler has four
// warps' dependent chains to interleave.  The fused Gram keeps one CTA per SM (one partial each).
__host__ __device__ constexpr int rowpass_ctas_per_sm(int np, bool syrk) { return !syrk && np <= 48 ? 2 : 1; }

// ---- power-of-two bounds used by the split-precision products ------------------------------------
// exp_bound(v): |v| < 2^e for a normal v (e = unbiased exponent + 1); kNoExp for 0 or subnormal.
constexpr int kNoExp = INT_MIN / 2;
__device__ __forceinline__ int exp_bound(double v) {
    const int ex = static_cast<int>((__double_as_longlong(v) >> 52) & 0x7FF);
    return ex == 0 ? kNoExp : ex - 1022;
}

// ---- square roots in 64-bit fixed point (sketch QR, Cholesky) -------------------------------------
// Both steps wait for a root and a reciprocal in every column.  An FP64 operation takes 65 clocks on GB300 and holds its
// scheduler's FP64 unit for 64 of them, and a square root or a division is a long sequence of them; a 64 x 64-bit high
// product takes about 30.  x = X 2^(k - 61) with X / 2^61 in [1, 4); an FP32 seed y ~ x^{-1/2} good to 2^-20 and one step of
// Halley's iteration t + t h, t = x y, h = e / 2 + 3 e^2 / 8, e = 1 - t y.  The third power left out and the truncations are
// below 2^-57 of the root.
__device__ __forceinline__ bool root_in_range(double x) {   // x >= 0 or NaN
    const int xe = (__double2hiint(x) >> 20) - 1023;
    return xe >= -900 && xe <= 900;
}
struct FixedRoot {
    unsigned long long X, Y, N;   // x (Q61), y (Q64), sqrt(x) (Q61), all of x's scaled value
    long long h;                  // Q61
    int k;                        // x's power of two, even
    float xf, yf;                 // the scaled x and its seed
};
__device__ __forceinline__ FixedRoot fixed_root(double x) {   // root_in_range(x)
    FixedRoot r;
    const unsigned long long xb = static_cast<unsigned long long>(__double_as_longlong(x));
    const int xe = static_cast<int>(xb >> 52) - 1023;
    r.k = xe & ~1;
    r.X = ((xb & ((1ull << 52) - 1)) | (1ull << 52)) << (9 + (xe - r.k));
    r.xf = static_cast<float>(static_cast<uint32_t>(r.X >> 32)) * 0x1p-29f;
    r.yf = fminf(rsqrtf(r.xf), 0x1.fffffep-1f);
    r.Y = static_cast<unsigned long long>(__float2uint_rz(r.yf * 0x1p32f)) << 32;
    const unsigned long long T = __umul64hi(r.X, r.Y);
    const long long E = static_cast<long long>((1ull << 61) - __umul64hi(T, r.Y));
    const long long eh = E >> 20;
    r.h = (E >> 1) + ((3 * ((eh * eh) >> 21)) >> 3);
    r.N = T + static_cast<unsigned long long>(__mul64hi(static_cast<long long>(T), r.h << 3));
    return r;
}
__device__ __forceinline__ double fixed_root_value(const FixedRoot& r) {
    return __longlong_as_double(static_cast<long long>((static_cast<unsigned long long>(1022 + r.k / 2) << 52) + ((r.N + 256) >> 9)));
}
// The Q63 number v > 0 times 2^p in FP64, rounded to nearest without leaving 64 bits (v's leading 64 bits may be 2^64 - 1).
__device__ __forceinline__ double from_q63(unsigned long long v, int p) {
    const int lz = __clzll(static_cast<long long>(v));
    const unsigned long long M = v << lz;
    return __longlong_as_double(
        static_cast<long long>((static_cast<unsigned long long>(1022 - lz + p) << 52) + (M >> 11) + ((M >> 10) & 1)));
}

// ---- status word: info[0] = status, info[1] = pivot ---------------------------------------------
__device__ __forceinline__ int load_status(const int32_t* info) {
    return *reinterpret_cast<const volatile int32_t*>(info);
}
// True for every thread of the CTA when a status is set: one answer for all of them.  A kernel that sets the status
// itself decides whether to run by this, not by each thread's own read: a CTA that starts late may find another CTA's
// status appear between the reads of its warps, and the warps that went on would wait for ever at a barrier with a fixed
// count, or work on tensor memory that the warp that left was to allocate.
__device__ __forceinline__ bool cta_stopped(const int32_t* info) { return __syncthreads_or(load_status(info) != 0) != 0; }
// First error wins.
__device__ __forceinline__ void set_status(int32_t* info, int status, int pivot = -1) {
    if (atomicCAS(info, 0, status) == 0 && pivot >= 0) info[1] = pivot;
}

// ---- FP64 tensor-core mma: D(16x8) += A(16x16) * B(16x8), all FP64 ------------------------------
// Fragment layouts (g = lane/4, t = lane%4):
//   A: a[i] = A[g + 8*(i&1)][t + 4*(i>>1)]      i = 0..7
//   B: b[i] = B[t + 4*i][g]                     i = 0..3
//   C: c[i] = C[g + 8*(i>>1)][2*t + (i&1)]      i = 0..3
__device__ __forceinline__ void mma_f64_16816(double (&d)[4], const double (&a)[8],
                                              const double (&b)[4]) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f64.f64.f64.f64 {%0,%1,%2,%3}, "
        "{%4,%5,%6,%7,%8,%9,%10,%11}, {%12,%13,%14,%15}, {%0,%1,%2,%3};\n"
        : "+d"(d[0]), "+d"(d[1]), "+d"(d[2]), "+d"(d[3])
        : "d"(a[0]), "d"(a[1]), "d"(a[2]), "d"(a[3]), "d"(a[4]), "d"(a[5]), "d"(a[6]), "d"(a[7]),
          "d"(b[0]), "d"(b[1]), "d"(b[2]), "d"(b[3]));
}

// D(16x8) += A(16x8) * B(8x8), FP64: the same fragment layouts restricted to k < 8
// (a[i] = A[g + 8*(i&1)][t + 4*(i>>1)], i = 0..3;  b[i] = B[t + 4*i][g], i = 0..1).
__device__ __forceinline__ void mma_f64_1688(double (&d)[4], const double (&a)[4], const double (&b)[2]) {
    asm volatile(
        "mma.sync.aligned.m16n8k8.row.col.f64.f64.f64.f64 {%0,%1,%2,%3}, "
        "{%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
        : "+d"(d[0]), "+d"(d[1]), "+d"(d[2]), "+d"(d[3])
        : "d"(a[0]), "d"(a[1]), "d"(a[2]), "d"(a[3]), "d"(b[0]), "d"(b[1]));
}

// ---- cp.async (Ampere+ LDGSTS), 8-byte granules with zero fill ----------------------------------
__device__ __forceinline__ void cp_async8(void* smem_dst, const void* gmem_src, bool valid) {
    unsigned s = static_cast<unsigned>(__cvta_generic_to_shared(smem_dst));
    int src_size = valid ? 8 : 0;
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(s), "l"(gmem_src),
                 "r"(src_size));
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

}  // namespace rpq
