// Streaming passes of Algorithm alg_2 (Section 4) over the rows of a tall-skinny matrix:
//
//   pass 1 ('precondition' + 'Gram'):  A1 = A R_s^{-1}  and  G1 += A1_panel^T A1_panel
//   pass 2 ('solve'):                  Q  = A1 R_1^{-1}  (in place over A1)
//
// Both are m independent row solves x_i^T = T^{-T} b_i^T (the row-wise view of Section 2.1).
//
// GB300 design.  FP64 on this part runs at about 1.05 TFLOP/s whether it is issued as DFMA or as the
// FP64 tensor-core mma.sync m16n8k16 (measured); HBM is ~100x faster than this FP64 work needs, so the
// kernels are organised to keep the FP64 pipe busy, not for bandwidth.  mma.sync m16n8k16 carries 2048
// FMAs per instruction, so the issue slots stay free for address math and shared-memory traffic:
//   * a CTA (8 warps; 4 for short matrices) owns a panel of 16 or 32 rows per warp (common.cuh) staged in
//     shared memory with cp.async; the row stride NP+4 doubles keeps every fragment load at the minimum two
//     wavefronts;
//   * the solve is blocked by 8 columns, left-looking: block J of a 16-row tile is
//       acc = X[:, J] - A1[:, <J] T[<J, J]          (mma m16n8k16, FP64, B = -T chunks)
//       A1[:, J] = acc T[J, J]^{-1}                 (8-column forward substitution, DFMA,
//                                                    one or two lanes per row, reciprocal diagonal)
//     each 16-row tile has two split-k accumulators;
//   * the Gram matrix keeps only the upper 16x8 tiles (72 tiles at n = 128), 9 per warp, accumulated in
//     registers across every panel the CTA visits; each CTA writes one partial and a second kernel sums the partials in a fixed order (deterministic, no atomics).
// Measured on GB300 (2^20 x 128): fused pass 1 41.5 -> 34.8 ms (0.99 TFLOP/s of the probe's 1.10), pass 2 23.3 -> 17.1
// ms with eight warps of 16 rows instead of four of 32 and the right-looking diagonal block; a 10000 x 50 factorisation
// 811 -> 479 us with 80-row panels on 125 SMs instead of 256-row panels on 40.
#include "rowpass.cuh"

namespace rpq {

__global__ void k_prep_tri(const double* __restrict__ T, int64_t ldt, int n, int np,
                           double* __restrict__ frag, double* __restrict__ diag,
                           const int32_t* info) {
    if (info && load_status(info) != 0) return;
    prep_tri_entry(T, ldt, n, np, frag, diag, blockIdx.x * blockDim.x + threadIdx.x);
}

// SHORT: 4 to 8 warps of 16 rows (the launch's), else the big panels.
template <int NP, bool SYRK, bool SHORT>
__global__ void __launch_bounds__(kRowpassWarps * 32, SHORT ? 1 : rowpass_ctas_per_sm(NP, SYRK))
k_rowpass(const double* X, int64_t ldx, double* Y, int64_t ldy, int64_t m, int n,
          const double* __restrict__ frag, const double* __restrict__ diag,
          double* __restrict__ gpart, int32_t* info, bool check_finite) {
    extern __shared__ double panel[];
    if (cta_stopped(info)) return;
    double* out = SYRK ? gpart + static_cast<size_t>(blockIdx.x) * NP * NP : nullptr;
    const int nw = SHORT ? blockDim.x >> 5 : kRowpassWarps;
    const bool bad = rowpass_panels<NP, SYRK, SHORT ? 16 : rowpass_rows_per_warp(NP),
                                    SHORT ? kRowpassMinWarps : kRowpassWarps, true, true>(
        nw, nw, X, ldx, Y, ldy, m, n, frag, diag, check_finite, blockIdx.x, gridDim.x, panel,
        [] {}, [out](int pr, int pc, double v) { out[pr * NP + pc] = v; });
    if (__syncthreads_or(bad) && threadIdx.x == 0) set_status(info, RPCHOLQR_ERR_NONFINITE);
}

// G[p][q] = G[q][p] = sum over CTAs b = 0..nparts-1 (in this order) of part_b[p][q], q >= p.
__global__ void k_gram_reduce(const double* __restrict__ gpart, int nparts, int np, int n,
                              double* __restrict__ G, int64_t ldg, const int32_t* info) {
    if (load_status(info) != 0) return;
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n * n) return;
    const int p = e / n, q = e - p * n;
    if (q < p) return;
    const double* gp = gpart + static_cast<int64_t>(p) * np + q;
    double sum = 0.0;
    int b = 0;
    for (; b + 15 < nparts; b += 16) {   // sixteen loads in flight, summed in order
        double v[16];
#pragma unroll
        for (int u = 0; u < 16; ++u) v[u] = gp[static_cast<size_t>(b + u) * np * np];
#pragma unroll
        for (int u = 0; u < 16; ++u) sum += v[u];
    }
    for (; b < nparts; ++b) sum += gp[static_cast<size_t>(b) * np * np];
    G[static_cast<int64_t>(p) * ldg + q] = sum;
    G[static_cast<int64_t>(q) * ldg + p] = sum;
}

// ---- host launchers ------------------------------------------------------------------------------
void launch_prep_tri(const double* T, int64_t ldt, int n, int np, double* frag, double* diag,
                     const int32_t* info, cudaStream_t st) {
    const int total = np * np + (np / 8) * 64;
    k_prep_tri<<<(total + 255) / 256, 256, 0, st>>>(T, ldt, n, np, frag, diag, info);
}


// The tables of every blk x blk diagonal block of T (n x n) at once: block J's at frag + J blk^2 and diag + J 8 blk, of
// the block padded to a multiple of 16 (the last one may be narrower).
__global__ void k_prep_blocks(const double* __restrict__ T, int64_t ldt, int n, int blk, double* __restrict__ frag,
                              double* __restrict__ diag, const int32_t* info) {
    if (info && load_status(info) != 0) return;
    const int J = blockIdx.y, nj = n - J * blk < blk ? n - J * blk : blk;
    prep_tri_entry(T + static_cast<int64_t>(J) * blk * ldt + J * blk, ldt, nj, pad16(nj), frag + static_cast<size_t>(J) * blk * blk,
                   diag + static_cast<size_t>(J) * blk * 8, blockIdx.x * blockDim.x + threadIdx.x);
}
void launch_prep_blocks(const double* T, int64_t ldt, int n, int blk, double* frag, double* diag, const int32_t* info,
                        cudaStream_t st) {
    k_prep_blocks<<<dim3((blk * blk + 8 * blk + 255) / 256, (n + blk - 1) / blk), 256, 0, st>>>(T, ldt, n, blk, frag, diag,
                                                                                             info);
}

template <int NP, bool SYRK, bool SHORT>
static cudaError_t launch_rowpass_t(const double* X, int64_t ldx, double* Y, int64_t ldy, int64_t m,
                                    int n, const double* frag, const double* diag, double* gpart,
                                    int32_t* info, int sms, cudaStream_t st, bool check) {
    const int rows = rowpass_rows(NP, m, sms), warps = SHORT ? rows / 16 : kRowpassWarps;
    auto kern = k_rowpass<NP, SYRK, SHORT>;
    cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           static_cast<int>(rowpass_smem_bytes(NP, SHORT ? 128 : rows)));
    if (err != cudaSuccess) return err;
    const int64_t panels = (m + rows - 1) / rows, cap = static_cast<int64_t>(sms) * (SHORT ? 1 : rowpass_ctas_per_sm(NP, SYRK));
    kern<<<static_cast<unsigned>(panels < cap ? panels : cap), 32 * warps, rowpass_smem_bytes(NP, rows), st>>>(
        X, ldx, Y, ldy, m, n, frag, diag, gpart, info, check);
    return cudaGetLastError();
}

template <bool SYRK>
static cudaError_t launch_rowpass_np(int np, const double* X, int64_t ldx, double* Y, int64_t ldy,
                                     int64_t m, int n, const double* frag, const double* diag,
                                     double* gpart, int32_t* info, int sms, cudaStream_t st, bool check) {
    const bool brief = rowpass_short_warps(np, m, sms) != 0;
    switch (np) {
#define RPQ_CASE(V)                                                                                     \
    case V:                                                                                             \
        return (brief ? launch_rowpass_t<V, SYRK, true> : launch_rowpass_t<V, SYRK, false>)(            \
            X, ldx, Y, ldy, m, n, frag, diag, gpart, info, sms, st, check);
        RPQ_CASE(16) RPQ_CASE(32) RPQ_CASE(48) RPQ_CASE(64) RPQ_CASE(80) RPQ_CASE(96) RPQ_CASE(112)
        RPQ_CASE(128)
#undef RPQ_CASE
        default: return cudaErrorInvalidValue;
    }
}

// sms: SMs to use; the fused Gram pass leaves rowpass_parts(np, m, sms) partials in gpart.
// check_finite: set NONFINITE when an input entry is NaN/Inf.
cudaError_t launch_rowpass(bool syrk, int np, const double* X, int64_t ldx, double* Y, int64_t ldy,
                           int64_t m, int n, const double* frag, const double* diag, double* gpart,
                           int32_t* info, int sms, cudaStream_t st, bool check_finite) {
    return syrk ? launch_rowpass_np<true>(np, X, ldx, Y, ldy, m, n, frag, diag, gpart, info, sms, st, check_finite)
                : launch_rowpass_np<false>(np, X, ldx, Y, ldy, m, n, frag, diag, gpart, info, sms, st, check_finite);
}

void launch_gram_reduce(const double* gpart, int nparts, int np, int n, double* G, int64_t ldg,
                        const int32_t* info, cudaStream_t st) {
    const int total = n * n;
    k_gram_reduce<<<(total + 255) / 256, 256, 0, st>>>(gpart, nparts, np, n, G, ldg, info);
}

}  // namespace rpq
