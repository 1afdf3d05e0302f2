// The sample's Householder QR A_s = Q_s R_s (Algorithm alg_2, Section 4): R_s with a positive diagonal.  The
// algorithm and its reasons are in sketchqr.cuh.
//
// Measured on GB300 (whole step, s = 3 n) against one 16-CTA cluster that shared the columns and applied each
// reflector to them in global memory: n = 50 0.26 -> 0.15 ms, 128 0.79 -> 0.40, 200 1.72 -> 0.75, 512 13.2 -> 3.0,
// 1000 80.7 -> 11.4, 2048 684 -> 64 ms.  Of the 0.40 ms at n = 128 the panels take 0.31 (about 1.8 us a column
// and 15 us a launch); of the 11.4 ms at n = 1000 the panels take 5.5 and the two FP64 products 5.8 (0.92 TFLOP/s).
#include "sketchqr.cuh"

namespace rpq {

// Panel of columns k0 .. k0 + nb - 1, on one cluster.  Bound: the chain of column steps (per column two CTA
// barriers, one exchange over the cluster and about 20 dependent FP64 operations).
template <bool SMEM>
__global__ void __launch_bounds__(kQrThreads)
k_qr_panel(double* W, int64_t lds, int s, int k0, int nb, QrWs ws, int32_t* info) {
    extern __shared__ double qr_panel_sm[];
    __shared__ QrShared sh;
    // every CTA of the cluster sees the same status, so all take the same number of barriers
    if (load_status(info) != 0) return;
    cluster_sync_all();   // (no CTA may set a status before every other one has read it)
    const bool ok = qr_panel<true, SMEM, kQrThreads>(W, lds, s, k0, nb, ws.L, kQrB, ws.g, ws.betas, qr_panel_sm, sh,
                                                     cluster_rank(), cluster_size());
    if (__syncthreads_or(!ok) && threadIdx.x == 0) set_status(info, RPCHOLQR_ERR_TIMEOUT);
}

// Y partials: CTA (row chunk, 16 columns), one 16 x 8 tile per warp.  Bound: FP64 pipe (a 16 x 8 x 16 product
// takes 4096 clocks of one SM quarter, so small samples need the small tiles to reach many SMs).
__global__ void __launch_bounds__(128)
k_qr_y(const double* __restrict__ W, int64_t lds, int s, int k0, int nb, int n, double* __restrict__ Y, const int32_t* info) {
    if (load_status(info) != 0) return;
    const int nrows = s - k0, nt = n - k0 - nb, ch = qr_chunk_rows(nrows), warp = threadIdx.x >> 5;
    const int c0 = blockIdx.y * 16 + 8 * (warp >> 1);
    if (c0 >= nt) return;
    qr_y_tile(W + static_cast<int64_t>(k0) * lds + k0, W + static_cast<int64_t>(k0 + nb + c0) * lds + k0, lds, nrows, nb,
              nt - c0, warp & 1, blockIdx.x * ch, (blockIdx.x + 1) * ch,
              Y + (static_cast<size_t>(blockIdx.x) * ((nt + 7) / 8 * 8) + c0) * kQrB);
}

// Z: one warp per column sums the partials in chunk order and solves.  Bound: latency (the substitution).
__global__ void __launch_bounds__(128)
k_qr_z(QrWs ws, int nb, int nt, int nchunks, const int32_t* info) {
    __shared__ double Ls[kQrB * kQrLd];
    if (load_status(info) != 0) return;
    const int lane = threadIdx.x & 31, col = blockIdx.x * 4 + (threadIdx.x >> 5);
    for (int e = threadIdx.x; e < kQrB * kQrB; e += 128) Ls[(e / kQrB) * kQrLd + e % kQrB] = ws.L[e];
    __syncthreads();
    if (col >= nt) return;
    const size_t step = static_cast<size_t>((nt + 7) / 8 * 8) * kQrB;
    const double* yp = ws.Y + static_cast<size_t>(col) * kQrB + lane;
    double p[kQrMaxChunks], y = 0.0;
#pragma unroll
    for (int q = 0; q < kQrMaxChunks; ++q) p[q] = q < nchunks ? yp[q * step] : 0.0;
#pragma unroll
    for (int q = 0; q < kQrMaxChunks; ++q)
        if (q < nchunks) y += p[q];
    ws.Z[static_cast<size_t>(col) * kQrB + lane] = qr_z_solve(y, Ls, lane < nb ? ws.g[lane] : 0.0, nb);
}

// W -= V Z: CTA 64 rows x 8 columns, a warp 16 rows.  Bound: FP64 pipe.
__global__ void __launch_bounds__(128)
k_qr_update(double* __restrict__ W, int64_t lds, int s, int k0, int nb, int n, const double* __restrict__ Z,
            const int32_t* info) {
    if (load_status(info) != 0) return;
    const int nrows = s - k0, nt = n - k0 - nb, r0 = blockIdx.x * 64 + 16 * (threadIdx.x >> 5), c0 = blockIdx.y * 8;
    if (r0 >= nrows) return;
    qr_update_tile(W + static_cast<int64_t>(k0) * lds + k0, W + static_cast<int64_t>(k0 + nb + c0) * lds + k0, lds, nrows, nb,
                   nt - c0 < 8 ? nt - c0 : 8, r0, Z + static_cast<size_t>(c0) * kQrB);
}

__global__ void __launch_bounds__(256)
k_qr_out(const double* __restrict__ W, int64_t lds, int n, int np, const double* __restrict__ betas, double* __restrict__ Rs,
         double* __restrict__ Rs_user, int32_t* info) {
    if (cta_stopped(info)) return;
    const int64_t e = static_cast<int64_t>(blockIdx.x) * 256 + threadIdx.x;
    const bool bad = e < static_cast<int64_t>(np) * np && !qr_out_entry(W, lds, n, np, betas, static_cast<int>(e), Rs, Rs_user);
    if (__syncthreads_or(bad) && threadIdx.x == 0) set_status(info, RPCHOLQR_ERR_SINGULAR_SKETCH);
}

// Longest sample a plan accepts is set by its columns' shared memory in the first design of this step; kept.
size_t householder_smem_bytes(int s, int n) { return (static_cast<size_t>(s) + n + 40) * sizeof(double); }
int householder_launches(int n) { return 4 * ((n + kQrB - 1) / kQrB) - 2; }
size_t householder_ws_bytes(int np) { return qr_ws_doubles(np) * sizeof(double); }

// W: s x n column-major (ld lds), overwritten.  qws: householder_ws_bytes(np) of device workspace.  One cluster of
// 16 CTAs per panel (16 needs the non-portable cluster size; 8 is used where the device refuses 16), the panel in
// shared memory while a CTA's rows fit.
cudaError_t launch_householder(double* W, int64_t lds, int s, int n, int np, double* Rs, double* Rs_user, double* qws,
                               int32_t* info, cudaStream_t st) {
    constexpr size_t kMaxPanel = 190 * 1024;
    const QrWs ws = qr_ws(qws, np);
    cudaError_t err =
        cudaFuncSetAttribute(k_qr_panel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kMaxPanel));
    if (err != cudaSuccess) return err;
    for (auto kern : {k_qr_panel<true>, k_qr_panel<false>}) {
        err = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (err != cudaSuccess) return err;
    }
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(kQrThreads, 1, 1);
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int csize = 0;
    for (int k0 = 0; k0 < n; k0 += kQrB) {
        const int nb = n - k0 < kQrB ? n - k0 : kQrB, nrows = s - k0, nt = n - k0 - nb;
        const int rg = (nrows + kQrGroups - 1) / kQrGroups;
        auto shape = [&](int c) {
            const size_t bytes = static_cast<size_t>(kQrGroups / c) * rg * kQrLd * sizeof(double);
            attr[0].val.clusterDim.x = c;
            cfg.gridDim = dim3(c, 1, 1);
            cfg.dynamicSmemBytes = bytes <= kMaxPanel ? bytes : 0;
            return bytes <= kMaxPanel;
        };
        for (int c = kQrCluster; csize == 0 && c >= 8; c /= 2) {   // once per call, for the panel with the most rows
            int clusters = 0;
            auto kern = shape(c) ? k_qr_panel<true> : k_qr_panel<false>;
            if (cudaOccupancyMaxActiveClusters(&clusters, kern, &cfg) == cudaSuccess && clusters >= 1) csize = c;
            else cudaGetLastError();
        }
        if (csize == 0) return cudaErrorInvalidConfiguration;
        err = cudaLaunchKernelEx(&cfg, shape(csize) ? k_qr_panel<true> : k_qr_panel<false>, W, lds, s, k0, nb, ws, info);
        if (err != cudaSuccess) return err;
        if (nt > 0) {
            const int ch = qr_chunk_rows(nrows), nchunks = (nrows + ch - 1) / ch;
            k_qr_y<<<dim3(nchunks, (nt + 15) / 16), 128, 0, st>>>(W, lds, s, k0, nb, n, ws.Y, info);
            k_qr_z<<<(nt + 3) / 4, 128, 0, st>>>(ws, nb, nt, nchunks, info);
            k_qr_update<<<dim3((nrows + 63) / 64, (nt + 7) / 8), 128, 0, st>>>(W, lds, s, k0, nb, n, ws.Z, info);
        }
    }
    const int64_t tot = static_cast<int64_t>(np) * np;
    k_qr_out<<<static_cast<unsigned>((tot + 255) / 256), 256, 0, st>>>(W, lds, n, np, ws.betas, Rs, Rs_user, info);
    return cudaGetLastError();
}

}  // namespace rpq
