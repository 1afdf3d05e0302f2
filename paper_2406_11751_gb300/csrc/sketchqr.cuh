// Device-side pieces of the sample's Householder QR (step 'factor' of Algorithm alg_2, Section 4), shared by
// its kernels (sketchqr.cu) and the persistent batched kernel (persist.cu).
//
// FP64 on GB300 retires two multiply-adds per clock per SM, one warp's instruction in 64 clocks of its scheduler, and a
// dependent one waits as long, so this step is bound by the chain of column steps and by how many SMs share the O(s n^2)
// work.
// Panels of kQrB columns: the panel is factored by one thread-block cluster with its ROWS shared out (one
// reduction over the cluster per column), then the columns to its right are updated by every SM:
//   panel   W[:, panel] -> reflectors H_j = I - g_j v_j v_j^T, v_j = x - beta e_j not normalised,
//           beta = -sign(alpha) ||x||, g_j = 1 / (||x|| (||x|| + |alpha|)) (no reflection when nothing is
//           below the diagonal); the reduction for column j gives sigma = sum of squares below the diagonal
//           and the products of x with every panel column at once: those to the right take the update, those
//           to the left are v_k^T v_j, the entries of the lower triangle L;
//   Y       partials over row chunks of V^T W (FP64 mma);
//   Z       (D + L) Z = sum of the partials, D = diag(1 / g) (the UT transform: Puglisi, SIAM J. Sci. Stat.
//           Comput. 1992; Joffrain et al., ACM TOMS 2006): forward substitution per column;
//   update  W -= V Z (FP64 mma).
// Every sum has a fixed order that depends on the shape alone (64 row groups, their sums in a fixed tree,
// row chunks in order), not on how many CTAs share the work: one CTA alone gives the cluster's bits.
#pragma once
#include <cfloat>
#include <type_traits>

#include "common.cuh"

namespace rpq {

constexpr int kQrB = 32;              // panel columns: one lane each
constexpr int kQrGroups = 64;         // row groups of a panel, one warp each (16 CTAs x 4 warps)
constexpr int kQrQuads = kQrGroups / 4;
constexpr int kQrCluster = 16;
constexpr int kQrThreads = 128;
constexpr int kQrLd = kQrB + 1;       // panel row stride in shared memory (doubles)
constexpr int kQrPartLd = kQrB + 4;   // partial sums: four rows at once hit distinct banks
constexpr int kQrMaxChunks = 16;

// Rows of one chunk of the Y partials: a multiple of 32, at most kQrMaxChunks chunks.
__host__ __device__ constexpr int qr_chunk_rows(int nrows) {
    return 32 * ((nrows + 32 * kQrMaxChunks - 1) / (32 * kQrMaxChunks));
}

struct QrShared {
    double part[kQrGroups][kQrPartLd];       // per row group (of this CTA): its sums
    double quad[2][kQrQuads][kQrPartLd];     // sums of four groups, from every CTA; alternating by column
    double row[2][kQrB];                     // the pivot row
    double row_out[kQrB];                    // the pivot row, in the CTA that holds it
    double D[kQrB];                          // the reduced sums
    uint64_t bar[2];                         // arrival of quad[p] and row[p] (cluster)
};
constexpr uint32_t kQrStepBytes = (kQrQuads + 1) * kQrB * sizeof(double);   // what a column step receives
constexpr long kQrSpinLimit = 1L << 24;

// Workspace of one factorisation (doubles): Y partials, Z, L and g of the current panel, betas.
struct QrWs {
    double *Y, *Z, *L, *g, *betas;
};
__host__ __device__ inline size_t qr_ws_doubles(int np) {
    return static_cast<size_t>(kQrMaxChunks + 1) * kQrB * np + kQrB * kQrB + kQrB + np;
}
__host__ __device__ inline QrWs qr_ws(double* w, int np) {
    QrWs q;
    q.Y = w;
    q.Z = q.Y + static_cast<size_t>(kQrMaxChunks) * kQrB * np;
    q.L = q.Z + static_cast<size_t>(kQrB) * np;
    q.g = q.L + kQrB * kQrB;
    q.betas = q.g + kQrB;
    return q;
}

__device__ __forceinline__ void cluster_sync_all() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;\n" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}
__device__ __forceinline__ unsigned cluster_rank() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;\n" : "=r"(r));
    return r;
}
__device__ __forceinline__ unsigned cluster_size() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_nctarank;\n" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t cluster_addr(uint32_t smem, unsigned cta) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(r) : "r"(smem), "r"(cta));
    return r;
}
// A store into another CTA's shared memory that completes its 8 bytes on that CTA's barrier: data and signal
// in one message (a store followed by the cluster barrier took 940 clocks a column for the barrier alone).
__device__ __forceinline__ void st_async(uint32_t addr, uint32_t bar, double v) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];\n" ::"r"(addr),
                 "l"(__double_as_longlong(v)), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void qr_bar_arm(uint64_t* bar) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(
                     static_cast<uint32_t>(__cvta_generic_to_shared(bar))),
                 "r"(kQrStepBytes)
                 : "memory");
}
__device__ __forceinline__ bool qr_bar_wait(uint64_t* bar, uint32_t parity) {
    uint32_t done = 0;
    for (long it = 0; it < kQrSpinLimit && !done; ++it)
        asm volatile(
            "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}\n"
            : "=r"(done)
            : "r"(static_cast<uint32_t>(__cvta_generic_to_shared(bar))), "r"(parity)
            : "memory");
    return done != 0;
}

// nrm = sqrt(x) (fixed_root) and g = 1 / (x + nrm |alpha|) for x = alpha^2 + sigma, both on the critical path of every column:
// an FP32 seed r ~ g, good to 2^-20, and the Neumann series g = r (1 + f + f^2), f = 1 - (x + nrm |alpha|) r.  Outside
// root_in_range the plain operations are used and false is returned.
__device__ __forceinline__ bool qr_scalars(double alpha, double x, double& nrm, double& g) {
    if (root_in_range(x)) {
        const unsigned long long ab = static_cast<unsigned long long>(__double_as_longlong(alpha));
        const FixedRoot q = fixed_root(x);
        const int ae = static_cast<int>((ab >> 52) & 0x7FF), sh = ae - 1023 - q.k / 2 + 9;
        const unsigned long long am = ae ? (ab & ((1ull << 52) - 1)) | (1ull << 52) : 0ull;
        const unsigned long long Al = sh >= 0 ? am << sh : (sh > -64 ? am >> -sh : 0ull);        // |alpha| <= 2, Q61
        const float af = static_cast<float>(static_cast<uint32_t>(Al >> 32)) * 0x1p-29f;
        const float rf = fminf(__frcp_rn(fmaf(q.xf * q.yf, af, q.xf)), 0x1.fffffep-1f);
        const unsigned long long R = static_cast<unsigned long long>(__float2uint_rz(rf * 0x1p32f)) << 32;
        nrm = fixed_root_value(q);
        const unsigned long long Dn = (q.X >> 1) + __umul64hi(q.N << 1, Al << 1);                 // <= 8, Q60
        const long long F = static_cast<long long>((1ull << 60) - __umul64hi(Dn, R));
        const long long fh = F >> 20;
        const unsigned long long S = (1ull << 60) + static_cast<unsigned long long>(F + ((fh * fh) >> 20));
        g = from_q63(__umul64hi(S << 3, R), -q.k);                                               // in [1/8, 1]
        return true;
    }
    nrm = sqrt(x);
    g = 1.0 / (nrm * (nrm + fabs(alpha)));
    return false;
}

// Factor the panel of columns k0 .. k0 + nb - 1 (rows k0 .. s - 1) of W (column-major, ld lds) by the calling
// CTA as CTA `rank` of `csize` (CLUSTER: a thread-block cluster, csize a power of two <= 16; otherwise one CTA).
// A column whose remaining norm is outside [2^-450, 2^450] is scaled by a power of two and its products are formed again:
// unscaled, g and the products over- or underflow.  H_j does not depend on the scale of v_j; R's entry takes it back.  A
// column whose squares below the diagonal all vanish (entries under 2^-537) has nothing to reflect, as one of zeros;
// where the sum of squares overflows, R's diagonal entry is infinite and the sketch counts as singular.
// W's panel columns become V (v_j from row j down, vp on the diagonal; g_j = 0 where nothing is reflected) with R
// above the diagonal; L[j * ldl + k] = v_j^T v_k (k < j), g and betas[k0 + j].  SMEM: panel is shared memory for
// this CTA's rows (kQrLd doubles each); otherwise the panel is worked on in place.
// Returns false when a wait for the cluster's sums gave up.
template <bool CLUSTER, bool SMEM, int NT>
__device__ __forceinline__ bool qr_panel(double* W, int64_t lds, int s, int k0, int nb, double* L, int ldl, double* g,
                                         double* betas, double* panel, QrShared& sh, unsigned rank, unsigned csize) {
    constexpr int NW = NT / 32;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nrows = s - k0;
    const int rg = (nrows + kQrGroups - 1) / kQrGroups;          // rows of a group
    const int ng = kQrGroups / static_cast<int>(csize);          // groups of this CTA
    const int g0 = static_cast<int>(rank) * ng;
    const int rbeg = g0 * rg < nrows ? g0 * rg : nrows;
    const int rend = (g0 + ng) * rg < nrows ? (g0 + ng) * rg : nrows;
    double* Wp = W + static_cast<int64_t>(k0) * lds + k0;        // entry (0, 0) of the panel
    // entry (i, c) of the panel, i in [rbeg, rend), at P[(i - rbeg) * kSi + c * sc]
    constexpr int kSi = SMEM ? kQrLd : 1;
    const int64_t sc = SMEM ? 1 : lds;
    double* P = SMEM ? panel : Wp + rbeg;
    const uint32_t sh_addr = static_cast<uint32_t>(__cvta_generic_to_shared(&sh));
    auto at = [&](const void* p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)) - sh_addr; };
    uint32_t remote[4] = {0u, 0u, 0u, 0u};   // this thread's destinations: CTAs tid % 4 + 4 i
    if constexpr (CLUSTER) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const unsigned c = (tid & 3) + 4 * i;
            remote[i] = c < csize ? cluster_addr(sh_addr, c) : 0u;
        }
        if (tid == 0) {
            for (int p = 0; p < 2; ++p)
                asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(
                    static_cast<uint32_t>(__cvta_generic_to_shared(&sh.bar[p]))));
            asm volatile("fence.mbarrier_init.release.cluster;\n");
            qr_bar_arm(&sh.bar[0]);
            qr_bar_arm(&sh.bar[1]);
        }
    }
    if constexpr (SMEM) {
        for (int i = lane; i < rend - rbeg; i += 32) {
            double v[kQrB / NW];   // all columns of this warp in flight
#pragma unroll
            for (int u = 0; u < kQrB / NW; ++u) {
                const int c = warp + u * NW;
                v[u] = c < nb ? Wp[static_cast<int64_t>(c) * lds + rbeg + i] : 0.0;
            }
#pragma unroll
            for (int u = 0; u < kQrB / NW; ++u) P[i * kQrLd + warp + u * NW] = v[u];
        }
    }
    __syncthreads();
    if constexpr (CLUSTER) cluster_sync_all();   // every CTA runs, its barriers set, before the first remote store
    const bool mine = lane < nb;
    double* Pl = P + (mine ? lane : 0) * sc;     // this lane's column
    bool ok = true;
    // Rows of group g0 + q from row `from` on: a -= x w, x the entry of column j (UPD: skipped before the first
    // column), and the products with column j + 1's entry over the rows below its pivot row.  One pass over the
    // panel per column: the new entries are multiplied while they are in registers.
    auto rows_step = [&](auto upd, int q, int j, double w) {
        constexpr bool UPD = decltype(upd)::value;
        int i = ((g0 + q) * rg > j + 2 ? (g0 + q) * rg : j + 2) - rbeg;
        const int i1 = ((g0 + q + 1) * rg < nrows ? (g0 + q + 1) * rg : nrows) - rbeg;
        const double* Pj = P + (UPD ? j : 0) * sc;
        double d[4] = {0.0, 0.0, 0.0, 0.0};
        for (; i + 7 < i1; i += 8) {
            double x[8], v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                v[u] = Pl[(i + u) * kSi];
                if constexpr (UPD) x[u] = Pj[(i + u) * kSi];
            }
            if constexpr (UPD) {
#pragma unroll
                for (int u = 0; u < 8; ++u) v[u] = fma(-x[u], w, v[u]);
#pragma unroll
                for (int u = 0; u < 8; ++u)
                    if (mine) Pl[(i + u) * kSi] = v[u];
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) d[u & 3] = fma(__shfl_sync(0xffffffffu, v[u], j + 1), v[u], d[u & 3]);
        }
        // the last rows, the fewer than eight in flight together as well
        double x[8], v[8];
#pragma unroll
        for (int u = 0; u < 7; ++u) {
            v[u] = i + u < i1 ? Pl[(i + u) * kSi] : 0.0;
            if constexpr (UPD) x[u] = i + u < i1 ? Pj[(i + u) * kSi] : 0.0;
        }
#pragma unroll
        for (int u = 0; u < 7; ++u)
            if (i + u < i1) {
                if constexpr (UPD) {
                    v[u] = fma(-x[u], w, v[u]);
                    if (mine) Pl[(i + u) * kSi] = v[u];
                }
                d[u & 3] = fma(__shfl_sync(0xffffffffu, v[u], j + 1), v[u], d[u & 3]);
            }
        sh.part[q][lane] = mine ? (d[0] + d[1]) + (d[2] + d[3]) : 0.0;
    };
    int pg = -g0, pend = rg;                     // the pivot row's group within this CTA, and that group's end
    // Pivot row j and the products of column j with every column, formed from the panel for exchange `ex`.
    auto products = [&](int j, int ex) {
        if (pg >= 0 && pg < ng && warp == pg % NW) {
            const double v = mine ? Pl[(j - rbeg) * kSi] : 0.0;
            if constexpr (CLUSTER) sh.row_out[lane] = v;
            else sh.row[ex & 1][lane] = v;
        }
        for (int q = warp; q < ng; q += NW) rows_step(std::false_type{}, q, j - 1, 0.0);
    };
    // The columns from j0 on; ex: exchanges so far.  Returns nb, or (not SCALE) the column that needs scaling, its exchange
    // made.  SCALE is a loop of its own, so that the usual one holds nothing of it (3 us a panel otherwise).
    auto columns = [&](auto scale_t, int j0, int ex) -> int {
        constexpr bool SCALE = decltype(scale_t)::value;
        bool scaled = false;                         // the current column is scaled,
        double unscale = 1.0;                        // and this takes it back
        for (int j = j0; j < nb;) {
            const int par = ex & 1;
            const bool owner_cta = pg >= 0 && pg < ng, owner = owner_cta && warp == pg % NW;
            __syncthreads();
            for (int e = tid; e < ng / 4 * 128; e += NT) {
                const int q = e >> 7, col = (e & 127) >> 2, sub = e & 3;
                if constexpr (CLUSTER) {
                    if (owner_cta && q == 0) {
                        const double v = sh.row_out[col];
#pragma unroll
                        for (int i = 0; i < 4; ++i)
                            if ((tid & 3) + 4 * i < csize)
                                st_async(remote[i] + at(&sh.row[par][col]), remote[i] + at(&sh.bar[par]), v);
                    }
                }
                double v = sh.part[4 * q + sub][col];
                v += __shfl_xor_sync(0xffffffffu, v, 1);
                v += __shfl_xor_sync(0xffffffffu, v, 2);
                if constexpr (CLUSTER) {
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        if ((tid & 3) + 4 * i < csize)
                            st_async(remote[i] + at(&sh.quad[par][g0 / 4 + q][col]), remote[i] + at(&sh.bar[par]), v);
                } else {
                    if (sub == 0) sh.quad[par][q][col] = v;
                }
            }
            if constexpr (CLUSTER) {
                if (ok) ok = qr_bar_wait(&sh.bar[par], static_cast<uint32_t>((ex >> 1) & 1));
                __syncwarp();
            } else {
                __syncthreads();
            }
            if (tid < 128) {
                const int col = tid >> 2, sub = tid & 3;
                double v = (sh.quad[par][sub][col] + sh.quad[par][sub + 4][col]) +
                           (sh.quad[par][sub + 8][col] + sh.quad[par][sub + 12][col]);
                v += __shfl_xor_sync(0xffffffffu, v, 1);
                v += __shfl_xor_sync(0xffffffffu, v, 2);
                if (sub == 0) sh.D[col] = v;
            }
            __syncthreads();
            // every thread has seen this phase; the next one of this barrier cannot complete before it is armed
            if (CLUSTER && tid == 0) qr_bar_arm(&sh.bar[par]);
            ++ex;
            // v = x - beta e_j with beta = -sign(alpha) nrm; t = v^T a_k, w = g t
            const double rk = sh.row[par][lane], alpha = sh.row[par][j], sigma = sh.D[j];
            const double u = fma(alpha, rk, sh.D[lane]), x = fma(alpha, alpha, sigma);
            const bool reflect = (__double_as_longlong(sigma) << 1) != 0;   // else nothing to reflect: v = 0
            double nrm = 0.0, gj = 0.0;
            const bool in_range = !reflect || qr_scalars(alpha, x, nrm, gj);
            if (!in_range) {   // (the same x in every thread of every CTA)
                if constexpr (!SCALE) return j;
                if (!scaled && isfinite(x)) {
                    const bool up = x < 1.0;
                    const double f = up ? 0x1p500 : 0x1p-600;
                    unscale = up ? 0x1p-500 : 0x1p600;
                    scaled = true;
                    for (int q = warp; q < ng; q += NW) {
                        const int ib = (g0 + q) * rg > j ? (g0 + q) * rg : j;
                        const int ie = (g0 + q + 1) * rg < nrows ? (g0 + q + 1) * rg : nrows;
                        for (int i = ib + lane; i < ie; i += 32) P[(i - rbeg) * kSi + j * sc] *= f;
                    }
                    __syncwarp();
                    products(j, ex);
                    continue;
                }
            }
            const double sn = alpha >= 0.0 ? nrm : -nrm;
            const double t = reflect ? fma(sn, rk, u) : 0.0;
            const double vp = reflect ? alpha + sn : 0.0;
            const double w = (lane > j && mine) ? gj * t : 0.0;
            if (rank == 0 && warp == 0) {
                if (lane < j) L[j * ldl + lane] = t;
                if (lane == j) {
                    g[j] = gj;
                    const double d = reflect ? -sn : alpha;
                    betas[k0 + j] = SCALE ? d * unscale : d;
                }
            }
            if (owner && mine && lane >= j) Pl[(j - rbeg) * kSi] = lane == j ? vp : fma(-vp, w, rk);
            if (j + 1 == nb) break;
            // the next pivot row first
            if (j + 1 == pend) {
                ++pg;
                pend += rg;
            }
            if (pg >= 0 && pg < ng && warp == pg % NW) {
                double v = 0.0;
                if (mine) {
                    v = fma(-P[(j + 1 - rbeg) * kSi + j * sc], w, Pl[(j + 1 - rbeg) * kSi]);
                    Pl[(j + 1 - rbeg) * kSi] = v;
                }
                if constexpr (CLUSTER) sh.row_out[lane] = v;
                else sh.row[par ^ 1][lane] = v;
            }
            for (int q = warp; q < ng; q += NW) rows_step(std::true_type{}, q, j, w);
            __syncwarp();
            ++j;
            scaled = false;
            unscale = 1.0;
        }
        return nb;
    };
    products(0, 0);
    const int stop = columns(std::false_type{}, 0, 0);
    if (stop < nb) {   // from here on, this column's products once more
        products(stop, stop + 1);
        columns(std::true_type{}, stop, stop + 1);
    }
    __syncthreads();
    if constexpr (SMEM) {
        for (int c = warp; c < nb; c += NW)
            for (int i = lane; i < rend - rbeg; i += 32)
                Wp[static_cast<int64_t>(c) * lds + rbeg + i] = P[i * kQrLd + c];
    }
    if constexpr (CLUSTER) cluster_sync_all();   // no CTA leaves while another may still store into it
    return ok;
}

// One warp: rows i0 .. i1 - 1 of Y = V^T C, sixteen columns of V (16 mt ..) by eight of C (entry (0, 0) at C, ld
// lds; ncol valid), into out[col * kQrB + k].  V: the panel just factored (entry (0, 0) at Wp, nb columns, nrows
// rows).
__device__ __forceinline__ void qr_y_tile(const double* Wp, const double* C, int64_t lds, int nrows, int nb, int ncol, int mt,
                                          int i0, int i1, double* out) {
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    if (i1 > nrows) i1 = nrows;
#pragma unroll 2
    for (int k = i0; k < i1; k += 16) {
        double a[8], b[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int r = k + t + 4 * i;
            b[i] = (r < i1 && g < ncol) ? C[static_cast<int64_t>(g) * lds + r] : 0.0;
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int c = 16 * mt + g + 8 * (i & 1), r = k + t + 4 * (i >> 1);
            a[i] = (r < i1 && c < nb && r >= c) ? Wp[static_cast<int64_t>(c) * lds + r] : 0.0;
        }
        mma_f64_16816(acc, a, b);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) out[(2 * t + (i & 1)) * kQrB + 16 * mt + g + 8 * (i >> 1)] = acc[i];
}

// Column solve (one warp, lane = panel column): (D + L) z = y, y in the lane; Ls: L in shared memory (ld kQrLd).
__device__ __forceinline__ double qr_z_solve(double y, const double* Ls, double gl, int nb) {
    const int lane = threadIdx.x & 31;
    double z = 0.0;
    for (int j = 0; j < nb; ++j) {
        const double zj = __shfl_sync(0xffffffffu, y * gl, j);
        if (lane == j) z = zj;
        if (lane > j) y = fma(-Ls[lane * kQrLd + j], zj, y);
    }
    return lane < nb ? z : 0.0;
}

// One warp: rows r0 .. r0 + 15 of C -= V Z for eight columns (Z: [col * kQrB + k]).
__device__ __forceinline__ void qr_update_tile(const double* Wp, double* C, int64_t lds, int nrows, int nb, int ncol, int r0,
                                               const double* Z) {
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    double acc[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int r = r0 + g + 8 * (i >> 1), c = 2 * t + (i & 1);
        acc[i] = (r < nrows && c < ncol) ? C[static_cast<int64_t>(c) * lds + r] : 0.0;
    }
#pragma unroll
    for (int kt = 0; kt < 2; ++kt) {
        double a[8], b[4];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int r = r0 + g + 8 * (i & 1), c = 16 * kt + t + 4 * (i >> 1);
            a[i] = (r < nrows && c < nb && r >= c) ? Wp[static_cast<int64_t>(c) * lds + r] : 0.0;
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) b[i] = g < ncol ? -Z[g * kQrB + 16 * kt + t + 4 * i] : 0.0;
        mma_f64_16816(acc, a, b);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int r = r0 + g + 8 * (i >> 1), c = 2 * t + (i & 1);
        if (r < nrows && c < ncol) C[static_cast<int64_t>(c) * lds + r] = acc[i];
    }
}

// Entry e of R_s (np x np row-major, identity padding): each row negated where its diagonal is negative.
// Returns false for a diagonal that is 0, subnormal or not finite.
__device__ __forceinline__ bool qr_out_entry(const double* W, int64_t lds, int n, int np, const double* betas, int e,
                                             double* Rs, double* Rs_user) {
    const int r = e / np, c = e - r * np;
    if (r >= n || c >= n) {
        Rs[e] = r == c ? 1.0 : 0.0;
        return true;
    }
    const double d = betas[r];
    const double v = c > r ? (d < 0.0 ? -1.0 : 1.0) * W[static_cast<int64_t>(c) * lds + r] : (c == r ? fabs(d) : 0.0);
    Rs[e] = v;
    if (Rs_user) Rs_user[static_cast<int64_t>(r) * n + c] = v;
    return c != r || (isfinite(d) && fabs(d) >= DBL_MIN);
}

// Shared memory one CTA alone needs: QrShared, L, g, betas, and a region that holds first the panel (where it
// fits: qr_one_bytes with the sample's rows), then the Y partials and Z of eight columns.
constexpr int kQrOneY = 8 * kQrB * (kQrMaxChunks + 1);
__host__ __device__ constexpr size_t qr_one_fixed(int n) {
    return sizeof(QrShared) + sizeof(double) * (kQrB * kQrLd + kQrB + static_cast<size_t>(n));
}
__host__ __device__ constexpr size_t qr_one_bytes(int n, int rows) {
    return qr_one_fixed(n) + sizeof(double) * (rows * kQrLd > kQrOneY ? static_cast<size_t>(rows) * kQrLd : kQrOneY);
}

// The whole factorisation by one CTA of NT threads (a multiple of 128): the cluster's bits.  sm: `smem_bytes`
// of shared memory, at least qr_one_bytes(n, 0); the panel stays in it where it fits, else in W.
template <int NT>
__device__ __forceinline__ void qr_factor_one_cta(double* W, int64_t lds, int s, int n, int np, double* Rs, int32_t* info,
                                                  double* sm, size_t smem_bytes) {
    constexpr int NW = NT / 32;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    QrShared& sh = *reinterpret_cast<QrShared*>(sm);
    double* Ls = sm + sizeof(QrShared) / sizeof(double);
    double* gs = Ls + kQrB * kQrLd;
    double* betas = gs + kQrB;
    double* Y = betas + n;                    // partials by chunk, then the eight Z columns; before them the panel
    double* Zs = Y + 8 * kQrB * kQrMaxChunks;
    for (int k0 = 0; k0 < n; k0 += kQrB) {
        const int nb = n - k0 < kQrB ? n - k0 : kQrB, nrows = s - k0;
        const bool fits = qr_one_bytes(n, nrows) <= smem_bytes;
        if (fits) qr_panel<false, true, NT>(W, lds, s, k0, nb, Ls, kQrLd, gs, betas, Y, sh, 0u, 1u);
        else qr_panel<false, false, NT>(W, lds, s, k0, nb, Ls, kQrLd, gs, betas, nullptr, sh, 0u, 1u);
        __syncthreads();
        const double* Wp = W + static_cast<int64_t>(k0) * lds + k0;
        const int nt = n - k0 - nb, ch = qr_chunk_rows(nrows), nchunks = (nrows + ch - 1) / ch;
        for (int c0 = 0; c0 < nt; c0 += 8) {
            const int ncol = nt - c0 < 8 ? nt - c0 : 8;
            double* C = W + static_cast<int64_t>(k0 + nb + c0) * lds + k0;
            for (int e = warp; e < 2 * nchunks; e += NW)
                qr_y_tile(Wp, C, lds, nrows, nb, ncol, e & 1, (e >> 1) * ch, ((e >> 1) + 1) * ch, Y + (e >> 1) * 8 * kQrB);
            __syncthreads();
            for (int col = warp; col < 8; col += NW) {
                double y = 0.0;
                for (int q = 0; q < nchunks; ++q) y += Y[q * 8 * kQrB + col * kQrB + lane];
                Zs[col * kQrB + lane] = qr_z_solve(y, Ls, lane < nb ? gs[lane] : 0.0, nb);
            }
            __syncthreads();
            for (int r0 = 16 * warp; r0 < nrows; r0 += 16 * NW) qr_update_tile(Wp, C, lds, nrows, nb, ncol, r0, Zs);
            __syncthreads();
        }
    }
    bool ok = true;
    for (int e = tid; e < np * np; e += NT) ok = qr_out_entry(W, lds, n, np, betas, e, Rs, nullptr) && ok;
    if (__syncthreads_or(!ok) && tid == 0) set_status(info, RPCHOLQR_ERR_SINGULAR_SKETCH);
}

}  // namespace rpq
