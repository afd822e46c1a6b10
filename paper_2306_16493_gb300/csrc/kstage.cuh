// Re->k sums of many grid points, factorised over the lattice axes (internal).
//
// A(k)[row][j] = sum_Re e^{ik.Re} w g(Re)[row][j] is needed at every window k-point.  With R_e in
// its bounding cube [-r, r]^3 (D = 2r + 1) the phase is a product over the axes, so
//   T1[n1 n2][k3] = sum_n3 e3 g,   T2[n1][k2 k3] = sum_n2 e2 T1,   A(k) = sum_n1 e1 T2,
// and the first two stages are shared by the k-points with the same k3 and by those of the same
// (k2, k3) column.  Per k-point the sum shrinks from n_Re to D terms, plus its share of the
// column's D^2.  Measured against the direct sum (one GB300): metal 48^3, 5^3 R_e, 6000 columns of g
// per R_e in FP32: 6.8 -> 0.69 ms; Si-like 100^3, 7^3 R_e: 53 -> 2.2 ms; Al-like 20^3 in FP64:
// 19.5 -> 1.45 ms.  What remains is writing T2 once, reading it once and writing ghat.  The
// errors against 64 bits fall (shorter sums).  The U^dag(k) contraction follows in the last stage, where an Epilogue writes
// the value of (state, row) in the layout of the kernel that reads it.
#pragma once

#include "epwi_internal.cuh"
#include "scatter.cuh"

// The (k2, k3) columns of a list of k-points, k3-major (device arrays).
struct ColumnSet {
    int ncol = 0, nk3 = 0, max_kp = 0;
    const int *id = nullptr;       // [ncol] k3 N2 + k2, ascending
    const int *start = nullptr;    // [ncol + 1] first entry of each column in kp
    const int *kp = nullptr;       // [nkp] list positions, grouped by column
    const int *k3 = nullptr;       // [nk3] distinct k3
    const int *k3col = nullptr;    // [nk3 + 1] first column of each distinct k3
};

// Builds the columns of kpts[0 .. nkp-1] in c->col_buf (synchronises the stream for the counts).
ColumnSet build_columns(epwi_ctx *c, const int *kpts, int64_t nkp);

// Multiply-adds of both forms per column of g, the factorised one twice over for its extra passes
// through T1 and T2; below the work that the column lists' launches and one synchronisation (about
// 40 us) are worth, the direct sum stays (tiny 8^3: 25 us).
inline bool ks_pays(int D, int nRe, int64_t nkp, double nk3, double ncol, int64_t nrow, int nw, bool fp64) {
    const double direct = (double)nRe * nkp, fac = (double)D * D * (D * nk3 + ncol) + (double)D * nkp;
    return 2.0 * fac < direct && direct * (double)nrow * nw > (fp64 ? 1e7 : 2e8);
}
// Whether the factorised sum is the faster one for a work set of nkp k-points of the current grid.
bool kstage_pays(const epwi_ctx *c, int64_t nkp, int64_t nrow, bool fp64);

// Rows per block so that the workspaces T1 [D D][nk3] and T2 [D][ncol] (times rows times W) stay within
// 1 GiB.  Fewer than one CTA's rows leave lanes idle, so a block has at least that many up to 4 GiB; beyond (wide
// planes with hundreds of thousands of columns) it has what 4 GiB hold.
inline int64_t ks_block_rows(int64_t D, int64_t nk3, int64_t ncol, int64_t nrow, int W, size_t elem, int cta) {
    const double per_row = ((double)D * D * nk3 + (double)D * ncol) * W * elem;
    const int64_t fit = (int64_t)((double)(int64_t(1) << 30) / per_row), most = (int64_t)((double)(int64_t(1) << 32) / per_row);
    if (fit >= nrow) return nrow;
    const int64_t cap = fit >= cta ? fit : most >= cta ? cta : most > 1 ? most : 1;
    const int64_t blocks = (nrow + cap - 1) / cap, rows = (nrow + blocks - 1) / blocks;      // equal blocks,
    const int64_t whole = cap >= cta ? (rows + cta - 1) / cta * cta : rows;                 // whole CTAs of rows
    return whole < nrow ? whole : nrow;
}

constexpr int kKsThreads = 128;    // rows per block of the last stage
constexpr int kKsBatch = 16;       // k-points staged at once

template <class C2>
struct KStageArgs {
    RestageArgs ra;
    ColumnSet cs;
    const C2 *T2;                  // [n1][ncol][rows of the block][W]
    const C2 *ph, *V;
    int D, rc;
    int row0, nrows;               // row block
};

__device__ __forceinline__ float2 cfma_t(float2 a, float2 b, float2 c) { return cfmaf(a, b, c); }
__device__ __forceinline__ double2 cfma_t(double2 a, double2 b, double2 c) { return cfma(a, b, c); }

template <class C2>
__device__ __forceinline__ C2 ks_phase(const C2 *ph, int n, int k, int s, int L) {
    int t = (int)((int64_t)n * k * s % L);
    return ph[t < 0 ? t + L : t];
}

// Last stage: one thread per row of one column.  The column's D W values of the row stay in
// registers while the block walks the column's k-points (WT, DT > 0); otherwise they are read
// again for each k-point.
template <class C2, int WT, int DT, class Epi>
__global__ void __launch_bounds__(kKsThreads) k_ks_axis1(KStageArgs<C2> a, Epi epi) {
    constexpr int WM = WT ? WT : epc::kMaxW;
    constexpr int DM = DT ? DT : 1;
    const int W = WT ? WT : a.ra.W;
    const int D = DT ? DT : a.D;
    __shared__ C2 P[kKsBatch][13];
    __shared__ int s_ik[kKsBatch], s_lo[kKsBatch], s_ns[kKsBatch];
    __shared__ int64_t s_s0[kKsBatch];
    const int col = blockIdx.x;                  // x: a grid can have more than 65535 columns
    const int r = blockIdx.y * kKsThreads + threadIdx.x;
    const bool live = r < a.nrows;
    const int64_t stride = (int64_t)a.cs.ncol * a.nrows * W;          // n1 stride of T2
    const C2 *src = a.T2 + ((int64_t)col * a.nrows + (live ? r : 0)) * W;
    C2 t2[DM][WT ? WT : 1];
    if constexpr (DT > 0) {
#pragma unroll
        for (int d = 0; d < DT; ++d)
#pragma unroll
            for (int j = 0; j < WM; ++j) t2[d][j] = src[d * stride + j];
    }
    const int p0 = a.cs.start[col], p1 = a.cs.start[col + 1];
    for (int b = p0; b < p1; b += kKsBatch) {
        const int nb = min(kKsBatch, p1 - b);
        __syncthreads();
        for (int e = threadIdx.x; e < nb * D; e += kKsThreads) {
            const int x = e / D, d = e - x * D;
            const int kp = a.cs.kp[b + x], ik = a.ra.kpts[kp];
            const int k1 = ik / (a.ra.g.n2 * a.ra.g.n3);
            P[x][d] = ks_phase(a.ph, d - a.rc, k1, a.ra.g.s1, a.ra.g.L);
            if (d == 0) {
                s_ik[x] = ik;
                s_lo[x] = a.ra.ovr_nsel >= 0 ? a.ra.ovr_lo : a.ra.win_lo[ik];
                s_ns[x] = a.ra.ovr_nsel >= 0 ? a.ra.ovr_nsel : a.ra.win_n[ik];
                s_s0[x] = a.ra.kp_state[kp] - a.ra.s_base;
            }
        }
        __syncthreads();
        if (!live) continue;
        for (int x = 0; x < nb; ++x) {
            C2 acc[WM];
            for (int j = 0; j < W; ++j) {
                C2 s;
                s.x = 0;
                s.y = 0;
                if constexpr (DT > 0) {
#pragma unroll
                    for (int d = 0; d < DT; ++d) s = cfma_t(P[x][d], t2[d][j], s);
                } else {
                    for (int d = 0; d < D; ++d) s = cfma_t(P[x][d], src[d * stride + j], s);
                }
                acc[j] = s;
            }
            const C2 *Vk = a.V + (int64_t)s_ik[x] * W * W + s_lo[x];
            for (int np = 0; np < s_ns[x]; ++np) {
                C2 o;
                o.x = 0;
                o.y = 0;
                for (int j = 0; j < W; ++j) o = cfma_t(acc[j], Vk[j * W + np], o);
                epi(s_s0[x] + np, a.row0 + r, o);
            }
        }
    }
}

// Stages 1 and 2 of rows [row0, row0 + nrows) into T2 (kstage.cu).
template <class C2>
void kstage_axes32(epwi_ctx *c, const ColumnSet &cs, const C2 *g, const C2 *ph, int64_t nrow, int W, int row0,
                   int nrows, C2 *T1, C2 *T2);

template <class C2, class Epi>
void kstage_run(epwi_ctx *c, const RestageArgs &ra, const C2 *g, const C2 *ph, const C2 *V, const Epi &epi) {
    const ColumnSet cs = build_columns(c, ra.kpts, ra.nkp);
    if (cs.ncol == 0) return;
    const int W = ra.W, D = 2 * c->fac_re_r + 1;
    const int64_t rows = ks_block_rows(D, cs.nk3, cs.ncol, ra.nrow, W, sizeof(C2), kKsThreads);
    const int64_t n1 = (int64_t)D * D * cs.nk3 * rows * W, n2 = (int64_t)D * cs.ncol * rows * W;
    c->ks_T.ensure(sizeof(C2) * (n1 + n2));
    KStageArgs<C2> a;
    a.ra = ra;
    a.cs = cs;
    a.ph = ph;
    a.V = V;
    a.D = D;
    a.rc = c->fac_re_r;
    a.T2 = c->ks_T.as<C2>() + n1;
    for (int64_t r0 = 0; r0 < ra.nrow; r0 += rows) {
        a.row0 = (int)r0;
        a.nrows = (int)(ra.nrow - r0 < rows ? ra.nrow - r0 : rows);
        kstage_axes32<C2>(c, cs, g, ph, ra.nrow, W, a.row0, a.nrows, c->ks_T.as<C2>(), c->ks_T.as<C2>() + n1);
        const dim3 grid((unsigned)cs.ncol, (unsigned)((a.nrows + kKsThreads - 1) / kKsThreads));
        // registers hold a column's D W values up to 112 (FP32) or 56 (FP64) of them
        constexpr bool f32 = sizeof(C2) == sizeof(float2);
        if (W == 4 && D == 3) k_ks_axis1<C2, 4, 3><<<grid, kKsThreads, 0, c->stream>>>(a, epi);
        else if (W == 4 && D == 5) k_ks_axis1<C2, 4, 5><<<grid, kKsThreads, 0, c->stream>>>(a, epi);
        else if (W == 4 && D == 7) k_ks_axis1<C2, 4, 7><<<grid, kKsThreads, 0, c->stream>>>(a, epi);
        else if (W == 8 && D == 3) k_ks_axis1<C2, 8, 3><<<grid, kKsThreads, 0, c->stream>>>(a, epi);
        else if (W == 8 && D == 5 && f32) k_ks_axis1<C2, 8, (f32 ? 5 : 0)><<<grid, kKsThreads, 0, c->stream>>>(a, epi);
        else if (W == 8 && D == 7 && f32) k_ks_axis1<C2, 8, (f32 ? 7 : 0)><<<grid, kKsThreads, 0, c->stream>>>(a, epi);
        else k_ks_axis1<C2, 0, 0><<<grid, kKsThreads, 0, c->stream>>>(a, epi);
        EPWI_CHECK_LAUNCH();
    }
}
