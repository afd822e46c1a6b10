// The (k2, k3) columns of a k-point list, and the first two stages of the factorised Re->k sum
// (kstage.cuh).
#include <algorithm>

#include "kstage.cuh"

namespace {

__global__ void k_col_count(int64_t nkp, const int *__restrict__ kpts, int N2, int N3, int *__restrict__ cnt) {
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= nkp) return;
    const int t = kpts[p] % (N2 * N3), k2 = t / N3, k3 = t - k2 * N3;
    atomicAdd(&cnt[k3 * N2 + k2], 1);
}

// Exclusive scan over the block of (a, b) packed in one 64-bit word; total in tot.
__device__ int64_t scan_pair(int64_t v, int64_t *sm, int64_t &tot) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int64_t x = v;
    for (int o = 1; o < 32; o <<= 1) {
        const int64_t t = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += t;
    }
    if (lane == 31) sm[wid] = x;
    __syncthreads();
    if (wid == 0) {
        int64_t s = sm[lane];
        for (int o = 1; o < 32; o <<= 1) {
            const int64_t t = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += t;
        }
        sm[lane] = s;
    }
    __syncthreads();
    const int64_t r = x - v + (wid ? sm[wid - 1] : 0);
    tot = sm[31];
    __syncthreads();
    return r;
}

// One block: the non-empty columns in k3-major order with their offsets, the distinct k3 with
// their first columns, and hdr = {columns, distinct k3, largest column}.  A grid has at most a
// few 10^4 columns, a few steps of this block.
__global__ void __launch_bounds__(1024) k_col_scan(int N2, int N3, const int *__restrict__ cnt, int *__restrict__ cursor,
                                                   int *__restrict__ id, int *__restrict__ start, int *__restrict__ k3,
                                                   int *__restrict__ k3col, int *__restrict__ hdr) {
    __shared__ int64_t sm[32];
    __shared__ int s_max;
    if (threadIdx.x == 0) s_max = 0;
    __syncthreads();
    const int n = N2 * N3;
    int64_t base = 0;                             // (columns, k-points) before this step
    for (int c0 = 0; c0 < n; c0 += 1024) {
        const int c = c0 + threadIdx.x;
        const int m = c < n ? cnt[c] : 0;
        int64_t tot;
        const int64_t off = base + scan_pair(m > 0 ? ((int64_t)1 << 32) + m : 0, sm, tot);
        if (m > 0) {
            id[off >> 32] = c;
            start[off >> 32] = (int)(off & 0xffffffff);
            cursor[c] = (int)(off & 0xffffffff);
            atomicMax(&s_max, m);
        }
        base += tot;
    }
    const int ncol = (int)(base >> 32);
    if (threadIdx.x == 0) start[ncol] = (int)(base & 0xffffffff);
    __syncthreads();
    int64_t b3 = 0;
    for (int c0 = 0; c0 < ncol; c0 += 1024) {
        const int c = c0 + threadIdx.x;
        const bool first = c < ncol && (c == 0 || id[c] / N2 != id[c - 1] / N2);
        int64_t tot;
        const int64_t off = b3 + scan_pair(first ? 1 : 0, sm, tot);
        if (first) {
            k3[off] = id[c] / N2;
            k3col[off] = c;
        }
        b3 += tot;
    }
    if (threadIdx.x == 0) {
        k3col[b3] = ncol;
        hdr[0] = ncol;
        hdr[1] = (int)b3;
        hdr[2] = s_max;
    }
}

__global__ void k_col_fill(int64_t nkp, const int *__restrict__ kpts, int N2, int N3, int *__restrict__ cursor,
                           int *__restrict__ kp) {
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= nkp) return;
    const int t = kpts[p] % (N2 * N3), k2 = t / N3, k3 = t - k2 * N3;
    kp[atomicAdd(&cursor[k3 * N2 + k2], 1)] = (int)p;
}

constexpr int kAxThreads = 256;
constexpr int kAxBatch = 32;       // k3 values / columns whose phases are staged at once

// T1[n1 n2][k3 i][e] = sum_n3 e3(k3) g(n1 n2 n3)[e]: one thread per element holds its D values
// of g in registers (g is read once) and walks the k3 values of the list.
template <class C2, int DT>
__global__ void __launch_bounds__(kAxThreads) k_ks_axis3(int rc, const int *__restrict__ cube, const C2 *__restrict__ g,
                                                         int64_t re_stride, int64_t e0, int64_t ne, int nk3,
                                                         const int *__restrict__ k3, int s3, int L,
                                                         const C2 *__restrict__ ph, C2 *__restrict__ T1) {
    __shared__ C2 P[kAxBatch][DT];
    const int64_t e = (int64_t)blockIdx.x * kAxThreads + threadIdx.x;
    const int n12 = blockIdx.y;
    const int b0 = blockIdx.z * kAxBatch, nb = min(kAxBatch, nk3 - b0);
    for (int x = threadIdx.x; x < nb * DT; x += kAxThreads)
        P[x / DT][x % DT] = ks_phase(ph, x % DT - rc, k3[b0 + x / DT], s3, L);
    __syncthreads();
    if (e >= ne) return;
    C2 v[DT];
#pragma unroll
    for (int d = 0; d < DT; ++d) {
        const int re = cube[n12 * DT + d];       // uniform over the block; -1: not in the set
        v[d].x = 0;
        v[d].y = 0;
        if (re >= 0) v[d] = g[re * re_stride + e0 + e];
    }
    for (int x = 0; x < nb; ++x) {
        C2 s;
        s.x = 0;
        s.y = 0;
#pragma unroll
        for (int d = 0; d < DT; ++d) s = cfma_t(P[x][d], v[d], s);
        T1[((int64_t)n12 * nk3 + b0 + x) * ne + e] = s;
    }
}

// T2[n1][col][e] = sum_n2 e2(k2) T1[n1 n2][k3][e] for the columns of one k3: one thread per
// element holds its D values of T1 and walks the columns.
template <class C2, int DT>
__global__ void __launch_bounds__(kAxThreads) k_ks_axis2(int rc, int64_t ne, ColumnSet cs, int N2, int s2, int L,
                                                         const C2 *__restrict__ ph, const C2 *__restrict__ T1,
                                                         C2 *__restrict__ T2) {
    __shared__ C2 P[kAxBatch][DT];
    const int64_t e = (int64_t)blockIdx.x * kAxThreads + threadIdx.x;
    const int n1 = blockIdx.y, i3 = blockIdx.z;
    const int c0 = cs.k3col[i3], c1 = cs.k3col[i3 + 1];
    C2 v[DT];
    if (e < ne) {
#pragma unroll
        for (int d = 0; d < DT; ++d) v[d] = T1[((int64_t)(n1 * DT + d) * cs.nk3 + i3) * ne + e];
    }
    for (int b = c0; b < c1; b += kAxBatch) {
        const int nb = min(kAxBatch, c1 - b);
        __syncthreads();
        for (int x = threadIdx.x; x < nb * DT; x += kAxThreads)
            P[x / DT][x % DT] = ks_phase(ph, x % DT - rc, cs.id[b + x / DT] % N2, s2, L);
        __syncthreads();
        if (e >= ne) continue;
        for (int x = 0; x < nb; ++x) {
            C2 s;
            s.x = 0;
            s.y = 0;
#pragma unroll
            for (int d = 0; d < DT; ++d) s = cfma_t(P[x][d], v[d], s);
            T2[((int64_t)n1 * cs.ncol + b + x) * ne + e] = s;
        }
    }
}

template <class C2, int DT>
void axes32(epwi_ctx *c, const ColumnSet &cs, const C2 *g, const C2 *ph, int64_t nrow, int W, int row0, int nrows,
            C2 *T1, C2 *T2) {
    const GridInfo gi = make_grid_info(c);
    const int64_t ne = (int64_t)nrows * W;
    const unsigned nb = (unsigned)((ne + kAxThreads - 1) / kAxThreads);
    const int rc = c->fac_re_r;
    k_ks_axis3<C2, DT><<<dim3(nb, DT * DT, (unsigned)((cs.nk3 + kAxBatch - 1) / kAxBatch)), kAxThreads, 0, c->stream>>>(
        rc, c->re_cube.as<int>(), g, nrow * W, (int64_t)row0 * W, ne, cs.nk3, cs.k3, gi.s3, gi.L, ph, T1);
    EPWI_CHECK_LAUNCH();
    k_ks_axis2<C2, DT><<<dim3(nb, DT, (unsigned)cs.nk3), kAxThreads, 0, c->stream>>>(rc, ne, cs, gi.n2, gi.s2, gi.L, ph,
                                                                                   T1, T2);
    EPWI_CHECK_LAUNCH();
}

}  // namespace

ColumnSet build_columns(epwi_ctx *c, const int *kpts, int64_t nkp) {
    ColumnSet cs;
    if (nkp <= 0) return cs;
    const int N2 = c->ng[1], N3 = c->ng[2];
    const int64_t n = (int64_t)N2 * N3, nc = std::min<int64_t>(n, nkp);
    // [cnt n][cursor n][id nc][start nc + 1][k3 N3][k3col N3 + 1][kp nkp][hdr 4]
    c->col_buf.ensure(sizeof(int) * (size_t)(2 * n + 2 * nc + 2 * N3 + nkp + 8));
    int *cnt = c->col_buf.as<int>(), *cursor = cnt + n, *id = cursor + n, *start = id + nc, *k3 = start + nc + 1,
        *k3col = k3 + N3, *kp = k3col + N3 + 1, *hdr = kp + nkp;
    EPWI_CUDA(cudaMemsetAsync(cnt, 0, sizeof(int) * n, c->stream));
    const unsigned nb = (unsigned)((nkp + 255) / 256);
    k_col_count<<<nb, 256, 0, c->stream>>>(nkp, kpts, N2, N3, cnt);
    EPWI_CHECK_LAUNCH();
    k_col_scan<<<1, 1024, 0, c->stream>>>(N2, N3, cnt, cursor, id, start, k3, k3col, hdr);
    EPWI_CHECK_LAUNCH();
    k_col_fill<<<nb, 256, 0, c->stream>>>(nkp, kpts, N2, N3, cursor, kp);
    EPWI_CHECK_LAUNCH();
    int h[3];
    EPWI_CUDA(cudaMemcpyAsync(h, hdr, sizeof(h), cudaMemcpyDeviceToHost, c->stream));
    EPWI_CUDA(cudaStreamSynchronize(c->stream));
    cs.ncol = h[0];
    cs.nk3 = h[1];
    cs.max_kp = h[2];
    cs.id = id;
    cs.start = start;
    cs.kp = kp;
    cs.k3 = k3;
    cs.k3col = k3col;
    return cs;
}

// The rule (ks_pays) with the window's counts of k3 and columns, or the largest the list can have.
bool kstage_pays(const epwi_ctx *c, int64_t nkp, int64_t nrow, bool fp64) {
    // one block scans the columns: leave planes of over 2^20 columns to the direct sum
    if (!c->re_cube_ok || nkp <= 0 || (int64_t)c->ng[1] * c->ng[2] > (1 << 20)) return false;
    double nk3 = (double)std::min<int64_t>(c->ng[2], nkp);
    double ncol = (double)std::min<int64_t>((int64_t)c->ng[1] * c->ng[2], nkp);
    if (c->win_ncol > 0 && nkp == c->nkp) {       // the window's own counts, where the sieve took them
        nk3 = c->win_nk3;
        ncol = c->win_ncol;
    }
    return ks_pays(2 * c->fac_re_r + 1, c->nRe, nkp, nk3, ncol, nrow, c->nw, fp64);
}

template <class C2>
void kstage_axes32(epwi_ctx *c, const ColumnSet &cs, const C2 *g, const C2 *ph, int64_t nrow, int W, int row0, int nrows,
                   C2 *T1, C2 *T2) {
    switch (2 * c->fac_re_r + 1) {
        case 1: axes32<C2, 1>(c, cs, g, ph, nrow, W, row0, nrows, T1, T2); break;
        case 3: axes32<C2, 3>(c, cs, g, ph, nrow, W, row0, nrows, T1, T2); break;
        case 5: axes32<C2, 5>(c, cs, g, ph, nrow, W, row0, nrows, T1, T2); break;
        case 7: axes32<C2, 7>(c, cs, g, ph, nrow, W, row0, nrows, T1, T2); break;
        case 9: axes32<C2, 9>(c, cs, g, ph, nrow, W, row0, nrows, T1, T2); break;
        case 11: axes32<C2, 11>(c, cs, g, ph, nrow, W, row0, nrows, T1, T2); break;
        case 13: axes32<C2, 13>(c, cs, g, ph, nrow, W, row0, nrows, T1, T2); break;
        default: throw EpwiError{EPWI_EUNSUPPORTED, "R_e beyond the factorised range"};
    }
}

template void kstage_axes32<float2>(epwi_ctx *, const ColumnSet &, const float2 *, const float2 *, int64_t, int, int, int,
                                    float2 *, float2 *);
template void kstage_axes32<double2>(epwi_ctx *, const ColumnSet &, const double2 *, const double2 *, int64_t, int, int,
                                     int, double2 *, double2 *);
