// Iterative Boltzmann transport equation (Sec. II C, the iteration equation after Eq. 10).
//
// Gamma storage: the sieved pairs of the window in pair order (k-point major, as the sieve
// writes them), and for every pair (k, q) one block Gamma[n][m] over the window bands n of k
// and m of k+q, blocks back to back.  A pair's block starts at its k-point's first entry, ent[k], plus
// the pair's 32-bit offset goff[pair].  The
// value stored is sum_nu |g|^2 [(N + f_m) e^{-x+^2/eta^2} + (1 + N - f_m) e^{-x-^2/eta^2}] (eV^2),
// the summand of Eq. 10 without its constant 2 pi / (hbar N_q sqrt(pi) eta), which the step
// applies once per state.
//
// Every Gamma entry has a 4-byte column word (written before the capture, with the offsets, in one
// pass over the pairs): the index of its final state
// (k+q, m) in the window's state list and the band n of k, (s << 5) | n.  The step is then a
// sparse product over entries, Gamma_e F_s accumulated into the row of band n of k: it reads one
// column word and one value per entry, gathers F at s, and needs no grid arithmetic or table
// lookups.  The pair list and the per-pair block offsets serve only the capture and are freed
// afterwards when they are large, so the resident index is the column word per entry plus 8 bytes per k-point
// (half the bytes of FP64 Gamma, equal to those of FP32 Gamma).
//
// Step: one block per window k-point, its entries split into eight contiguous warp ranges;
// lanes take entries 32 apart, several at a time with their loads issued together (coalesced
// column and value loads, F gathers from a table that stays in L2).  The k-point's bands are
// accumulated in registers in groups of 1, 2, 4 or 8 (the smallest covering the crystal's
// bands) with the band selection specialised to the window's exact band count (none for one
// band).  With FP32 Gamma (split paths) the lanes accumulate and reduce in FP32 from an FP32
// copy of F; the sum over warps, the per-state update and F itself are FP64.  Per-state sums
// are reduced in a fixed order (lanes by a butterfly, then warps in index order), so the result
// does not depend on scheduling.
#include <algorithm>
#include <cstring>
#include <type_traits>

#include "epwi_internal.cuh"
#include "scatter.cuh"
#include "scatter_sf.cuh"
#include "sieve.cuh"

namespace {

constexpr int kIbThreads = 256;
constexpr int kIbWarps = kIbThreads / 32;
constexpr int kIbMaxBands = 8;  // bands of k accumulated in registers at a time (at most)
constexpr int kIbUnroll = 4;    // entries per lane whose loads are issued together

// Per grid point: its first window state << 5 | window bands (0 bands outside the window).
__global__ void k_ib_points(int64_t nkp, const int *__restrict__ kpts, const int64_t *__restrict__ kp_state,
                            unsigned *__restrict__ pt) {
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p < nkp) pt[kpts[p]] = (unsigned)kp_state[p] << 5 | (unsigned)(kp_state[p + 1] - kp_state[p]);
}

// k+q of the pairs of one k-point, with the divisions by launch constants.
struct IbGrid {
    GridInfo g;
    FDiv fplane, fn3;
    int k1, k2, k3;
    __device__ __forceinline__ void at(int ik) { grid_coords(g, ik, k1, k2, k3); }
    __device__ __forceinline__ int64_t kq(int q) const {
        const int i1 = fdiv(q, fplane), r = q - i1 * (int)fplane.d, i2 = fdiv(r, fn3), i3 = r - i2 * g.n3;
        int b1 = k1 + i1, b2 = k2 + i2, b3 = k3 + i3;
        if (b1 >= g.n1) b1 -= g.n1;
        if (b2 >= g.n2) b2 -= g.n2;
        if (b3 >= g.n3) b3 -= g.n3;
        return grid_index(g, b1, b2, b3);
    }
};

// Gamma entries of every window k-point: n_window(k) times the sum of n_window(k+q) over its
// pairs.  One block per k-point.
__global__ void __launch_bounds__(kIbThreads) k_ib_entries(IbGrid g, const int *__restrict__ kpts,
                                                           const unsigned *__restrict__ pt,
                                                           const int64_t *__restrict__ kp_pairs,
                                                           const int *__restrict__ pairs, int64_t *__restrict__ n_ent) {
    __shared__ unsigned long long tot;
    const int kp = blockIdx.x, ik = kpts[kp];
    g.at(ik);
    if (threadIdx.x == 0) tot = 0;
    __syncthreads();
    unsigned n = 0;
    for (int64_t p = kp_pairs[kp] + threadIdx.x; p < kp_pairs[kp + 1]; p += kIbThreads) n += pt[g.kq(pairs[p])] & 31u;
    n = __reduce_add_sync(0xffffffffu, n);
    if ((threadIdx.x & 31) == 0 && n) atomicAdd(&tot, (unsigned long long)n);
    __syncthreads();
    if (threadIdx.x == 0) n_ent[kp] = (int64_t)tot * (pt[ik] & 31u);
}

// Block offsets of the pairs, relative to their k-point's first entry, and the column words of the
// entries: entry ent[kp] + goff[p] + n nw + j of pair p = (k, q) gets ((s + j) << 5) | n, s the
// first window state of k+q, j its band, n the band of k.  One block per k-point; a block scan
// per 256 pairs, in pair order.
__global__ void __launch_bounds__(kIbThreads) k_ib_index(IbGrid g, const int *__restrict__ kpts,
                                                         const unsigned *__restrict__ pt,
                                                         const int64_t *__restrict__ kp_pairs,
                                                         const int *__restrict__ pairs, const int64_t *__restrict__ ent,
                                                         uint32_t *__restrict__ goff, unsigned *__restrict__ col) {
    __shared__ unsigned sm[2][kIbWarps];
    const int kp = blockIdx.x, ik = kpts[kp];
    g.at(ik);
    const unsigned nsel = pt[ik] & 31u;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int64_t p1 = kp_pairs[kp + 1];
    unsigned *c0 = col + ent[kp];
    unsigned base = 0;
    int buf = 0;
    for (int64_t p0 = kp_pairs[kp]; p0 < p1; p0 += kIbThreads, buf ^= 1) {
        const int64_t p = p0 + threadIdx.x;
        const unsigned w = p < p1 ? pt[g.kq(pairs[p])] : 0u;
        const unsigned nw = w & 31u, size = nsel * nw;
        unsigned x = size;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) sm[buf][wid] = x;
        __syncthreads();                          // two buffers: one barrier per step
        unsigned before = base, tot = 0;
#pragma unroll
        for (int v = 0; v < kIbWarps; ++v) {
            const unsigned y = sm[buf][v];
            if (v < wid) before += y;
            tot += y;
        }
        const unsigned off = before + x - size;
        base += tot;
        if (p < p1) {
            goff[p] = off;
            for (unsigned n = 0; n < nsel; ++n)
                for (unsigned j = 0; j < nw; ++j) c0[off + n * nw + j] = (((w >> 5) + j) << 5) | n;
        }
    }
}

// F0 = v tau (tau = 1 / (1/tau), 0 where 1/tau = 0); F = F0
__global__ void k_ib_f0(int64_t ns, int W, const int *__restrict__ st_k, const int *__restrict__ st_n,
                        const double *__restrict__ inv_tau, const double *__restrict__ vel,
                        double *__restrict__ F0, double *__restrict__ F, float4 *__restrict__ F32) {
    const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= ns) return;
    const double r = inv_tau[s];
    const double tau = r > 0 ? 1.0 / r : 0.0;
    const int64_t idx = (int64_t)st_k[s] * W + st_n[s];
    float4 f32 = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int a = 0; a < 3; ++a) {
        const double f = vel[idx * 3 + a] * tau;
        F0[s * 3 + a] = f;
        F[s * 3 + a] = f;
        reinterpret_cast<float *>(&f32)[a] = (float)f;
    }
    if (F32) F32[s] = f32;
}

template <typename GT>
struct StepArgs {
    const int *kpts, *win_n;
    const int64_t *kp_state;
    const int64_t *ent;                   // first Gamma entry of each window k-point
    const unsigned *col;                  // per entry ((final state) << 5) | band of k
    const GT *gam;
    const double *inv_tau, *F0, *Fin;
    double *Fout;
    const float4 *Fin32;                  // FP32 copy of Fin (split paths), w unused
    float4 *Fout32;
    double pref;                          // 2 pi / (hbar N_q sqrt(pi) eta), s^-1 per eV^2
    unsigned long long *red;              // [2] max |dF|, max |F| of this step as bit patterns
    const unsigned long long *red_prev;   // the same of the step before, or nullptr
    double tol;
};

// The stop rule of the iteration; with it met the steps queued behind do nothing.
__host__ __device__ inline bool ib_done(double dmax, double fmax_, double tol) { return dmax <= tol * fmax_; }

// Accumulation type of the lane and warp sums: FP64 with FP64 Gamma; FP32 with FP32 Gamma
// (GB300 issues FP64 at 1/64 of the FP32 rate, so FP64 sums would bind the split paths on
// the FP64 pipe).  The sum over warps is FP64.
template <typename GT> struct Acc { using T = double; };
template <> struct Acc<float> { using T = float; };

__device__ __forceinline__ void load_F(const StepArgs<double> &a, int64_t s, double &x, double &y, double &z) {
    const double *f = a.Fin + s * 3;
    x = __ldg(f);
    y = __ldg(f + 1);
    z = __ldg(f + 2);
}
__device__ __forceinline__ void load_F(const StepArgs<float> &a, int64_t s, float &x, float &y, float &z) {
    const float4 f = __ldg(a.Fin32 + s);
    x = f.x;
    y = f.y;
    z = f.z;
}

// The warp's entries [e0, e1) for the bands b0 .. b0+NBX-1 of the k-point: y[n] += Gamma_e F_s
// for every entry e whose column word holds state s and band b0 + n.  Lane l takes entries
// e0 + l, e0 + l + 32, ...; kIbUnroll of them have their column, value and F loads issued
// before their multiplies.  ALL: every entry's band lies in the group (one group covers the
// window); otherwise an entry of another group adds zero products.
template <typename GT, int NB, int NBX, bool ALL>
__device__ __forceinline__ void step_entries(const StepArgs<GT> &a, int b0, int64_t e0, int64_t e1, int lane,
                                             typename Acc<GT>::T (&y)[NB][3]) {
    using AT = typename Acc<GT>::T;
    for (int64_t eb = e0 + lane; eb < e1; eb += 32 * kIbUnroll) {
        unsigned cw[kIbUnroll];
        AT g[kIbUnroll], fx[kIbUnroll], fy[kIbUnroll], fz[kIbUnroll];
#pragma unroll
        for (int u = 0; u < kIbUnroll; ++u) {
            const int64_t e = eb + 32 * u;
            cw[u] = e < e1 ? __ldg(a.col + e) : 0u;
            g[u] = e < e1 ? (AT)__ldg(a.gam + e) : AT(0);
        }
#pragma unroll
        for (int u = 0; u < kIbUnroll; ++u) load_F(a, (int64_t)(cw[u] >> 5), fx[u], fy[u], fz[u]);
#pragma unroll
        for (int u = 0; u < kIbUnroll; ++u) {
            if constexpr (NBX == 1 && ALL) {
                y[0][0] = fma(g[u], fx[u], y[0][0]);
                y[0][1] = fma(g[u], fy[u], y[0][1]);
                y[0][2] = fma(g[u], fz[u], y[0][2]);
            } else {
                const int n = (int)(cw[u] & 31u) - b0;
#pragma unroll
                for (int b = 0; b < NBX; ++b) {
                    const AT gb = n == b ? g[u] : AT(0);
                    y[b][0] = fma(gb, fx[u], y[b][0]);
                    y[b][1] = fma(gb, fy[u], y[b][1]);
                    y[b][2] = fma(gb, fz[u], y[b][2]);
                }
            }
        }
    }
}

template <typename GT, int NB, int NBX>
__device__ __forceinline__ void step_group(const StepArgs<GT> &a, bool all, int b0, int64_t e0, int64_t e1, int lane,
                                           typename Acc<GT>::T (&y)[NB][3]) {
    if (all) step_entries<GT, NB, NBX, true>(a, b0, e0, e1, lane, y);
    else step_entries<GT, NB, NBX, false>(a, b0, e0, e1, lane, y);
}

// One block per window k-point; its entries split into eight contiguous warp ranges.  The
// k-point's bands are taken in groups of NB (the smallest of 1, 2, 4, 8 covering the crystal's
// bands; wider windows loop over groups).  Lanes reduce by a butterfly in the accumulation
// type, warps in index order in FP64, so the result does not depend on scheduling.  Entry 0 of
// an unused column word (col 0, value 0) adds exactly zero.
template <typename GT, int NB>
__global__ void __launch_bounds__(kIbThreads, NB <= 4 ? 4 : 2) k_ib_step(StepArgs<GT> a) {
    using AT = typename Acc<GT>::T;
    __shared__ AT part[kIbWarps][NB][3];
    if (a.red_prev) {
        // a step that met the stop rule marks the next one's maxima with NaN patterns, and so on
        const unsigned long long d = a.red_prev[0], f = a.red_prev[1];
        if (d == ~0ull || ib_done(__longlong_as_double((long long)d), __longlong_as_double((long long)f), a.tol)) {
            if (threadIdx.x == 0) a.red[0] = ~0ull;
            return;
        }
    }
    const int kp = blockIdx.x;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int ik = a.kpts[kp];
    const int nsel = a.win_n[ik];
    const int64_t s0 = a.kp_state[kp];
    const int64_t q0 = a.ent[kp], ne = a.ent[kp + 1] - q0;
    const int64_t e0 = q0 + ne * wid / kIbWarps, e1 = q0 + ne * (wid + 1) / kIbWarps;
    double dmax = 0, fmax_ = 0;
    for (int b0 = 0; b0 < nsel; b0 += NB) {
        const int nb = min(NB, nsel - b0);
        AT y[NB][3];
#pragma unroll
        for (int n = 0; n < NB; ++n) y[n][0] = y[n][1] = y[n][2] = 0;
        // exact band count of this group (uniform over the block)
        const bool all = nsel <= NB;
        switch (nb) {
        case 1: step_group<GT, NB, 1>(a, all, b0, e0, e1, lane, y); break;
        case 2: if constexpr (NB >= 2) step_group<GT, NB, 2>(a, all, b0, e0, e1, lane, y); break;
        case 3: if constexpr (NB >= 3) step_group<GT, NB, 3>(a, all, b0, e0, e1, lane, y); break;
        case 4: if constexpr (NB >= 4) step_group<GT, NB, 4>(a, all, b0, e0, e1, lane, y); break;
        default: if constexpr (NB > 4) step_group<GT, NB, NB>(a, all, b0, e0, e1, lane, y); break;
        }
#pragma unroll
        for (int n = 0; n < NB; ++n) {
            if (n >= nb) break;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                AT v = y[n][c];
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
                if (lane == 0) part[wid][n][c] = v;
            }
        }
        __syncthreads();
        if (threadIdx.x < nb * 3) {
            const int n = threadIdx.x / 3, c = threadIdx.x % 3;
            double sum = 0;
#pragma unroll
            for (int w = 0; w < kIbWarps; ++w) sum += (double)part[w][n][c];
            const int64_t s = s0 + b0 + n;
            const double r = a.inv_tau[s];
            const double tau = r > 0 ? 1.0 / r : 0.0;
            const double f = a.F0[s * 3 + c] + tau * (a.pref * sum);
            a.Fout[s * 3 + c] = f;
            if (a.Fout32) reinterpret_cast<float *>(a.Fout32 + s)[c] = (float)f;
            dmax = fmax(dmax, fabs(f - a.Fin[s * 3 + c]));
            fmax_ = fmax(fmax_, fabs(f));
        }
        __syncthreads();
    }
    // max is order independent: the bit patterns of non-negative doubles order like the values
    if (threadIdx.x < 3 * NB && (dmax > 0 || fmax_ > 0)) {
        atomicMax(&a.red[0], (unsigned long long)__double_as_longlong(dmax));
        atomicMax(&a.red[1], (unsigned long long)__double_as_longlong(fmax_));
    }
}

template <typename GT>
void launch_step(epwi_ctx *c, const double *Fin, double *Fout, const float4 *Fin32, float4 *Fout32,
                 unsigned long long *red, const unsigned long long *red_prev, double tol) {
    StepArgs<GT> a;
    a.kpts = c->kpts.as<int>();
    a.win_n = c->win_n.as<int>();
    a.kp_state = c->kp_state.as<int64_t>();
    a.ent = c->ib_ent.as<int64_t>();
    a.col = c->ib_col.as<unsigned>();
    a.gam = c->ib_gam.as<GT>();
    a.inv_tau = c->inv_tau.as<double>();
    a.F0 = c->ib_F0.as<double>();
    a.Fin = Fin;
    a.Fout = Fout;
    a.Fin32 = Fin32;
    a.Fout32 = Fout32;
    a.pref = 2.0 * epc::kPi / epc::kHbarEVs / (double)c->nk / (sqrt(epc::kPi) * c->eta);
    a.red = red;
    a.red_prev = red_prev;
    a.tol = tol;
    // band group: the smallest of 1, 2, 4, 8 covering the bands (wider windows loop)
    const unsigned grid = (unsigned)c->nkp;
    if (c->nw <= 1) k_ib_step<GT, 1><<<grid, kIbThreads, 0, c->stream>>>(a);
    else if (c->nw <= 2) k_ib_step<GT, 2><<<grid, kIbThreads, 0, c->stream>>>(a);
    else if (c->nw <= 4) k_ib_step<GT, 4><<<grid, kIbThreads, 0, c->stream>>>(a);
    else k_ib_step<GT, kIbMaxBands><<<grid, kIbThreads, 0, c->stream>>>(a);
    EPWI_CHECK_LAUNCH();
}

}  // namespace

// Pair list, Gamma layout and storage for the window of the current call; the caller then
// runs the interpolation over the returned work set (which also fills inv_tau).
void ibte_prepare(epwi_ctx *c, WorkSet &ws) {
    const int64_t nkp = c->nkp, npairs = c->npairs;
    const bool fp64 = c->opt.precision == EPWI_FP64;
    c->ib_pairs.ensure(sizeof(int) * (npairs + 1));
    // the sum-factorised kernels find a pair's place in the list by the runs' first pairs
    int *runs = nullptr;
    if (c->opt.precision == EPWI_FP32 || (fp64 && sf64_ok(c))) {
        c->runs.ensure(sizeof(int) * (nkp * run_stride(make_grid_info(c)) + 1));
        runs = c->runs.as<int>();
    }
    sieve_fill_chunk(c, 0, nkp, c->ib_pairs.as<int>(), runs);
    ws.runs_dev = runs;
    EPWI_REQUIRE(c->nstates < (int64_t(1) << 27), EPWI_EUNSUPPORTED, "iterative BTE needs fewer than 2^27 states");
    c->ib_pt.ensure(sizeof(unsigned) * c->nk);
    EPWI_CUDA(cudaMemsetAsync(c->ib_pt.p, 0, sizeof(unsigned) * c->nk, c->stream));
    c->ib_goff.ensure(sizeof(uint32_t) * (npairs + 1));
    c->ib_ent.ensure(sizeof(int64_t) * (nkp + 1));
    c->counts.ensure(sizeof(int64_t) * (nkp + 1));
    IbGrid g;
    g.g = make_grid_info(c);
    g.fplane = make_fdiv((uint32_t)(g.g.n2 * g.g.n3));
    g.fn3 = make_fdiv((uint32_t)g.g.n3);
    g.k1 = g.k2 = g.k3 = 0;
    if (nkp > 0) {
        k_ib_points<<<(unsigned)((nkp + 255) / 256), 256, 0, c->stream>>>(nkp, c->kpts.as<int>(),
                                                                        c->kp_state.as<int64_t>(), c->ib_pt.as<unsigned>());
        EPWI_CHECK_LAUNCH();
        k_ib_entries<<<(unsigned)nkp, kIbThreads, 0, c->stream>>>(g, c->kpts.as<int>(), c->ib_pt.as<unsigned>(),
                                                                 c->kp_pairs.as<int64_t>(), c->ib_pairs.as<int>(),
                                                                 c->counts.as<int64_t>());
        EPWI_CHECK_LAUNCH();
    }
    scan_exclusive_i64(c, c->counts.as<int64_t>(), c->ib_ent.as<int64_t>(), nkp, nullptr);
    std::vector<int64_t> h_ent(nkp + 1);
    EPWI_CUDA(cudaMemcpyAsync(h_ent.data(), c->ib_ent.p, sizeof(int64_t) * (nkp + 1), cudaMemcpyDeviceToHost, c->stream));
    EPWI_CUDA(cudaStreamSynchronize(c->stream));
    const int64_t nent = h_ent[nkp];
    for (int64_t p = 0; p < nkp; ++p)
        EPWI_REQUIRE(h_ent[p + 1] - h_ent[p] < (int64_t(1) << 32), EPWI_EUNSUPPORTED,
                     "iterative BTE: more than 2^32 couplings of one k-point");
    c->ib_col.ensure(sizeof(unsigned) * (nent + 1));
    if (nkp > 0) {
        k_ib_index<<<(unsigned)nkp, kIbThreads, 0, c->stream>>>(
            g, c->kpts.as<int>(), c->ib_pt.as<unsigned>(), c->kp_pairs.as<int64_t>(), c->ib_pairs.as<int>(),
            c->ib_ent.as<int64_t>(), c->ib_goff.as<uint32_t>(), c->ib_col.as<unsigned>());
        EPWI_CHECK_LAUNCH();
    }
    const size_t eb = fp64 ? sizeof(double) : sizeof(float);
    const size_t gam_bytes = eb * (size_t)(nent + 1);
    c->ib_gam.ensure(gam_bytes);
    // the sum-factorised kernels write only the bands they do not skip (the others are exactly zero)
    if (c->opt.precision == EPWI_FP32 || fp64) EPWI_CUDA(cudaMemsetAsync(c->ib_gam.p, 0, gam_bytes, c->stream));
    c->ib_stats.n_entries = nent;
    c->ib_stats.entry_bytes = (int32_t)eb;
    ws.pairs_dev = c->ib_pairs.as<int>();
    ws.goff = c->ib_goff.as<uint32_t>();
    ws.gent = c->ib_ent.as<int64_t>();
    if (fp64) ws.gam64 = c->ib_gam.as<double>();
    else ws.gam32 = c->ib_gam.as<float>();
}

// Iterates from F0 = v tau; leaves the last iterate in c->ib_F.
void ibte_iterate(epwi_ctx *c, int max_iter, double tol) {
    const int64_t ns = c->nstates;
    const bool fp64 = c->opt.precision == EPWI_FP64;
    c->ib_F0.ensure(sizeof(double) * 3 * (ns + 1));
    c->ib_F.ensure(sizeof(double) * 3 * (ns + 1));
    c->ib_Fn.ensure(sizeof(double) * 3 * (ns + 1));
    if (!fp64) {
        c->ib_F32.ensure(sizeof(float4) * (ns + 1));
        c->ib_Fn32.ensure(sizeof(float4) * (ns + 1));
    }
    const int64_t nent = c->ib_stats.n_entries, nkp = c->nkp;
    // the pair list and the offsets served the capture; up to 4 GiB of them stay for the next call
    if (c->ib_goff.bytes + c->ib_pairs.bytes > (size_t(4) << 30)) {
        EPWI_CUDA(cudaStreamSynchronize(c->stream));
        c->ib_goff.release();
        c->ib_pairs.release();
    }
    if (ns > 0) {
        k_ib_f0<<<(unsigned)((ns + 255) / 256), 256, 0, c->stream>>>(
            ns, c->nw, c->st_k.as<int>(), c->st_n.as<int>(), c->inv_tau.as<double>(), c->vel.as<double>(),
            c->ib_F0.as<double>(), c->ib_F.as<double>(), fp64 ? nullptr : c->ib_F32.as<float4>());
        EPWI_CHECK_LAUNCH();
    }
    // Steps are queued kQueue at a time; each looks at the maxima of the one before and does nothing
    // once the stop rule is met, so the host reads the maxima only once per kQueue steps.
    constexpr int kQueue = 8;
    c->ib_red.ensure(sizeof(unsigned long long) * 2 * (kQueue + 1));
    unsigned long long *red = c->ib_red.as<unsigned long long>();   // maxima of step i in slot i + 1
    cudaEvent_t e0, e1;
    EPWI_CUDA(cudaEventCreate(&e0));
    EPWI_CUDA(cudaEventCreate(&e1));
    auto cleanup = [&] {
        cudaEventDestroy(e0);
        cudaEventDestroy(e1);
    };
    int it = 0;
    double change = 0, ms_steps = 0;
    try {
        bool done = false;
        while (!done && it < max_iter && nkp > 0) {
            const int n = std::min(kQueue, max_iter - it);
            EPWI_CUDA(cudaMemsetAsync(red, 0, sizeof(unsigned long long) * 2 * (kQueue + 1), c->stream));
            EPWI_CUDA(cudaEventRecord(e0, c->stream));
            double *F[2] = {c->ib_F.as<double>(), c->ib_Fn.as<double>()};
            float4 *F32[2] = {c->ib_F32.as<float4>(), c->ib_Fn32.as<float4>()};
            for (int i = 0; i < n; ++i) {
                unsigned long long *r = red + 2 * (i + 1), *rp = i ? red + 2 * i : nullptr;
                if (fp64) launch_step<double>(c, F[i & 1], F[~i & 1], nullptr, nullptr, r, rp, tol);
                else launch_step<float>(c, F[i & 1], F[~i & 1], F32[i & 1], F32[~i & 1], r, rp, tol);
            }
            EPWI_CUDA(cudaEventRecord(e1, c->stream));
            unsigned long long h[2 * (kQueue + 1)];
            EPWI_CUDA(cudaMemcpyAsync(h, red, sizeof(h), cudaMemcpyDeviceToHost, c->stream));
            EPWI_CUDA(cudaStreamSynchronize(c->stream));
            float ms = 0;
            EPWI_CUDA(cudaEventElapsedTime(&ms, e0, e1));
            ms_steps += ms;
            int ran = 0;                                  // steps of this queue that did their work
            for (int i = 0; i < n && !done; ++i) {
                double dmax, fmax_;
                std::memcpy(&dmax, &h[2 * (i + 1)], sizeof(double));
                std::memcpy(&fmax_, &h[2 * (i + 1) + 1], sizeof(double));
                EPWI_REQUIRE(std::isfinite(dmax) && std::isfinite(fmax_), EPWI_ENUMERIC,
                             "non-finite mean free path in the iteration");
                ++ran;
                change = fmax_ > 0 ? dmax / fmax_ : 0.0;
                done = ib_done(dmax, fmax_, tol);
            }
            it += ran;
            if (ran & 1) {                                // the newest iterate is in Fn
                std::swap(c->ib_F, c->ib_Fn);
                std::swap(c->ib_F32, c->ib_Fn32);
            }
        }
    } catch (...) {
        cleanup();
        throw;
    }
    cleanup();
    c->ib_stats.iters = it;
    c->ib_stats.change = change;
    c->ib_stats.ms_step = it > 0 ? ms_steps / it : 0.0;
    // one step reads the column words and Gamma once, F0, 1/tau and F at the states, writes F
    c->ib_stats.index_bytes = 4 * nent + 8 * (nkp + 1);
    c->ib_stats.bytes_per_step = (double)c->ib_stats.index_bytes +
                                 (double)c->ib_stats.entry_bytes * (double)c->ib_stats.n_entries +
                                 8.0 * (double)ns * (3 + 1 + 3 + 3);
}
