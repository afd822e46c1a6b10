// Sum-factorised Rp->q stage in FP64 (precision EPWI_FP64, sieved rates), fused with the
// rotations and the delta sum of Eq. 10: the same reordering of the R_p sum as the fp32 mode
// (scatter_sf.cu: +-R recombination of the bounding cube's axes, Y per plane block, U per run,
// the last axis per pair), every value and sum in FP64.  Results differ from the direct sum of
// k_scatter_fp64 by the order of summation only.
//
// The FP64 units bind (2 FMA per SM and clock): per (pair, band) the direct sum takes
// 4 n_Rp N_m W FMA (6000 for 5^3 and W = 4), this one 2 (D - 1) N_m W for the last axis (96), the
// rotations of the bands within reach (84 each), about 55 for the pair's share of U, and two
// exponentials per mode inside the Gaussian's support.  Measured on one GB300, Al-like 20^3 (6.6 M
// pairs): 75 ms with the direct sum, 10.6 ms here.  Per-pair index arithmetic and gathers run
// in the shadow of the FP64 pipe, so the kernel keeps the plain layouts of the FP64 tables.
#include <algorithm>

#include "epwi_internal.cuh"
#include "scatter.cuh"
#include "scatter_sf.cuh"
#include "sieve.cuh"

namespace {

struct Sf64Args {
    GridInfo g;
    int nplane;                     // N2 N3
    FDiv fplane, fjq;
    int jq, njg, pbmax;
    const double2 *ph64;
    const double2 *ghat;            // [state - s_base][D^3 forms][N_m][W]
    const int *kpts, *win_lo, *win_n;
    const int64_t *kp_state;
    int64_t s_base;
    const int64_t *kp_pairs;        // chunk-local pair offsets, minus p_off
    int64_t p_off;
    const int *pairs;
    const double2 *V, *u;           // [k][i][m], [q][mu][nu]
    const double *eps, *hw, *focc, *nocc;
    const float *hwmax32;
    double omega_min, eta, ceta;
    double pref;                    // 2 pi / (hbar N_q sqrt(pi) eta)
    double *inv_tau;
    int nkp;
    double *gam;                    // Gamma capture or nullptr (see scatter_sf.cu)
    const uint32_t *goff;
    const int64_t *gent;
};

// One CTA per (k-point, band): blockIdx.x runs over the chunk's states; the k-point is found in
// kp_state.  Layout and runs as in k_scatter_sf.
template <int W, int NM, int RC, bool GAM>
__global__ void __launch_bounds__(kSfThreads) k_scatter_sf64(Sf64Args a) {
    constexpr int D = 2 * RC + 1;
    constexpr int NF = D - 1;
    constexpr int X = NM * W;
    extern __shared__ __align__(16) double2 sm64[];
    const int N1 = a.g.n1, N2 = a.g.n2, N3 = a.g.n3, L = a.g.L;
    const int JQ = a.jq, NJG = a.njg;
    const SfSmem lay = sf_smem_layout(D, X, JQ, N1, N2, N3, NJG, a.pbmax, sizeof(double));
    double2 *Y = sm64;                           // [D f1][D f3][JQ][X]
    double *CS = reinterpret_cast<double *>(Y + lay.y + lay.u);   // [N1 + N2 + N3][NF]
    int *cq = reinterpret_cast<int *>(CS + lay.cs);
    int *ss = cq + kSieveBlock;
    int *se = ss + N1 * NJG;
    int *gl = se + N1 * NJG;
    int *pbs = gl + N1;
    int *nglist = pbs + a.pbmax + 1;
    __shared__ double wsum[kSfWarps];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    double2 *Uw = Y + lay.y + (size_t)wid * D * JQ * X;
    const int64_t s = a.s_base + blockIdx.x;     // global state
    // last k-point whose first state is <= s (every listed k-point has at least one state)
    const int kp = (int)lower_bound(0, a.nkp, s + 1, [&](int64_t p) { return a.kp_state[p + 1]; });
    const int n = (int)(s - a.kp_state[kp]);
    const int ik = a.kpts[kp];
    const int lo = a.win_lo[ik];
    const double2 *gs = a.ghat + (size_t)blockIdx.x * D * D * D * X;
    for (int e = tid; e < (N1 + N2 + N3) * RC; e += kSfThreads) {
        const int R = e % RC + 1, x = e / RC;
        int xx, st;
        if (x < N1) { xx = x; st = a.g.s1; }
        else if (x < N1 + N2) { xx = x - N1; st = a.g.s2; }
        else { xx = x - N1 - N2; st = a.g.s3; }
        const double2 v = a.ph64[(int)(((int64_t)xx * st % L) * R % L)];
        CS[x * NF + 2 * (R - 1)] = v.x;
        CS[x * NF + 2 * (R - 1) + 1] = v.y;
    }
    const double *CS1 = CS, *CS2 = CS + N1 * NF, *CS3 = CS + (N1 + N2) * NF;
    const int nplane = a.nplane;
    const int pb_n = (nplane + kSieveBlock - 1) / kSieveBlock;
    const int64_t P0 = a.kp_pairs[kp] - a.p_off, P1 = a.kp_pairs[kp + 1] - a.p_off;
    const int *pl = a.pairs + P0;
    const int np = (int)(P1 - P0);
    for (int pb = tid; pb <= pb_n; pb += kSfThreads)
        pbs[pb] = (int)lower_bound(0, np, pb, [&](int64_t p) {
            const int q = pl[p];
            return (int64_t)((q - fdiv(q, a.fplane) * nplane) / kSieveBlock);
        });
    int k1, k2, k3;
    grid_coords(a.g, ik, k1, k2, k3);
    const double en = a.eps[(int64_t)ik * W + lo + n];
    const double ieta = 1.0 / a.eta;
    double acc = 0;                              // this lane's pairs
    __syncthreads();
    for (int pb = 0; pb < pb_n; ++pb) {
        const int seg0 = pbs[pb], nseg = pbs[pb + 1] - seg0;
        if (nseg == 0) continue;
        const int *pp = pl + seg0;
        const int c_lo = pb * kSieveBlock, c_hi = min(nplane, c_lo + kSieveBlock) - 1;
        const int q2lo = c_lo / N3, nq2 = c_hi / N3 - q2lo + 1;
        const int njg = (nq2 + JQ - 1) / JQ;
        for (int t = tid; t < kSieveBlock; t += kSfThreads) {
            const int c = c_lo + t, q2 = c / N3;
            cq[t] = ((q2 - q2lo) << 16) | (c - q2 * N3);
        }
        for (int t = tid; t < N1 * NJG; t += kSfThreads) ss[t] = -1;
        __syncthreads();
        auto keyof = [&](int t) -> int {
            const int q = pp[t];
            const int q1 = fdiv(q, a.fplane);
            return q1 * NJG + fdiv(cq[q - q1 * nplane - c_lo] >> 16, a.fjq);
        };
        for (int t = tid; t < nseg; t += kSfThreads) {
            const int key = keyof(t);
            if (t == 0 || keyof(t - 1) != key) ss[key] = t;
            if (t == nseg - 1 || keyof(t + 1) != key) se[key] = t + 1;
        }
        __syncthreads();
        for (int jg = 0; jg < njg; ++jg) {
            const int j0 = jg * JQ, jn = min(JQ, nq2 - j0);
            if (wid == 0) {
                int cnt = 0;
                for (int q0 = 0; q0 < N1; q0 += 32) {
                    const int q1 = q0 + lane;
                    const bool on = q1 < N1 && ss[q1 * NJG + jg] >= 0;
                    const unsigned b = __ballot_sync(0xffffffffu, on);
                    if (on) gl[cnt + __popc(b & ((1u << lane) - 1u))] = q1;
                    cnt += __popc(b);
                }
                if (lane == 0) *nglist = cnt;
            }
            const int per = jn * X;
            for (int e = tid; e < D * D * per; e += kSfThreads) {
                const int r13 = e / per, e2 = e - r13 * per;
                const int jj = e2 / X, col = e2 - jj * X;
                const int f3 = r13 % D, f1 = r13 / D;
                const double *c2 = CS2 + (q2lo + j0 + jj) * NF;
                const double2 *src = gs + ((f1 * D) * D + f3) * X + col;
                double2 v = __ldg(src);
#pragma unroll
                for (int f2 = 1; f2 < D; ++f2) {
                    const double2 w = __ldg(src + f2 * D * X);
                    v.x = fma(c2[f2 - 1], w.x, v.x);
                    v.y = fma(c2[f2 - 1], w.y, v.y);
                }
                Y[(r13 * JQ + jj) * X + col] = v;
            }
            __syncthreads();
            const int ng = *nglist;
            for (int r = wid; r < ng; r += kSfWarps) {
                const int q1 = gl[r];
                const int t0 = ss[q1 * NJG + jg], t1 = se[q1 * NJG + jg];
                double c1[NF];
#pragma unroll
                for (int f = 0; f < NF; ++f) c1[f] = CS1[q1 * NF + f];
                for (int f3 = 0; f3 < D; ++f3)
                    for (int e = lane; e < per; e += 32) {
                        const double2 *src = Y + (size_t)f3 * JQ * X + e;
                        double2 v = src[0];
#pragma unroll
                        for (int f1 = 1; f1 < D; ++f1) {
                            const double2 w = src[f1 * D * JQ * X];
                            v.x = fma(c1[f1 - 1], w.x, v.x);
                            v.y = fma(c1[f1 - 1], w.y, v.y);
                        }
                        Uw[(size_t)f3 * JQ * X + e] = v;
                    }
                __syncwarp();
                int b1 = k1 + q1;
                if (b1 >= N1) b1 -= N1;
                const int qbase = q1 * nplane + c_lo;
                for (int t = t0 + lane; t < t1; t += 32) {
                    const int q = pp[t];
                    const int jq = cq[q - qbase];
                    const int j = jq >> 16, q3 = jq & 0xffff;
                    int b2 = k2 + q2lo + j, b3 = k3 + q3;
                    if (b2 >= N2) b2 -= N2;
                    if (b3 >= N3) b3 -= N3;
                    const int64_t ikq = ((int64_t)b1 * N2 + b2) * N3 + b3;
                    // final bands within reach of a mode (a superset; the others add zero)
                    const double lim = (double)__ldg(a.hwmax32 + q) + a.ceta + 1e-6;
                    unsigned mask = 0;
#pragma unroll
                    for (int m = 0; m < W; ++m) mask |= (fabs(en - __ldg(a.eps + ikq * W + m)) <= lim ? 1u : 0u) << m;
                    if (!mask) continue;
                    const double2 *Ub = Uw + (j - j0) * X;
                    double c3[NF];
#pragma unroll
                    for (int f = 0; f < NF; ++f) c3[f] = CS3[q3 * NF + f];
                    int lokq = 0, nwkq = 0;
                    int64_t grow = 0;
                    if constexpr (GAM) {
                        lokq = __ldg(a.win_lo + ikq);
                        nwkq = __ldg(a.win_n + ikq);
                        grow = a.gent[kp] + a.goff[P0 + seg0 + t] + (int64_t)n * nwkq - lokq;
                    }
                    constexpr bool kPreG = X <= 12;   // G kept for all bands of the pair
                    auto column = [&](int x) {
                        double2 v = Ub[x];
#pragma unroll
                        for (int f = 1; f < D; ++f) {
                            const double2 w = Ub[f * JQ * X + x];
                            v.x = fma(c3[f - 1], w.x, v.x);
                            v.y = fma(c3[f - 1], w.y, v.y);
                        }
                        return v;
                    };
                    double2 Gp[kPreG ? X : 1];
                    if constexpr (kPreG) {
#pragma unroll
                        for (int x = 0; x < X; ++x) Gp[x] = column(x);
                    }
                    const double2 *uq = a.u + (int64_t)q * NM * NM;
                    while (mask) {
                        const int m = __ffs(mask) - 1;
                        mask &= mask - 1;
                        const double em = __ldg(a.eps + ikq * W + m), fm = __ldg(a.focc + ikq * W + m);
                        const double2 *vp = a.V + ikq * W * W + m;
                        double2 Vc[W], gv[NM];
#pragma unroll
                        for (int i = 0; i < W; ++i) Vc[i] = __ldg(vp + i * W);
#pragma unroll
                        for (int nu = 0; nu < NM; ++nu) gv[nu] = make_double2(0, 0);
#pragma unroll
                        for (int mu = 0; mu < NM; ++mu) {
                            double2 h = make_double2(0, 0);
#pragma unroll
                            for (int i = 0; i < W; ++i) {
                                double2 Gi;
                                if constexpr (kPreG) Gi = Gp[mu * W + i];
                                else Gi = column(mu * W + i);
                                h = cfmac(Vc[i], Gi, h);
                            }
#pragma unroll
                            for (int nu = 0; nu < NM; ++nu) gv[nu] = cfma(h, __ldg(uq + mu * NM + nu), gv[nu]);
                        }
                        double gm = 0;
#pragma unroll
                        for (int nu = 0; nu < NM; ++nu) {
                            const double w = __ldg(a.hw + (int64_t)q * NM + nu);
                            if (!(w >= a.omega_min)) continue;
                            const double x1 = (en + w) - em, x2 = (en - w) - em;
                            const bool in1 = fabs(x1) <= a.ceta, in2 = fabs(x2) <= a.ceta;
                            if (!(in1 || in2)) continue;
                            const double N = __ldg(a.nocc + (int64_t)q * NM + nu);
                            double term = 0;
                            if (in1) {
                                const double y = x1 * ieta;
                                term += (N + fm) * exp(-y * y);
                            }
                            if (in2) {
                                const double y = x2 * ieta;
                                term += (1.0 + N - fm) * exp(-y * y);
                            }
                            gm = fma(gv[nu].x * gv[nu].x + gv[nu].y * gv[nu].y, term, gm);
                        }
                        acc += gm;
                        if constexpr (GAM) {
                            if (m >= lokq && m < lokq + nwkq) a.gam[grow + m] = gm;
                        }
                    }
                }
                __syncwarp();                                // Uw is rewritten by the next run
            }
            __syncthreads();                                 // gl, nglist and Y are rewritten next
        }
    }
    // lanes by a fixed tree, warps in order: deterministic, independent of the chunking
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) wsum[wid] = acc;
    __syncthreads();
    if (tid == 0) {
        double t = 0;
        for (int w = 0; w < kSfWarps; ++w) t += wsum[w];
        a.inv_tau[s] = a.pref * t;
    }
}

template <int W, int NM, int RC>
void launch(epwi_ctx *c, const Sf64Args &a, int64_t nstates, size_t sm) {
    auto go = [&](auto kern) {
        EPWI_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
        kern<<<(unsigned)nstates, kSfThreads, sm, c->stream>>>(a);
        EPWI_CHECK_LAUNCH();
    };
    if (a.gam) go(k_scatter_sf64<W, NM, RC, true>);
    else go(k_scatter_sf64<W, NM, RC, false>);
}

}  // namespace

bool sf64_ok(const epwi_ctx *c) {
    const int W = c->nw, NM = c->nm, r = c->sf_r;
    if (!c->keep_g64 || c->rp_twice || c->h_rp_cube.empty() || !sf_shape_built(W, NM, r)) return false;
    if (c->nk >= (int64_t(1) << 31) || c->ng[0] * 2 > 4096 || c->ng[2] > 0xffff) return false;
    const SfPlan p = sf_plan(2 * r + 1, NM * W, sf_q2max(c->ng[1], c->ng[2]), c->ng[0], c->ng[1], c->ng[2], sizeof(double));
    return p.smem <= 200 * 1024 && (int64_t)c->ng[0] * p.njg <= 8192 && p.pbmax <= 8192;
}

size_t sf64_state_bytes(const epwi_ctx *c) { return 2 * sf_state_bytes(c); }

void sf64_scatter(epwi_ctx *c, const ScatterArgs &sa, int64_t nkp, const int64_t *kp_pairs_local, int64_t p_off) {
    const int W = c->nw, NM = c->nm, r = c->sf_r;
    const SfPlan plan = sf_plan(2 * r + 1, NM * W, sf_q2max(sa.g.n2, sa.g.n3), sa.g.n1, sa.g.n2, sa.g.n3, sizeof(double));
    Sf64Args a;
    a.g = sa.g;
    a.nplane = sa.g.n2 * sa.g.n3;
    a.fplane = make_fdiv((uint32_t)a.nplane);
    a.fjq = make_fdiv((uint32_t)plan.jq);
    a.jq = plan.jq;
    a.njg = plan.njg;
    a.pbmax = plan.pbmax;
    a.ph64 = sa.ph64;
    a.ghat = sa.ghat64;
    a.kpts = sa.kpts;
    a.win_lo = sa.win_lo;
    a.win_n = sa.win_n;
    a.kp_state = sa.kp_state;
    a.s_base = sa.s_base;
    a.kp_pairs = kp_pairs_local;
    a.p_off = p_off;
    a.pairs = sa.pairs;
    a.V = sa.V64;
    a.u = sa.u64;
    a.eps = sa.eps;
    a.hw = sa.hw;
    a.focc = sa.focc;
    a.nocc = sa.nocc;
    a.hwmax32 = c->hwmax32.as<float>();
    a.omega_min = sa.omega_min;
    a.eta = sa.eta;
    a.ceta = sa.ceta;
    a.pref = 2.0 * epc::kPi / epc::kHbarEVs / (double)c->nk / (sqrt(epc::kPi) * sa.eta);
    a.inv_tau = c->inv_tau.as<double>();
    a.nkp = (int)nkp;
    a.gam = sa.gam64;
    a.goff = sa.goff;
    a.gent = sa.gent;
    const int64_t ns = sa.nstates_chunk;
    if (ns <= 0) return;
    if (W == 4 && r == 1) launch<4, 3, 1>(c, a, ns, plan.smem);
    else if (W == 4 && r == 2) launch<4, 3, 2>(c, a, ns, plan.smem);
    else if (W == 4 && r == 3) launch<4, 3, 3>(c, a, ns, plan.smem);
    else if (W == 1 && r == 1) launch<1, 3, 1>(c, a, ns, plan.smem);
    else if (W == 1 && r == 2) launch<1, 3, 2>(c, a, ns, plan.smem);
    else if (r == 1) launch<8, 6, 1>(c, a, ns, plan.smem);
    else if (r == 2) launch<8, 6, 2>(c, a, ns, plan.smem);
    else launch<8, 6, 3>(c, a, ns, plan.smem);
}
