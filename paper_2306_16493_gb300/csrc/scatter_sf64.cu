// Sum-factorised Rp->q stage in FP64 (precision EPWI_FP64, sieved rates), fused with the
// rotations and the delta sum of Eq. 10: the same reordering of the R_p sum as the fp32 mode
// (scatter_sf.cu: +-R recombination of the bounding cube's axes, Y per plane block, U per run,
// the last axis per pair), every value and sum in FP64.  Results differ from the direct sum of
// k_scatter_fp64 by the order of summation only.
//
// The FP64 units bind (2 FMA per SM and clock): per (pair, band) the direct sum takes
// 4 n_Rp N_m W FMA (6000 for 5^3 and W = 4), this one 2 (D - 1) N_m W for the last axis (96), 84 for
// the rotations, a share of about 30 of U (the runs q1 and -q1 from one pass over Y), and up to two
// exponentials per mode (12 operations each from a 64-entry table).  As in the fp32 kernel the pairs
// of the two runs form one list, and bands beyond a pair's first are worked off together, so that
// nearly all lanes of an FP64 instruction carry work.  Index arithmetic, gathers and the FP32
// pre-test of the bands run in the shadow of the FP64 pipe, so the kernel keeps the plain layouts of
// the FP64 tables.  Two CTAs per SM (plane-block groups sized for that, sf_plan) keep the pipe busy
// across the barriers: with one, it was 73 % busy.  Measured on one GB300, Al-like 20^3 (6.6 M pairs):
// direct sum 75 ms; factorised with a run per warp pass, every band of a pair in its lane and CUDA's exp
// 10.6 ms; paired runs, band list and table exponential 9.1 ms; two CTAs and items from a counter 7.6 ms.
#include <algorithm>

#include "epwi_internal.cuh"
#include "scatter.cuh"
#include "scatter_sf.cuh"
#include "sieve.cuh"

namespace {

struct Sf64Args {
    GridInfo g;
    int nplane;                     // N2 N3
    FDiv fn3, fper;                 // fper: division by jq X
    int jq, njg, pbmax;
    const double *coef;             // [N1 + N2 + N3][D - 1] cos, sin of theta R (k_sf_coef)
    const double2 *ghat;            // [state - s_base][D^3 forms][N_m][W]
    const int *kpts, *win_lo, *win_n;
    const int64_t *kp_state;
    int64_t s_base;
    const uint32_t *mask;           // sieve decisions of the chunk's k-points (rows of mask_words)
    int64_t mask_words;
    const double2 *V, *u;           // [k][i][m], [q][mu][nu]
    const double *eps, *hw, *focc, *nocc;
    const float *hwmax32, *eps32;
    float lim32;                    // c eta with the FP32 rounding of the pre-test
    double omega_min, eta, ceta;
    double pref;                    // 2 pi / (hbar N_q sqrt(pi) eta)
    double *inv_tau;
    int nkp;
    double *gam;                    // Gamma capture or nullptr (see scatter_sf.cu)
    const uint32_t *goff;
    const int64_t *gent;
    const int64_t *kp_pairs;        // with a capture: chunk-local pair offsets, minus p_off, and the
    int64_t p_off;                  // run tables (sieve.cuh)
    const int *runs;
    int64_t run_stride;
};

// e^x for -690 <= x <= 0 by Tang's table-driven method (ACM TOMS 15, 144 (1989)): x = n ln2 / 64 + r,
// e^x = 2^(n >> 6) T[n & 63] e^r with T[j] = 2^(j/64) and the Taylor polynomial of degree 5 (|r| <=
// 0.0055: remainder below 4e-17).
__device__ __forceinline__ double exp_neg(double x, const double *T) {
    if (x < -690.0) return exp(x);
    const double big = 6755399441055744.0;                 // 1.5 2^52: rounds to integer
    const double t = fma(x, 92.332482616893656768, big);   // 64 / ln 2
    const int n = __double2loint(t);
    const double nd = t - big;
    double r = fma(nd, -0x1.62e42fefap-7, x);              // ln2 / 64: 36 bits, then the rest
    r = fma(nd, -0x1.cf79abc9e3b3ap-46, r);
    double p = fma(r, 1.0 / 120.0, 1.0 / 24.0);
    p = fma(r, p, 1.0 / 6.0);
    p = fma(r, p, 0.5);
    p = fma(r, p, 1.0);
    const double tj = T[n & 63];
    const double v = fma(tj * r, p, tj);
    return __hiloint2double(__double2hiint(v) + (n >> 6) * (1 << 20), __double2loint(v));
}

// One CTA per (k-point, band): blockIdx.x runs over the chunk's states.  Groups, items and lists as
// in k_scatter_sf.
template <int W, int NM, int RC, bool GAM>
__global__ void __launch_bounds__(kSfThreads) k_scatter_sf64(Sf64Args a) {
    constexpr int D = 2 * RC + 1;
    constexpr int NF = D - 1;
    constexpr int X = NM * W;
    extern __shared__ __align__(16) double2 sm64[];
    const int N1 = a.g.n1, N2 = a.g.n2, N3 = a.g.n3;
    const int JQ = a.jq, NJG = a.njg;
    const SfSmem lay = sf_smem_layout(D, X, W, JQ, N1, N3, NJG, a.pbmax, sizeof(double));
    double2 *Y = sm64;                           // [D f1][D f3][JQ][X]
    double *CS3 = reinterpret_cast<double *>(Y + lay.y + lay.u);  // [N3][NF]: axis-3 coefficients
    const int nh = N1 / 2 + 1;
    double *rs = CS3 + lay.cs;                   // [nh]: sums of the current group's items
    int *lists = reinterpret_cast<int *>(rs + lay.rs);  // two item lists (list_items)
    uint32_t *flags = reinterpret_cast<uint32_t *>(lists + 2 * (nh + 2));
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    uint8_t *clist = reinterpret_cast<uint8_t *>(flags + lay.flags) + wid * kSieveBlock;
    uint16_t *left = reinterpret_cast<uint16_t *>(reinterpret_cast<uint8_t *>(flags + lay.flags) + kSfWarps * kSieveBlock) +
                     wid * 32 * W;
    __shared__ double T[64];
    const int ustride = D * JQ * X;
    double2 *Uw = Y + lay.y + (size_t)wid * 2 * ustride;
    const int64_t s = a.s_base + blockIdx.x;     // global state
    // last k-point whose first state is <= s (every listed k-point has at least one state)
    const int kp = (int)lower_bound(0, a.nkp, s + 1, [&](int64_t p) { return a.kp_state[p + 1]; });
    const int n = (int)(s - a.kp_state[kp]);
    const int ik = a.kpts[kp];
    const int lo = a.win_lo[ik];
    const double2 *gs = a.ghat + (size_t)blockIdx.x * D * D * D * X;
    if (tid < 64) T[tid] = exp2((double)tid / 64.0);
    const double *CS1 = a.coef, *CS2 = CS1 + N1 * NF;
    for (int e = tid; e < N3 * NF; e += kSfThreads) CS3[e] = CS2[N2 * NF + e];
    const int nplane = a.nplane;
    const uint32_t *mrow = a.mask + (int64_t)kp * a.mask_words;   // [pb][q1][8 words]
    const SfGroups groups{mrow, flags, a.fn3, N1, N3, nplane, JQ, NJG};
    mark_groups(groups, (int)lay.flags);
    int k1, k2, k3;
    grid_coords(a.g, ik, k1, k2, k3);
    const double en = a.eps[(int64_t)ik * W + lo + n];
    const float en32 = a.eps32[(int64_t)ik * W + lo + n];
    const double ieta = 1.0 / a.eta;
    double acc = 0;                              // warp 0: sums of the items lane, lane + 32, ...
    __syncthreads();
    int f = groups.next(-1), buf = 0;
    if (wid == 0 && f >= 0) list_items(groups.group(f), N1, lists);
    for (; f >= 0; buf ^= 1) {
        const SfGroup grp = groups.group(f);
        const int c_lo = grp.c_lo, q2lo = grp.q2lo, j0 = grp.j0, jn = grp.jn;
        int *gl = lists + buf * (nh + 2);
        const int fnext = groups.next(f);
        for (int e = tid; e < D * D * JQ * X; e += kSfThreads) {
            const int r13 = fdiv(e, a.fper), e2 = e - r13 * JQ * X;
            const int jj = e2 / X, col = e2 - jj * X;
            if (jj >= jn) continue;
            const int f1 = r13 / D, f3 = r13 - f1 * D;
            const double *c2 = CS2 + (q2lo + j0 + jj) * NF;
            const double2 *src = gs + ((f1 * D) * D + f3) * X + col;
            double2 v = __ldg(src);
#pragma unroll
            for (int f2 = 1; f2 < D; ++f2) {
                const double2 w = __ldg(src + f2 * D * X);
                v.x = fma(c2[f2 - 1], w.x, v.x);
                v.y = fma(c2[f2 - 1], w.y, v.y);
            }
            Y[e] = v;
        }
        __syncthreads();
        const int ng = gl[nh], per = jn * X;
        int r = 0;
        // items are taken from a counter; each writes its own sum, as in k_scatter_sf
        while (true) {
            if (lane == 0) r = atomicAdd(gl + nh + 1, 1);
            r = __shfl_sync(0xffffffffu, r, 0);
            if (r >= ng) break;
            const int q1 = gl[r];
            const int q1b = q1 == 0 || 2 * q1 == N1 ? q1 : N1 - q1;
            // lanes 0-7 and 8-15: the words of the two runs; na, nb: their pairs
            const int wx = lane & 7;
            uint32_t word = 0u;
            if (lane < 8 || (lane < 16 && q1b != q1)) word = __ldg(grp.mpb + (lane < 8 ? q1 : q1b) * 8 + wx);
            int skip = 0;                                    // pairs of the run in earlier groups (capture)
            if (NJG > 1) {
                if constexpr (GAM) skip = __popc(word & (grp.r0 > 32 * wx + 31 ? ~0u : grp.r0 > 32 * wx ? ~(~0u << (grp.r0 - 32 * wx)) : 0u));
                word &= grp.bits(wx);
            }
            int npc = __popc(word);
#pragma unroll
            for (int o = 1; o < 8; o <<= 1) {
                npc += __shfl_xor_sync(0xffffffffu, npc, o);
                if constexpr (GAM) skip += __shfl_xor_sync(0xffffffffu, skip, o);
            }
            const int na = __shfl_sync(0xffffffffu, npc, 0), nb = __shfl_sync(0xffffffffu, npc, 8);
            int t0 = 0, t0b = 0;                             // capture: list positions of the runs' pairs
            if constexpr (GAM) {
                const int *ru = a.runs + (int64_t)kp * a.run_stride + c_lo / kSieveBlock * N1;
                t0 = ru[q1] + __shfl_sync(0xffffffffu, skip, 0);
                t0b = ru[q1b] + __shfl_sync(0xffffffffu, skip, 8);
            }
            // U of the runs q1 and -q1 from one pass over Y: with E the even part (form 0 and
            // the cosine forms) and O the odd part (the sine forms), U(+-q1) = E +- O
            double c1[NF];
#pragma unroll
            for (int f = 0; f < NF; ++f) c1[f] = __ldg(CS1 + q1 * NF + f);
            for (int f3 = 0; f3 < D; ++f3)
                for (int e = lane; e < per; e += 32) {
                    const double2 *src = Y + (size_t)f3 * JQ * X + e;
                    double2 v = src[0], o = make_double2(0, 0);
#pragma unroll
                    for (int R = 1; R <= RC; ++R) {
                        const double2 w = src[(2 * R - 1) * D * JQ * X], z = src[2 * R * D * JQ * X];
                        v.x = fma(c1[2 * R - 2], w.x, v.x);
                        v.y = fma(c1[2 * R - 2], w.y, v.y);
                        o.x = fma(c1[2 * R - 1], z.x, o.x);
                        o.y = fma(c1[2 * R - 1], z.y, o.y);
                    }
                    double2 *dst = Uw + (size_t)f3 * JQ * X + e;
                    dst[0] = make_double2(v.x + o.x, v.y + o.y);
                    dst[ustride] = make_double2(v.x - o.x, v.y - o.y);
                }
            double rate = 0;
            int b1a = k1 + q1, b1b = k1 + q1b;
            if (b1a >= N1) b1a -= N1;
            if (b1b >= N1) b1b -= N1;
            const int parts = na + nb <= kSieveBlock ? 1 : 2;
            for (int part = 0; part < parts; ++part) {
                const int npa = part == 0 ? na : 0, npr = parts == 1 ? na + nb : part == 0 ? na : nb;
                __syncwarp();                                    // Uw is complete, clist is consumed
                {
                    int at = 0;
                    for (int x = part * 8; x < (parts == 1 || part == 1 ? 16 : 8); ++x) {
                        const uint32_t w = __shfl_sync(0xffffffffu, word, x);
                        if (w == 0u) continue;                   // uniform over the warp
                        if ((w >> lane) & 1u) clist[at + __popc(w & ((1u << lane) - 1u))] = (uint8_t)((x & 7) * 32 + lane);
                        at += __popc(w);
                    }
                }
                int base = 0, nleft = 0;
                while (true) {
                    __syncwarp();
                    const bool fresh = base < npr && nleft < 32;
                    if (!fresh && nleft == 0) break;
                    int tt, m = 0;
                    bool have;
                    if (fresh) {
                        tt = base + lane;
                        have = tt < npr;
                        base += 32;
                    } else {
                        const int take = min(nleft, 32);
                        nleft -= take;
                        have = lane < take;
                        const int e = have ? left[nleft + lane] : 0;
                        __syncwarp();                            // before the entries are rewritten
                        tt = e >> 3;
                        m = e & 7;
                    }
                    const bool second = tt >= npa;
                    const int c = have ? clist[tt] : 0;
                    const int q = (second ? q1b : q1) * nplane + c_lo + c;
                    const int q2 = fdiv(c_lo + c, a.fn3), q3 = c_lo + c - q2 * N3, j = q2 - q2lo;
                    int b2 = k2 + q2, b3 = k3 + q3;
                    if (b2 >= N2) b2 -= N2;
                    if (b3 >= N3) b3 -= N3;
                    const int64_t ikq = ((int64_t)(second ? b1b : b1a) * N2 + b2) * N3 + b3;
                    if (fresh) {
                        // final bands within reach of a mode (a superset, in FP32; the others add zero)
                        unsigned mask = 0;
                        if (have) {
                            const float lim = __ldg(a.hwmax32 + q) + a.lim32;
#pragma unroll
                            for (int mm = 0; mm < W; ++mm)
                                mask |= (fabsf(en32 - __ldg(a.eps32 + ikq * W + mm)) <= lim ? 1u : 0u) << mm;
                        }
                        have = mask != 0;
                        m = have ? __ffs(mask) - 1 : 0;
                        mask &= mask - 1;
                        unsigned more;
                        while ((more = __ballot_sync(0xffffffffu, have && mask)) != 0) {
                            if (have && mask) {
                                left[nleft + __popc(more & ((1u << lane) - 1u))] = (uint16_t)(tt << 3 | (__ffs(mask) - 1));
                                mask &= mask - 1;
                            }
                            nleft += __popc(more);
                        }
                        __syncwarp();
                    }
                    if (!have) continue;
                    const double2 *Ub = Uw + (second ? ustride : 0) + (j - j0) * X;
                    double c3[NF];
#pragma unroll
                    for (int f = 0; f < NF; ++f) c3[f] = CS3[q3 * NF + f];
                    const double em = __ldg(a.eps + ikq * W + m), fm = __ldg(a.focc + ikq * W + m);
                    const double2 *vp = a.V + ikq * W * W + m;
                    const double2 *uq = a.u + (int64_t)q * NM * NM;
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
                            double2 G = Ub[mu * W + i];
#pragma unroll
                            for (int f = 1; f < D; ++f) {
                                const double2 w = Ub[f * JQ * X + mu * W + i];
                                G.x = fma(c3[f - 1], w.x, G.x);
                                G.y = fma(c3[f - 1], w.y, G.y);
                            }
                            h = cfmac(Vc[i], G, h);
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
                        const double N = __ldg(a.nocc + (int64_t)q * NM + nu);
                        double term = 0;
                        if (fabs(x1) <= a.ceta) {
                            const double y = x1 * ieta;
                            term = (N + fm) * exp_neg(-y * y, T);
                        }
                        if (fabs(x2) <= a.ceta) {
                            const double y = x2 * ieta;
                            term = fma(1.0 + N - fm, exp_neg(-y * y, T), term);
                        }
                        gm = fma(gv[nu].x * gv[nu].x + gv[nu].y * gv[nu].y, term, gm);
                    }
                    rate += gm;
                    if constexpr (GAM) {
                        const int lokq = __ldg(a.win_lo + ikq), nwkq = __ldg(a.win_n + ikq);
                        const int t = second ? t0b + tt - npa : t0 + tt;    // the pair's place in the k-point's list
                        if (m >= lokq && m < lokq + nwkq)
                            a.gam[a.gent[kp] + a.goff[a.kp_pairs[kp] - a.p_off + t] + (int64_t)n * nwkq + (m - lokq)] = gm;
                    }
                }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) rate += __shfl_xor_sync(0xffffffffu, rate, o);
            if (lane == 0) rs[r] = rate;
            __syncwarp();                                // Uw is rewritten by the next item
        }
        // the first warp without an item lists the next group's
        if (r == ng && fnext >= 0) list_items(groups.group(fnext), N1, lists + (buf ^ 1) * (nh + 2));
        __syncthreads();                                 // the list, rs and Y are rewritten next
        if (wid == 0) {
            for (int x = lane; x < ng; x += 32) acc += rs[x];
            __syncwarp();                                // before rs is rewritten by this warp's items
        }
        f = fnext;
    }
    // lanes by a fixed tree: deterministic, independent of the chunking
    if (wid == 0) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (lane == 0) a.inv_tau[s] = a.pref * acc;
    }
}

template <int W, int NM, int RC>
void launch(epwi_ctx *c, const Sf64Args &a, int64_t nstates, size_t sm) {
    auto go = [&](auto kern) {
        allow_smem(kern);
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
    const SfPlan p = sf_plan(2 * r + 1, NM * W, W, sf_q2max(c->ng[1], c->ng[2]), c->ng[0], c->ng[1], c->ng[2], sizeof(double));
    return p.smem <= 200 * 1024 && (int64_t)c->ng[0] * p.njg <= 8192 && p.pbmax <= 8192;
}

size_t sf64_state_bytes(const epwi_ctx *c) { return 2 * sf_state_bytes(c); }

void sf64_scatter(epwi_ctx *c, const ScatterArgs &sa, int64_t nkp, const int64_t *kp_pairs_local, int64_t p_off) {
    const int W = c->nw, NM = c->nm, r = c->sf_r;
    const SfPlan plan = sf_plan(2 * r + 1, NM * W, W, sf_q2max(sa.g.n2, sa.g.n3), sa.g.n1, sa.g.n2, sa.g.n3, sizeof(double));
    Sf64Args a;
    a.g = sa.g;
    a.nplane = sa.g.n2 * sa.g.n3;
    a.fn3 = make_fdiv((uint32_t)sa.g.n3);
    a.fper = make_fdiv((uint32_t)(plan.jq * NM * W));
    a.mask = sa.mask;
    a.mask_words = sa.mask_words;
    a.runs = sa.runs;
    a.run_stride = run_stride(sa.g);
    a.eps32 = c->eps32.as<float>();
    // |e| <= E in FP32: each energy and their difference are off by less than 2^-24 (2 E + |x|)
    a.lim32 = (float)(sa.ceta + 1e-5 + 4e-7 * (2.0 * c->eabs_max + 1.0));
    a.jq = plan.jq;
    a.njg = plan.njg;
    a.pbmax = plan.pbmax;
    a.coef = c->sf_coef.as<double>();
    a.ghat = sa.ghat64;
    a.kpts = sa.kpts;
    a.win_lo = sa.win_lo;
    a.win_n = sa.win_n;
    a.kp_state = sa.kp_state;
    a.s_base = sa.s_base;
    a.kp_pairs = kp_pairs_local;
    a.p_off = p_off;
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
