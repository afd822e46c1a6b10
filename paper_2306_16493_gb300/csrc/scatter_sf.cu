// Sum-factorised Rp->q stage in FP32 (precision EPWI_FP32), fused with the rotations and the
// delta sum of Eq. 10.
//
// Any R_p set is embedded in its bounding cube [-r, r]^3 (vectors outside the set carry zero
// weight), so the phase of Eq. 16 factorises per axis: e^{iq.Rp} = e1(q1,R1) e2(q2,R2)
// e3(q3,R3), e_a(x, R) = e^{i theta R}, theta = 2 pi x / N_a.  Along each axis the values at
// +R and -R are recombined once, at setup, into
//     v'[0] = v[0],  v'[2R-1] = v[R] + v[-R],  v'[2R] = i (v[R] - v[-R])      (R = 1..r)
// so that sum_R e^{i theta R} v[R] = v'[0] + sum_R (cos(theta R) v'[2R-1] + sin(theta R) v'[2R]):
// every stage below is a contraction with REAL coefficients (2 FMAs per complex term instead
// of 4).  The recombination acts on the R_p index only, so it commutes with the Re->k sum and
// the U^dag(k) rotation and is applied to g(Re, Rp) itself (k_sf_transform).
//
// The sieve decides the pairs of a k-point in plane blocks pb of 256 consecutive (q2, q3)
// combinations, by q1 (8 mask words a run).  For the state (k, n) of one CTA:
//   Y[f1][f3][j]  = sum_f2 c2(q2_j)[f2] ghat'[f1][f2][f3]    per plane block and group of q2 values j
//   U[f3][j]      = sum_f1 c1(q1)[f1]  Y[f1][f3][j]           per run (plane block, q1, q2 group)
//   G             = sum_f3 c3(q3)[f3]  U[f3][j(q)]            per pair
// with ghat' = (g' P^el) U^dag(k) from the FP32 Re->k stage, every column (mu, i) at once.
// A warp takes the two runs q1 and N1 - q1 of a group: U = E +- O from one pass over Y, their mask
// words expanded to a list of combinations in shared memory, then 32 pairs at a time.  Per pair,
// the final bands m that have a mode within c eta of either energy shell count (others add
// exactly zero); a lane does its first one, further ones go to a list that is worked off 32 at a
// time.  Per band the modes mu are streamed: h = sum_i conj(V_im(k+q)) G[mu][i], g_nu += h u_mu,nu(q); then
// |g|^2 and the two delta terms, in FP32.  With a Gamma capture (iterative BTE) the CTA also writes
// its band's row of every pair's Gamma block (rows of bands out of range stay at the zero the
// buffer was cleared to), a pair's place in the list being its run's first plus its rank there.  Lane
// sums are FP32 within an item (the two runs), FP64 across items, added in a fixed order, so the
// result is deterministic and independent of k-point chunking.
//
// Bound by the instructions and gathers of the pairs (k_kq_table, k_q_table: tiles of 64 grid points, so
// that the 32 neighbouring points of a warp share cache lines).  Reading the mask directly needs no pair
// lists (4 bytes per pair written and read twice) and no search for the runs in them.  Measured on
// one GB300, Al-like 48^3 (1.26 G pairs), list fill and this kernel together: 57.1 ms with a run per
// warp pass, 50.7 ms with both runs from one pass and the runs' bounds from a table, 49.3 ms from the
// mask, 47.9 ms with packed multiply-adds (__ffma2_rn: two FP32 FMAs per issue slot) and a group's
// items listed while the group before is worked off; 20 x 27 x 45 (61 M pairs) 4.6, 3.4, 3.3 and 3.0 ms;
// Si-like 100^3 14.6 -> 13.4 ms by the last.  With the mode energies loaded ahead of the rotation 45.4
// (48^3), 2.8 (20 x 27 x 45) and 11.9 ms (Si-like).
#include <algorithm>

#include "epwi_internal.cuh"
#include "kstage.cuh"
#include "scatter.cuh"
#include "scatter_sf.cuh"
#include "sieve.cuh"

namespace {

// Re->k in FP32: ghat32[state][row] = sum_j [sum_Re w e^{ik.Re} g(Re)[row][j]] V_{j, lo+n}(k),
// row = (cube form, mu, i); one thread per row, KG k-points per block row.
template <int WT, int KG>
__global__ void __launch_bounds__(128) k_restage_f32(RestageArgs a, float2 *__restrict__ out) {
    constexpr int WM = WT ? WT : epc::kMaxW;
    const int W = WT ? WT : a.W;
    extern __shared__ float2 P32[];                 // [KG][nRe]
    const int kg0 = blockIdx.y * KG;
    for (int idx = threadIdx.x; idx < KG * a.nRe; idx += blockDim.x) {
        const int kk = idx / a.nRe, r = idx % a.nRe;
        float2 p = make_float2(0.f, 0.f);
        if (kg0 + kk < a.nkp) {
            int i1, i2, i3;
            grid_coords(a.g, a.kpts[kg0 + kk], i1, i2, i3);
            p = a.ph32[phase_index(i1 * a.g.s1 % a.g.L, i2 * a.g.s2 % a.g.L, i3 * a.g.s3 % a.g.L,
                                   a.Re[3 * r], a.Re[3 * r + 1], a.Re[3 * r + 2], a.g.L)];
        }
        P32[idx] = p;
    }
    __syncthreads();
    const int row = blockIdx.x * blockDim.x + threadIdx.x;
    if (row >= a.nrow) return;
    float2 acc[KG][WM];
    for (int kk = 0; kk < KG; ++kk)
        for (int j = 0; j < W; ++j) acc[kk][j] = make_float2(0.f, 0.f);
    const float2 *gw = a.gw32 + (size_t)row * W;
    for (int r = 0; r < a.nRe; ++r) {
        float2 gv[WM];
        for (int j = 0; j < W; ++j) gv[j] = gw[(size_t)r * a.nrow * W + j];
        for (int kk = 0; kk < KG; ++kk) {
            const float2 p = P32[kk * a.nRe + r];
            for (int j = 0; j < W; ++j) acc[kk][j] = cfmaf(p, gv[j], acc[kk][j]);
        }
    }
    for (int kk = 0; kk < KG; ++kk) {
        if (kg0 + kk >= a.nkp) break;
        const int ik = a.kpts[kg0 + kk];
        const int lo = a.win_lo[ik], ns = a.win_n[ik];
        const int64_t s0 = a.kp_state[kg0 + kk] - a.s_base;
        const float2 *Vk = a.V32 + (int64_t)ik * W * W;
        for (int np = 0; np < ns; ++np) {
            float2 o = make_float2(0.f, 0.f);
            for (int j = 0; j < W; ++j) o = cfmaf(acc[kk][j], Vk[j * W + lo + np], o);
            out[(s0 + np) * a.nrow + row] = o;
        }
    }
}

// The same Re->k stage with one thread per (row, j) and 32 k-points per thread: the phases of
// the block's 32 k-points are staged in shared memory in chunks of 32 R_e and read as
// broadcasts, g'[Re][row][j] is read once per 32 k-points (coalesced over (row, j)), and the
// contraction with V_{j,n}(k) is a shuffle reduction over the W lanes of a row.  Sums over R_e
// run in R_e order; the sum over j is a fixed tree.
template <int W>
__global__ void __launch_bounds__(256) k_restage_f32_kb(RestageArgs a, float2 *__restrict__ out) {
    constexpr int KB = 32, RCH = 32, RPB = 256 / W;   // k-points per block, R_e per chunk, rows per block
    __shared__ float2 Ps[RCH][KB];
    const int tid = threadIdx.x, j = tid % W;
    const int row = blockIdx.x * RPB + tid / W;
    const int k0 = blockIdx.y * KB;
    const bool live = row < a.nrow;
    float2 acc[KB];
#pragma unroll
    for (int x = 0; x < KB; ++x) acc[x] = make_float2(0.f, 0.f);
    for (int re0 = 0; re0 < a.nRe; re0 += RCH) {
        __syncthreads();                          // Ps of the previous chunk is consumed
        for (int e = tid; e < RCH * KB; e += 256) {
            const int rr = e / KB, kk = e % KB, re = re0 + rr;
            float2 p = make_float2(0.f, 0.f);
            if (k0 + kk < a.nkp && re < a.nRe) {
                int i1, i2, i3;
                grid_coords(a.g, a.kpts[k0 + kk], i1, i2, i3);
                p = a.ph32[phase_index(i1 * a.g.s1 % a.g.L, i2 * a.g.s2 % a.g.L, i3 * a.g.s3 % a.g.L,
                                       a.Re[3 * re], a.Re[3 * re + 1], a.Re[3 * re + 2], a.g.L)];
            }
            Ps[rr][kk] = p;
        }
        __syncthreads();
        const int nr = min(RCH, a.nRe - re0);
        if (live) {
            for (int rr = 0; rr < nr; ++rr) {
                const float2 gv = __ldg(a.gw32 + ((size_t)(re0 + rr) * a.nrow + row) * W + j);
#pragma unroll
                for (int x = 0; x < KB; x += 2) {
                    const float4 p2 = reinterpret_cast<const float4 *>(&Ps[rr][x])[0];
                    acc[x] = cfmaf(make_float2(p2.x, p2.y), gv, acc[x]);
                    acc[x + 1] = cfmaf(make_float2(p2.z, p2.w), gv, acc[x + 1]);
                }
            }
        }
    }
    // out[state][row] = sum_j acc[k][j] V_{j, lo+n}(k): lanes j of a row are adjacent
#pragma unroll
    for (int x = 0; x < KB; ++x) {
        const int kp = k0 + x;
        if (kp >= a.nkp) continue;               // uniform over the block
        const int ik = a.kpts[kp];
        const int lo = a.win_lo[ik], ns = a.win_n[ik];
        const int64_t s0 = a.kp_state[kp] - a.s_base;
        const float2 *Vk = a.V32 + (int64_t)ik * W * W;
        for (int np = 0; np < ns; ++np) {
            float2 o = cmulf(acc[x], Vk[j * W + lo + np]);
#pragma unroll
            for (int off = W / 2; off > 0; off >>= 1) {
                o.x += __shfl_xor_sync(0xffffffffu, o.x, off);
                o.y += __shfl_xor_sync(0xffffffffu, o.y, off);
            }
            if (live && j == 0) out[(s0 + np) * a.nrow + row] = o;
        }
    }
}

// The value of (state, row) in the fp32 mode's layout.
struct SfStore {
    float2 *out;
    int64_t nrow;
    __device__ __forceinline__ void operator()(int64_t s, int row, float2 v) const { out[s * nrow + row] = v; }
};

// g'(Re, f1 f2 f3) = (T x T x T) g(Re, cube): along each axis, form 0 is R = 0, form 2R-1 is
// v[R] + v[-R] and form 2R is i (v[R] - v[-R]).  cube: upload_rp_map (points without a vector have
// zero weight).  One thread per output element; FP64 sums, output in FP32
// or FP64.
template <class C2>
__global__ void k_sf_transform(int64_t n, int nRp, int Dc, int rc, int rowlen, const int *__restrict__ cube,
                               const double2 *__restrict__ g64, const float2 *__restrict__ g32,
                               C2 *__restrict__ out) {
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= n) return;
    const int e = (int)(idx % rowlen);              // (mu, i, j) within the (Re, form) block
    const int64_t t = idx / rowlen;
    const int D3 = Dc * Dc * Dc;
    const int cf = (int)(t % D3);
    const int64_t re = t / D3;
    const int f[3] = {cf / (Dc * Dc), (cf / Dc) % Dc, cf % Dc};
    int Rv[3][2], nt[3], pw[3][2];                  // terms per axis: R, and the power of i
    for (int a = 0; a < 3; ++a) {
        const int R = (f[a] + 1) / 2, even = f[a] && !(f[a] & 1);
        nt[a] = f[a] ? 2 : 1;
        Rv[a][0] = R;
        Rv[a][1] = -R;
        pw[a][0] = even ? 1 : 0;                    // i v[R]
        pw[a][1] = even ? 3 : 0;                    // -i v[-R]
    }
    double2 s = make_double2(0, 0);
    for (int x = 0; x < nt[0]; ++x)
        for (int y = 0; y < nt[1]; ++y)
            for (int z = 0; z < nt[2]; ++z) {
                const int c = ((Rv[0][x] + rc) * Dc + (Rv[1][y] + rc)) * Dc + (Rv[2][z] + rc);
                double2 v = make_double2(0, 0);
                for (int rp = cube[c]; rp >= 0; rp = cube[D3 + rp]) {
                    const size_t gi = ((size_t)re * nRp + rp) * rowlen + e;
                    v = cadd(v, g64 ? g64[gi] : make_double2(g32[gi].x, g32[gi].y));
                }
                const int p = (pw[0][x] + pw[1][y] + pw[2][z]) & 3;     // s += i^p v
                const double px = p & 1 ? v.y : v.x, py = p & 1 ? v.x : v.y;
                s.x += p == 1 || p == 2 ? -px : px;
                s.y += p & 2 ? -py : py;
            }
    using R = decltype(C2::x);
    C2 o;
    o.x = (R)s.x;
    o.y = (R)s.y;
    out[idx] = o;
}

// Gather tables (FP32) in blocks of 64 grid points, one row of 64 per element, so that lanes on
// nearby points read contiguous memory and one address serves every element of a point (the rows
// lie at fixed distances).
// k+q side, [k / 64][m]: W / 2 rows of two V_im(k) each (odd W: W rows of one), then one row of
// (eps_mk - mu, f_mk).  q side, [q / 64]: N_m^2 rows of u_mu,nu(q), then N_m rows of
// (hbar omega, N).  Sizes in float2.
constexpr int kTb = 64;
__host__ __device__ constexpr int kq_block(int W) { return kTb * (W + 1); }
__host__ __device__ constexpr int q_block(int NM) { return kTb * (NM * NM + NM); }

__global__ void k_kq_table(int64_t nk, int W, const float2 *__restrict__ V, const float *__restrict__ erel,
                           const float *__restrict__ f32, float2 *__restrict__ out) {
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t k = idx / W;
    const int m = (int)(idx % W);
    if (k >= nk) return;
    float2 *o = out + ((k / kTb) * W + m) * kq_block(W);
    const int x = (int)(k % kTb), w = W % 2 ? 1 : 2;
    for (int i = 0; i < W; ++i) o[(i / w) * (kTb * w) + x * w + i % w] = V[k * W * W + i * W + m];
    o[kTb * W + x] = make_float2(erel[idx], f32[idx]);
}

__global__ void k_q_table(int64_t nq, int NM, const float2 *__restrict__ u, const float *__restrict__ hw,
                          const float *__restrict__ n, float2 *__restrict__ out) {
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t q = idx % nq;
    const int e = (int)(idx / nq);
    if (e >= NM * NM + NM) return;
    float2 v;
    if (e < NM * NM) v = u[q * NM * NM + e];
    else v = make_float2(hw[q * NM + e - NM * NM], n[q * NM + e - NM * NM]);
    out[(q / kTb) * q_block(NM) + e * kTb + q % kTb] = v;
}

struct SfArgs {
    GridInfo g;
    int nplane;                     // N2 N3
    FDiv fn3, fper;                 // division by N3 and by the columns of a group (jq X / 2 or jq X)
    int jq;                         // q2 values per group (Y and the U buffers hold one group)
    int njg;                        // groups per plane block (over the largest block)
    int pbmax;                      // plane blocks
    const float *coef;              // [N1 + N2 + N3][D - 1] cos, sin of theta R (k_sf_coef)
    const float2 *ghat;             // [state - s_base][D^3 forms][N_m][W]
    const int *kpts, *win_lo, *win_n;
    const int64_t *kp_state;        // chunk k-points' first states (global)
    int64_t s_base;
    const uint32_t *mask;           // sieve decisions of the chunk's k-points (rows of mask_words)
    int64_t mask_words;
    const float2 *kqt, *qt;         // gather tables (k_kq_table, k_q_table)
    const float *erel, *hwmax32;
    float ceta32, inv_eta32;
    double pref;                    // 2 pi / (hbar N_q sqrt(pi) eta)
    double *inv_tau;
    int nkp;                        // k-points of the chunk
    float *gam;                     // Gamma capture (iterative BTE) or nullptr: row n of each
    const uint32_t *goff;           // pair's block, block start gent[kp] + goff[chunk pair]
    const int64_t *gent;
    const int64_t *kp_pairs;        // with a capture: chunk-local pair offsets, minus p_off, and the
    int64_t p_off;                  // run tables (sieve.cuh), which place a pair in the list
    const int *runs;
    int64_t run_stride;
};

template <int NF>
__device__ __forceinline__ void load_coef(const float *p, float (&c)[NF]) {
    if constexpr (NF == 4) {
        const float4 v = *reinterpret_cast<const float4 *>(p);
        c[0] = v.x; c[1] = v.y; c[2] = v.z; c[3] = v.w;
    } else {
#pragma unroll
        for (int f = 0; f < NF; f += 2) {
            const float2 v = *reinterpret_cast<const float2 *>(p + f);
            c[f] = v.x;
            c[f + 1] = v.y;
        }
    }
}

template <int NF>
__device__ __forceinline__ void load_coef_g(const float *__restrict__ p, float (&c)[NF]) {
    if constexpr (NF == 4) {
        const float4 v = __ldg(reinterpret_cast<const float4 *>(p));
        c[0] = v.x; c[1] = v.y; c[2] = v.z; c[3] = v.w;
    } else {
#pragma unroll
        for (int f = 0; f < NF; f += 2) {
            const float2 v = __ldg(reinterpret_cast<const float2 *>(p + f));
            c[f] = v.x;
            c[f + 1] = v.y;
        }
    }
}

// v += c w, two packed multiply-adds (one issue slot for two FP32 FMAs)
__device__ __forceinline__ void ffma4(float c, const float4 &w, float4 &v) {
    const float2 cc = make_float2(c, c);
    const float2 lo = __ffma2_rn(cc, make_float2(w.x, w.y), make_float2(v.x, v.y));
    const float2 hi = __ffma2_rn(cc, make_float2(w.z, w.w), make_float2(v.z, v.w));
    v = make_float4(lo.x, lo.y, hi.x, hi.y);
}

template <int W, int NM, int RC, bool GAM>
__global__ void __launch_bounds__(kSfThreads, (W <= 4 ? 3 : 2)) k_scatter_sf(SfArgs a) {
    constexpr int D = 2 * RC + 1;
    constexpr int NF = D - 1;                    // forms with a cos / sin coefficient
    constexpr int X = NM * W;                    // columns (mu, i)
    constexpr bool V2 = (W % 2) == 0;            // rows of W float2 are 16-byte aligned
    constexpr int kMuUnroll = NM <= 3 ? NM : 1;  // wide systems: one mode row at a time (registers)
    extern __shared__ __align__(16) float2 sm[];
    const int N1 = a.g.n1, N2 = a.g.n2, N3 = a.g.n3;
    const int JQ = a.jq, NJG = a.njg;
    const SfSmem lay = sf_smem_layout(D, X, W, JQ, N1, N3, NJG, a.pbmax, sizeof(float));
    float2 *Y = sm;                              // [D f1][D f3][JQ][X]
    float *CS3 = reinterpret_cast<float *>(Y + lay.y + lay.u);  // [N3][NF]: axis-3 coefficients
    const int nh = N1 / 2 + 1;
    float *rs = CS3 + lay.cs;                           // [nh]: sums of the current group's items
    // two lists, of the current group and the next: [nh] items (q1, N1 - q1), their number, next one to take
    int *lists = reinterpret_cast<int *>(rs + lay.rs);
    uint32_t *flags = reinterpret_cast<uint32_t *>(lists + 2 * (nh + 2));   // bit pb NJG + jg: the group has pairs
    uint8_t *clist = reinterpret_cast<uint8_t *>(flags + lay.flags) + (threadIdx.x >> 5) * kSieveBlock;
    uint16_t *left = reinterpret_cast<uint16_t *>(reinterpret_cast<uint8_t *>(flags + lay.flags) + kSfWarps * kSieveBlock) +
                     (threadIdx.x >> 5) * 32 * W;       // see below
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int ustride = D * JQ * X;
    float2 *Uw = Y + lay.y + (size_t)wid * 2 * ustride;  // this warp's two runs: [2][D f3][JQ][X]
    const int64_t s = a.s_base + blockIdx.x;     // global state
    // its k-point: the last one whose first state is <= s (every listed k-point has a state)
    const int kp = (int)lower_bound(0, a.nkp, s + 1, [&](int64_t p) { return a.kp_state[p + 1]; });
    const int n = (int)(s - a.kp_state[kp]);
    const int ik = a.kpts[kp];
    const int lo = a.win_lo[ik];
    const float2 *gs = a.ghat + (size_t)(s - a.s_base) * D * D * D * X;
    const float *CS1 = a.coef, *CS2 = CS1 + N1 * NF;
    for (int e = tid; e < N3 * NF; e += kSfThreads) CS3[e] = CS2[N2 * NF + e];
    const int nplane = a.nplane;
    const uint32_t *mrow = a.mask + (int64_t)kp * a.mask_words;   // [pb][q1][8 words]
    const SfGroups groups{mrow, flags, a.fn3, N1, N3, nplane, JQ, NJG};
    mark_groups(groups, (int)lay.flags);
    int k1, k2, k3;
    grid_coords(a.g, ik, k1, k2, k3);
    const float en = a.erel[(int64_t)ik * W + lo + n];
    const float ceta = a.ceta32, ieta = a.inv_eta32;
    double acc = 0;                              // warp 0: sums of the items lane, lane + 32, ...
    __syncthreads();                             // flags and CS3 are complete
    int f = groups.next(-1), buf = 0;
    if (wid == 0 && f >= 0) list_items(groups.group(f), N1, lists);
    for (; f >= 0; buf ^= 1) {
        const SfGroup grp = groups.group(f);
        const int c_lo = grp.c_lo, q2lo = grp.q2lo, j0 = grp.j0, jn = grp.jn;
        int *gl = lists + buf * (nh + 2);
        const int fnext = groups.next(f);
        // Y of this group's q2 values (all threads), read from ghat' (L1 / L2): two columns per
        // thread and step; the index is taken apart by a launch constant and compile-time ones
        if constexpr (X % 2 == 0) {
            const int per4 = JQ * (X / 2);
            for (int e = tid; e < D * D * per4; e += kSfThreads) {
                const int r13 = fdiv(e, a.fper), e2 = e - r13 * per4;
                const int jj = e2 / (X / 2), col2 = e2 - jj * (X / 2);
                if (jj >= jn) continue;
                const int f1 = r13 / D, f3 = r13 - f1 * D;
                float c2[NF];
                load_coef_g<NF>(CS2 + (q2lo + j0 + jj) * NF, c2);
                const float4 *src = reinterpret_cast<const float4 *>(gs + ((f1 * D) * D + f3) * X) + col2;
                float4 v = __ldg(src);                   // form f2 = 0
#pragma unroll
                for (int f2 = 1; f2 < D; ++f2) {
                    ffma4(c2[f2 - 1], __ldg(src + f2 * D * X / 2), v);
                }
                reinterpret_cast<float4 *>(Y)[e] = v;    // [r13][jj][col], rows of JQ X
            }
        } else {
            for (int e = tid; e < D * D * JQ * X; e += kSfThreads) {
                const int r13 = fdiv(e, a.fper), e2 = e - r13 * JQ * X;
                const int jj = e2 / X, col = e2 - jj * X;
                if (jj >= jn) continue;
                const int f1 = r13 / D, f3 = r13 - f1 * D;
                const float *c2 = CS2 + (q2lo + j0 + jj) * NF;
                const float2 *src = gs + ((f1 * D) * D + f3) * X + col;
                float2 v = __ldg(src);
#pragma unroll
                for (int f2 = 1; f2 < D; ++f2) {
                    const float c = c2[f2 - 1];
                    const float2 w = __ldg(src + f2 * D * X);
                    v.x = fmaf(c, w.x, v.x);
                    v.y = fmaf(c, w.y, v.y);
                }
                Y[e] = v;
            }
        }
        __syncthreads();
        const int ng = gl[nh];
        // items are taken from a counter; each writes its own sum, so the result does not
        // depend on which warp takes it
        int r = 0;
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
            {
                float c1[NF];
                load_coef_g<NF>(CS1 + q1 * NF, c1);
                if constexpr (X % 2 == 0) {
                    // (f3, e2) over D rows of per4 float4, walked as one list by the lanes
                    const int per4 = jn * X / 2;
                    int f3 = 0, e2 = lane;
                    while (true) {
                        while (e2 >= per4 && f3 < D) {
                            e2 -= per4;
                            ++f3;
                        }
                        if (f3 >= D) break;
                        const float4 *src = reinterpret_cast<const float4 *>(Y + (size_t)f3 * JQ * X) + e2;
                        float4 v = src[0], o = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                        for (int R = 1; R <= RC; ++R) {
                            const float4 w = src[(2 * R - 1) * D * JQ * X / 2], z = src[2 * R * D * JQ * X / 2];
                            ffma4(c1[2 * R - 2], w, v);
                            ffma4(c1[2 * R - 1], z, o);
                        }
                        float4 *dst = reinterpret_cast<float4 *>(Uw + (size_t)f3 * JQ * X) + e2;
                        dst[0] = make_float4(v.x + o.x, v.y + o.y, v.z + o.z, v.w + o.w);
                        dst[ustride / 2] = make_float4(v.x - o.x, v.y - o.y, v.z - o.z, v.w - o.w);
                        e2 += 32;
                    }
                } else {
                    const int per = jn * X;
#pragma unroll
                    for (int f3 = 0; f3 < D; ++f3) {
                        const float2 *src = Y + (size_t)f3 * JQ * X;
                        float2 *dst = Uw + (size_t)f3 * JQ * X;
                        for (int e = lane; e < per; e += 32) {
                            float2 v = src[e], o = make_float2(0.f, 0.f);
#pragma unroll
                            for (int R = 1; R <= RC; ++R) {
                                const float2 w = src[e + (2 * R - 1) * D * JQ * X], z = src[e + 2 * R * D * JQ * X];
                                v.x = fmaf(c1[2 * R - 2], w.x, v.x);
                                v.y = fmaf(c1[2 * R - 2], w.y, v.y);
                                o.x = fmaf(c1[2 * R - 1], z.x, o.x);
                                o.y = fmaf(c1[2 * R - 1], z.y, o.y);
                            }
                            dst[e] = make_float2(v.x + o.x, v.y + o.y);
                            dst[e + ustride] = make_float2(v.x - o.x, v.y - o.y);
                        }
                    }
                }
            }
            float rate = 0.f;
            int b1a = k1 + q1, b1b = k1 + q1b;
            if (b1a >= N1) b1a -= N1;
            if (b1b >= N1) b1b -= N1;
            // The pairs of both runs as one list of combinations (one run at a time where both hold
            // more than a plane block's worth), 32 at a time, each lane with the first final band
            // within reach of its pair.  The few further bands are kept in a list of the
            // warp, (pair, band), and worked off 32 at a time as well: one lane with two bands
            // would otherwise hold up the other 31 for a second pass over the band.
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
                    const int ikq = ((second ? b1b : b1a) * N2 + b2) * N3 + b3;   // nk W^2 < 2^31 (checked on the host)
                    if (fresh) {
                        // final bands within the largest kept mode energy + c eta of e_nk (a superset
                        // of the bands with a mode inside c eta of either shell; the others add zero)
                        unsigned mask = 0;
                        if (have) {
                            const float lim = __ldg(a.hwmax32 + q) + ceta + 1e-5f;
                            if constexpr (W % 4 == 0) {
#pragma unroll
                                for (int m4 = 0; m4 < W / 4; ++m4) {
                                    const float4 e4 = __ldg(reinterpret_cast<const float4 *>(a.erel + ikq * W) + m4);
                                    mask |= (fabsf(en - e4.x) <= lim ? 1u : 0u) << (4 * m4);
                                    mask |= (fabsf(en - e4.y) <= lim ? 2u : 0u) << (4 * m4);
                                    mask |= (fabsf(en - e4.z) <= lim ? 4u : 0u) << (4 * m4);
                                    mask |= (fabsf(en - e4.w) <= lim ? 8u : 0u) << (4 * m4);
                                }
                            } else {
#pragma unroll
                                for (int mm = 0; mm < W; ++mm)
                                    mask |= (fabsf(en - __ldg(a.erel + ikq * W + mm)) <= lim ? 1u : 0u) << mm;
                            }
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
                    const float2 *Ub = Uw + (second ? ustride : 0) + (j - j0) * X;   // form f3 at + f3 JQ X
                    float c3[NF];
                    load_coef<NF>(CS3 + q3 * NF, c3);
                    const float2 *uq = a.qt + (int64_t)(q / kTb) * q_block(NM) + q % kTb;   // element e at + e kTb
                    const float2 *kt = a.kqt + ((int64_t)(ikq / kTb) * W + m) * kq_block(W);
                    const int x64 = ikq % kTb;
                    int lokq = 0, nwkq = 0;
                    int64_t grow = 0;                        // this band's row of the pair's Gamma block
                    if constexpr (GAM) {
                        lokq = __ldg(a.win_lo + ikq);
                        nwkq = __ldg(a.win_n + ikq);
                        const int t = second ? t0b + tt - npa : t0 + tt;    // the pair's place in the k-point's list
                        grow = a.gent[kp] + a.goff[a.kp_pairs[kp] - a.p_off + t] + (int64_t)n * nwkq - lokq;
                    }
                    const float2 emf = __ldg(kt + kTb * W + x64);
                    const float em = emf.x, fm = emf.y;
                    float2 Vc[W];                        // column m of V(k+q)
                    if constexpr (V2) {
#pragma unroll
                        for (int i = 0; i < W / 2; ++i) {
                            const float4 v = __ldg(reinterpret_cast<const float4 *>(kt) + i * kTb + x64);
                            Vc[2 * i] = make_float2(v.x, v.y);
                            Vc[2 * i + 1] = make_float2(v.z, v.w);
                        }
                    } else {
#pragma unroll
                        for (int i = 0; i < W; ++i) Vc[i] = __ldg(kt + i * kTb + x64);
                    }
                    // (hbar omega, N) of the modes, loaded ahead of the rotation.  Wide systems form the
                    // occupation x delta factors ahead as well, while V and u travel, and pass over a band
                    // without any (Si-like 100^3 12.8 -> 11.9 ms; for W = 4 the registers are missed: 48^3
                    // 45.4 -> 46.3 ms).
                    constexpr bool kEarly = W > 4;
                    float2 wn[NM];
#pragma unroll
                    for (int nu = 0; nu < NM; ++nu) wn[nu] = __ldg(uq + (NM * NM + nu) * kTb);
                    auto factor = [&](int nu) -> float {
                        const float w = wn[nu].x, nq = wn[nu].y;
                        const float x1 = (en + w) - em;
                        const float x2 = (en - w) - em;
                        float tt = 0.f;
                        if (fabsf(x1) <= ceta) {
                            const float y = x1 * ieta;
                            tt += (nq + fm) * __expf(-y * y);
                        }
                        if (fabsf(x2) <= ceta) {
                            const float y = x2 * ieta;
                            tt += (1.f + nq - fm) * __expf(-y * y);
                        }
                        return tt;
                    };
                    float td[kEarly ? NM : 1];
                    if constexpr (kEarly) {
                        bool any = GAM;
#pragma unroll
                        for (int nu = 0; nu < NM; ++nu) {
                            td[nu] = wn[nu].x < 0.f ? 0.f : factor(nu);
                            any |= td[nu] != 0.f;
                        }
                        if (!any) continue;
                    }
                        float2 gr[NM], gi[NM];
#pragma unroll
                        for (int nu = 0; nu < NM; ++nu) gr[nu] = gi[nu] = make_float2(0.f, 0.f);
#pragma unroll kMuUnroll
                        for (int mu = 0; mu < NM; ++mu) {
                            float2 G[W];
                            const float2 *u0 = Ub + mu * W;
                            if constexpr (V2) {
#pragma unroll
                                for (int i = 0; i < W / 2; ++i) {
                                    const float4 v = reinterpret_cast<const float4 *>(u0)[i];
                                    G[2 * i] = make_float2(v.x, v.y);
                                    G[2 * i + 1] = make_float2(v.z, v.w);
                                }
#pragma unroll
                                for (int f = 1; f < D; ++f) {
                                    const float2 c = make_float2(c3[f - 1], c3[f - 1]);
                                    const float4 *uf = reinterpret_cast<const float4 *>(u0 + f * JQ * X);
#pragma unroll
                                    for (int i = 0; i < W / 2; ++i) {
                                        const float4 v = uf[i];
                                        G[2 * i] = __ffma2_rn(c, make_float2(v.x, v.y), G[2 * i]);
                                        G[2 * i + 1] = __ffma2_rn(c, make_float2(v.z, v.w), G[2 * i + 1]);
                                    }
                                }
                            } else {
#pragma unroll
                                for (int i = 0; i < W; ++i) G[i] = u0[i];
#pragma unroll
                                for (int f = 1; f < D; ++f) {
                                    const float2 c = make_float2(c3[f - 1], c3[f - 1]);
#pragma unroll
                                    for (int i = 0; i < W; ++i) G[i] = __ffma2_rn(c, u0[f * JQ * X + i], G[i]);
                                }
                            }
                            // h = sum_i conj(V_i) G_i and g_nu += h u as real and imaginary factor
                            // times (x, y), put together at the end
                            float2 hr = make_float2(0.f, 0.f), hi = make_float2(0.f, 0.f);
#pragma unroll
                            for (int i = 0; i < W; ++i) {
                                hr = __ffma2_rn(make_float2(Vc[i].x, Vc[i].x), G[i], hr);
                                hi = __ffma2_rn(make_float2(Vc[i].y, Vc[i].y), G[i], hi);
                            }
                            const float hx = hr.x + hi.y, hy = hr.y - hi.x;
#pragma unroll
                            for (int nu = 0; nu < NM; ++nu) {
                                const float2 u = __ldg(uq + (mu * NM + nu) * kTb);
                                gr[nu] = __ffma2_rn(make_float2(hx, hx), u, gr[nu]);
                                gi[nu] = __ffma2_rn(make_float2(hy, hy), u, gi[nu]);
                            }
                        }
                        float gm = 0.f;                      // Gamma capture: sum over modes
#pragma unroll
                        for (int nu = 0; nu < NM; ++nu) {
                            if (!kEarly && wn[nu].x < 0.f) continue;
                            const float gx = gr[nu].x - gi[nu].y, gy = gr[nu].y + gi[nu].x;
                            const float g2 = gx * gx + gy * gy;
                            const float tt = kEarly ? td[kEarly ? nu : 0] : factor(nu);
                            rate = fmaf(g2, tt, rate);
                            if constexpr (GAM) gm = fmaf(g2, tt, gm);
                        }
                        if constexpr (GAM) {
                            if (m >= lokq && m < lokq + nwkq) a.gam[grow + m] = gm;
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
            for (int r = lane; r < ng; r += 32) acc += (double)rs[r];
            __syncwarp();                                // before rs is rewritten by this warp's items
        }
        f = fnext;
    }
    // rs of the last group was consumed by warp 0: lanes by a fixed tree
    if (wid == 0) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (lane == 0) a.inv_tau[s] = a.pref * acc;
    }
}

template <int W, int NM, int RC, bool GAM>
void launch_sf_t(epwi_ctx *c, const SfArgs &a, int nitems, size_t sm) {
    allow_smem(k_scatter_sf<W, NM, RC, GAM>);
    EPWI_CUDA(cudaFuncSetAttribute(k_scatter_sf<W, NM, RC, GAM>, cudaFuncAttributePreferredSharedMemoryCarveout, 100));
    if (nitems > 0) {
        k_scatter_sf<W, NM, RC, GAM><<<(unsigned)nitems, kSfThreads, sm, c->stream>>>(a);
        EPWI_CHECK_LAUNCH();
    }
}

template <int W, int NM, int RC>
void launch_sf(epwi_ctx *c, const SfArgs &a, int nitems, size_t sm) {
    if (a.gam) launch_sf_t<W, NM, RC, true>(c, a, nitems, sm);
    else launch_sf_t<W, NM, RC, false>(c, a, nitems, sm);
}

}  // namespace

size_t sf_state_bytes(const epwi_ctx *c) {
    const size_t Dc = 2 * (size_t)c->sf_r + 1;
    return sizeof(float2) * Dc * Dc * Dc * c->nm * c->nw;
}

void sf_check(const epwi_ctx *c) {
    const int W = c->nw, NM = c->nm, r = c->sf_r;
    EPWI_REQUIRE(c->nk * std::max(W * W, NM * NM) < (int64_t(1) << 31), EPWI_EUNSUPPORTED,
                 "fp32 mode: grid too large for its 32-bit table offsets");
    EPWI_REQUIRE(sf_shape_built(W, NM, r), EPWI_EUNSUPPORTED,
                 "fp32 mode built for (nw, modes) in {(4,3), (8,6)} with R_p within |n| <= 3, and (1,3) "
                 "within |n| <= 2");
    EPWI_REQUIRE(c->ng[0] * 2 <= 4096 && c->ng[2] <= 0xffff, EPWI_EUNSUPPORTED, "fp32 mode: grid too large");
}

// cos and sin of theta R, R = 1 .. rc, for every point of the three axes (x R reduced exactly onto
// the L roots; x st < L): [N1 + N2 + N3][rc] pairs.
template <typename V2, typename V>
__global__ void k_sf_coef(GridInfo g, int rc, const V2 *__restrict__ ph, V *__restrict__ coef) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (g.n1 + g.n2 + g.n3) * rc) return;
    const int R = e % rc + 1, x = e / rc;
    const int p = x < g.n1 ? x * g.s1 : x < g.n1 + g.n2 ? (x - g.n1) * g.s2 : (x - g.n1 - g.n2) * g.s3;
    const V2 v = ph[p * R % g.L];
    coef[2 * e] = v.x;
    coef[2 * e + 1] = v.y;
}

template <typename V2, typename V>
void build_coef(epwi_ctx *c, const V2 *ph) {
    const GridInfo g = make_grid_info(c);
    const int nc = (g.n1 + g.n2 + g.n3) * c->sf_r;
    c->sf_coef.ensure(sizeof(V2) * nc);
    k_sf_coef<V2, V><<<(unsigned)((nc + 127) / 128), 128, 0, c->stream>>>(g, c->sf_r, ph, c->sf_coef.as<V>());
    EPWI_CHECK_LAUNCH();
}

// g' in the recombined cube forms (once per system).
template <class C2>
static void build_gsf(epwi_ctx *c, DevBuf &out) {
    const int Dc = 2 * c->sf_r + 1, rowlen = c->nm * c->nw * c->nw;
    const int64_t n = (int64_t)c->nRe * Dc * Dc * Dc * rowlen;
    DevBuf cube;
    upload_rp_map(c, cube);
    out.ensure(sizeof(C2) * n);
    k_sf_transform<C2><<<(unsigned)((n + 255) / 256), 256, 0, c->stream>>>(
        n, c->nRp, Dc, c->sf_r, rowlen, cube.as<int>(), c->keep_g64 ? c->gw64.as<double2>() : nullptr,
        c->gw32.as<float2>(), out.as<C2>());
    EPWI_CHECK_LAUNCH();
    EPWI_CUDA(cudaStreamSynchronize(c->stream));   // cube is released next
    cube.release();
}

void sf64_prepare(epwi_ctx *c) {
    build_coef<double2, double>(c, c->ph64.as<double2>());
    if (c->sf_g64_ready) return;
    build_gsf<double2>(c, c->gsf64);
    c->sf_g64_ready = true;
}

// Builds what the fp32 mode reads besides the eigen-tables: g' (cube embedding and the +-R
// recombination of the R_p axes, once per system) and the band-major FP32 V and (eps - mu, f)
// tables (per rates call).
void sf_prepare(epwi_ctx *c) {
    const int W = c->nw, NM = c->nm;
    if (!c->sf_g_ready) {
        build_gsf<float2>(c, c->gsf32);
        c->sf_g_ready = true;
    }
    build_coef<float2, float>(c, c->ph32.as<float2>());
    const int64_t nbk = (c->nk + kTb - 1) / kTb;
    c->sf_kqt.ensure(sizeof(float2) * nbk * W * kq_block(W));
    k_kq_table<<<(unsigned)((c->nk * W + 255) / 256), 256, 0, c->stream>>>(
        c->nk, W, c->V32.as<float2>(), c->tc_erel.as<float>(), c->tc_f32.as<float>(), c->sf_kqt.as<float2>());
    EPWI_CHECK_LAUNCH();
    c->sf_qt.ensure(sizeof(float2) * nbk * q_block(NM));
    k_q_table<<<(unsigned)((c->nk * (NM * NM + NM) + 255) / 256), 256, 0, c->stream>>>(
        c->nk, NM, c->u32.as<float2>(), c->tc_hw32.as<float>(), c->tc_n32.as<float>(), c->sf_qt.as<float2>());
    EPWI_CHECK_LAUNCH();
}

void sf_restage(epwi_ctx *c, const RestageArgs &ra_in) {
    RestageArgs ra = ra_in;
    const int Dc = 2 * c->sf_r + 1;
    ra.gw32 = c->gsf32.as<float2>();
    ra.nrow = Dc * Dc * Dc * c->nm * c->nw;
    const int W = ra.W;
    float2 *out = static_cast<float2 *>(ra.ghat_raw);
    if (kstage_pays(c, ra.nkp_all, ra.nrow, false)) {
        kstage_run<float2>(c, ra, c->gsf32.as<float2>(), c->ph32.as<float2>(), c->V32.as<float2>(), SfStore{out, ra.nrow});
        return;
    }
    auto go = [&](auto kern, int KG) {
        dim3 grid((ra.nrow + 127) / 128, (unsigned)((ra.nkp + KG - 1) / KG));
        const size_t sm = sizeof(float2) * KG * ra.nRe;
        if (sm > 48 * 1024) allow_smem(kern);
        kern<<<grid, 128, sm, c->stream>>>(ra, out);
        EPWI_CHECK_LAUNCH();
    };
    auto kb = [&](auto kern, int rows_per_block) {
        dim3 grid((ra.nrow + rows_per_block - 1) / rows_per_block, (unsigned)((ra.nkp + 31) / 32));
        kern<<<grid, 256, 0, c->stream>>>(ra, out);
        EPWI_CHECK_LAUNCH();
    };
    // measured: the k-blocked kernel pays for the Si-like shape (72 -> 53 ms at 100^3) and not
    // for W = 4 (6.8 -> 9.2 ms at 48^3)
    if (W == 4) go(k_restage_f32<4, 8>, 8);
    else if (W == 8) kb(k_restage_f32_kb<8>, 32);
    else if (W == 1) go(k_restage_f32<1, 8>, 8);
    else go(k_restage_f32<0, 1>, 1);
}

// The grids that the mode takes, a fixed rule: at most 8192 (q1, q2 group) runs per plane block and 8192
// plane blocks, and 200 KB for one run's U per warp, Y, the three axes' coefficients and the
// run bounds.  The kernel's own layout (sf_smem_layout) of every such grid is within 227 KB.
static void sf_check_grid(int D, int X, int q2max, const GridInfo &g) {
    const size_t per_j = sizeof(float2) * D * X;
    const int jmax = std::max(1, std::min({q2max, (int)(40 * 1024 / (per_j * D)), (int)(36 * 1024 / (per_j * kSfWarps))}));
    const int64_t njg = (q2max + jmax - 1) / jmax, jq = (q2max + njg - 1) / njg;
    const int64_t blocks = ((int64_t)g.n2 * g.n3 + kSieveBlock - 1) / kSieveBlock;
    EPWI_REQUIRE(g.n1 * njg <= 8192 && blocks <= 8192, EPWI_EUNSUPPORTED, "fp32 mode: too many runs or plane blocks");
    EPWI_REQUIRE(jq * per_j * (D + kSfWarps) + sizeof(float) * ((int64_t)g.n1 + g.n2 + g.n3) * (D - 1) +
                         sizeof(int) * (kSieveBlock + 2 * g.n1 * njg + g.n1 + blocks + 5) <= 200 * 1024,
                 EPWI_EUNSUPPORTED, "fp32 mode: the plane-block tables of this grid do not fit in shared memory");
}

// Rates of the chunk's states: one CTA per (k-point, band), written straight into inv_tau.
void sf_scatter(epwi_ctx *c, const ScatterArgs &sa, int64_t nkp, const int64_t *kp_pairs_local, int64_t p_off) {
    const int W = c->nw, NM = c->nm, r = c->sf_r;
    const int D = 2 * r + 1, X = NM * W;
    SfArgs a;
    a.g = sa.g;
    a.nplane = sa.g.n2 * sa.g.n3;
    const int q2max = sf_q2max(sa.g.n2, sa.g.n3);
    sf_check_grid(D, X, q2max, sa.g);
    const SfPlan plan = sf_plan(D, X, W, q2max, sa.g.n1, sa.g.n2, sa.g.n3, sizeof(float));
    a.jq = plan.jq;
    a.njg = plan.njg;
    a.pbmax = plan.pbmax;
    a.fn3 = make_fdiv((uint32_t)sa.g.n3);
    a.fper = make_fdiv((uint32_t)(X % 2 ? plan.jq * X : plan.jq * (X / 2)));
    a.coef = c->sf_coef.as<float>();
    a.mask = sa.mask;
    a.mask_words = sa.mask_words;
    a.runs = sa.runs;
    a.run_stride = run_stride(sa.g);
    a.hwmax32 = c->hwmax32.as<float>();
    a.ghat = static_cast<const float2 *>(sa.ghat_raw);
    a.kpts = sa.kpts;
    a.win_lo = sa.win_lo;
    a.win_n = sa.win_n;
    a.kp_state = sa.kp_state;
    a.s_base = sa.s_base;
    a.kp_pairs = kp_pairs_local;
    a.p_off = p_off;
    a.kqt = c->sf_kqt.as<float2>();
    a.qt = c->sf_qt.as<float2>();
    a.erel = c->tc_erel.as<float>();
    a.ceta32 = (float)sa.ceta;
    a.inv_eta32 = (float)(1.0 / sa.eta);
    a.pref = 2.0 * epc::kPi / epc::kHbarEVs / (double)c->nk / (sqrt(epc::kPi) * sa.eta);
    a.inv_tau = c->inv_tau.as<double>();
    a.nkp = (int)nkp;
    a.gam = sa.gam32;
    a.goff = sa.goff;
    a.gent = sa.gent;
    const int ni = (int)sa.nstates_chunk;
    const size_t sm = plan.smem;
    if (W == 4 && NM == 3 && r == 1) launch_sf<4, 3, 1>(c, a, ni, sm);
    else if (W == 4 && NM == 3 && r == 2) launch_sf<4, 3, 2>(c, a, ni, sm);
    else if (W == 4 && NM == 3 && r == 3) launch_sf<4, 3, 3>(c, a, ni, sm);
    else if (W == 1 && NM == 3 && r == 1) launch_sf<1, 3, 1>(c, a, ni, sm);
    else if (W == 1 && NM == 3 && r == 2) launch_sf<1, 3, 2>(c, a, ni, sm);
    else if (W == 8 && NM == 6 && r == 1) launch_sf<8, 6, 1>(c, a, ni, sm);
    else if (W == 8 && NM == 6 && r == 2) launch_sf<8, 6, 2>(c, a, ni, sm);
    else if (W == 8 && NM == 6 && r == 3) launch_sf<8, 6, 3>(c, a, ni, sm);
    else sf_check(c);
}
