// Pieces shared by the sum-factorised Rp->q kernels (scatter_sf.cu in FP32, scatter_sf64.cu in
// FP64; internal).
#pragma once

#include <algorithm>

#include "epwi_internal.cuh"
#include "sieve.cuh"

constexpr int kSfThreads = 256;
constexpr int kSfWarps = kSfThreads / 32;

// Division by a divisor fixed at launch (x < 2^31): q = (umulhi(x, m) + x) >> l with
// l = ceil(log2 d), m = floor(2^32 (2^l - d) / d) + 1 (Granlund & Montgomery, PLDI 1994).
struct FDiv {
    uint32_t d, m, l;
};
inline FDiv make_fdiv(uint32_t d) {
    FDiv f;
    f.d = d;
    uint32_t l = 0;
    while ((uint64_t(1) << l) < d) ++l;
    f.l = l;
    f.m = (uint32_t)(((uint64_t(1) << 32) * ((uint64_t(1) << l) - d)) / d + 1);
    return f;
}
__device__ __forceinline__ int fdiv(int x, const FDiv &f) {
    return (int)((__umulhi((uint32_t)x, f.m) + (uint32_t)x) >> f.l);
}

// first position in [lo, hi) whose key is >= key (keys ascending)
template <typename F>
__device__ __forceinline__ int64_t lower_bound(int64_t lo, int64_t hi, int64_t key, F keyof) {
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if (keyof(mid) < key) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

// Shared-memory layout of the kernels (in units of their real type, then bytes): Y of one q2 group, two
// runs' U per warp, the axis-3 coefficients, the sums of a group's items; the items, the flags of the
// groups, and per warp a list of combinations and one of left-over bands.
struct SfSmem {
    size_t y, u, cs, rs, flags, bytes;           // complex, complex, real, real, words, bytes
};
__host__ __device__ inline SfSmem sf_smem_layout(int D, int X, int W, int jq, int N1, int N3, int njg, int pbmax,
                                                 size_t real) {
    SfSmem s;
    s.y = ((size_t)D * D * jq * X + 1) & ~size_t(1);       // an even count: what follows stays 16-byte aligned
    s.u = (size_t)kSfWarps * 2 * D * jq * X;
    s.cs = ((size_t)N3 * (D - 1) + 3) & ~size_t(3);
    s.rs = (size_t)(N1 / 2 + 1);
    s.flags = ((size_t)pbmax * njg + 31) / 32;
    s.bytes = 2 * real * (s.y + s.u) + real * (s.cs + s.rs) + sizeof(int) * (2 * (s.rs + 2) + s.flags) +
              kSfWarps * ((size_t)kSieveBlock + 64 * (size_t)W);
    return s;
}

struct SfPlan {
    int jq, njg, pbmax;
    size_t smem;
};

// q2 values per group (jq): Y of one group and two runs' U per warp within budgets that keep two or
// more CTAs per SM (FP32: three for 12 columns, 74 KiB at jq = 7; FP64: two for 12 columns, 103 KiB at
// jq = 5, and one CTA's FP64 instructions run while the other waits at a barrier).
inline SfPlan sf_plan(int D, int X, int W, int q2max, int N1, int N2, int N3, size_t real) {
    const size_t ybudget = 10240 * real, ubudget = (real == 8 ? 10240 : 13824) * real;
    SfPlan p;
    const size_t per_j = 2 * real * D * X;
    const int jmax = std::max(1, std::min({q2max, (int)(ybudget / (per_j * D)), (int)(ubudget / (per_j * kSfWarps * 2))}));
    p.njg = (q2max + jmax - 1) / jmax;             // groups of equal size
    p.jq = (q2max + p.njg - 1) / p.njg;
    p.pbmax = (N2 * N3 + kSieveBlock - 1) / kSieveBlock;
    p.smem = sf_smem_layout(D, X, W, p.jq, N1, N3, p.njg, p.pbmax, real).bytes;
    return p;
}

// Most q2 values that a plane block of kSieveBlock consecutive (q2, q3) touches.
inline int sf_q2max(int64_t n2, int64_t n3) {
    int64_t q2max = 1;
    for (int64_t c0 = 0; c0 < n2 * n3; c0 += kSieveBlock) {
        const int64_t c1 = std::min<int64_t>(n2 * n3, c0 + kSieveBlock) - 1;
        q2max = std::max(q2max, c1 / n3 - c0 / n3 + 1);
    }
    return (int)q2max;
}

inline bool sf_shape_built(int W, int NM, int r) {
    return (W == 4 && NM == 3 && r >= 1 && r <= 3) || (W == 1 && NM == 3 && r >= 1 && r <= 2) ||
           (W == 8 && NM == 6 && r >= 1 && r <= 3);
}

// Groups of a state's pairs: plane block pb and group jg of its q2 values, f = pb NJG + jg.
struct SfGroup {
    int c_lo, q2lo, j0, jn;                      // first combination and q2 of the plane block; the group's q2
    int r0, r1;                                  // combinations [r0, r1) of the plane block belong to it
    const uint32_t *mpb;                         // mask words of the plane block
    // bits of word x (of 8) of a run that belong to the group
    __device__ uint32_t bits(int x) const {
        const int a0 = min(max(r0 - 32 * x, 0), 32), a1 = min(max(r1 - 32 * x, 0), 32);
        const uint32_t lo_m = a0 < 32 ? ~0u << a0 : 0u, hi_m = a1 < 32 ? ~(~0u << a1) : ~0u;
        return lo_m & hi_m;
    }
};
struct SfGroups {
    const uint32_t *mrow;                        // mask words of the k-point: [pb][q1][8]
    uint32_t *flags;                             // bit f: the group has pairs
    FDiv fn3;
    int N1, N3, nplane, JQ, NJG;
    __device__ int blocks() const { return (nplane + kSieveBlock - 1) / kSieveBlock; }
    // next group with pairs, or -1
    __device__ int next(int f) const {
        for (++f; f < blocks() * NJG; f = (f | 31) + 1) {
            const uint32_t b = flags[f >> 5] >> (f & 31);
            if (b) return f + __ffs(b) - 1;
        }
        return -1;
    }
    __device__ SfGroup group(int f) const {
        SfGroup u;
        const int pb = NJG == 1 ? f : f / NJG, jg = f - pb * NJG;
        u.c_lo = pb * kSieveBlock;
        u.q2lo = fdiv(u.c_lo, fn3);
        const int nq2 = fdiv(min(nplane, u.c_lo + kSieveBlock) - 1, fn3) - u.q2lo + 1;
        u.j0 = jg * JQ;
        u.jn = min(JQ, nq2 - u.j0);
        u.r0 = max(0, (u.q2lo + u.j0) * N3 - u.c_lo);
        u.r1 = min(kSieveBlock, (u.q2lo + u.j0 + u.jn) * N3 - u.c_lo);
        u.mpb = mrow + (int64_t)pb * N1 * 8;
        return u;
    }
};

// Flags of the groups with pairs (the whole CTA, up to a barrier that the caller has): every thread takes
// runs (pb, q1) and marks the groups of their set bits.
__device__ __forceinline__ void mark_groups(const SfGroups &g, int nflags) {
    for (int e = threadIdx.x; e < nflags; e += kSfThreads) g.flags[e] = 0u;
    __syncthreads();
    for (int r = threadIdx.x; r < g.blocks() * g.N1; r += kSfThreads) {
        const uint4 *w4 = reinterpret_cast<const uint4 *>(g.mrow) + 2 * (int64_t)r;
        const uint4 u = __ldg(w4), v = __ldg(w4 + 1);
        const uint32_t w[8] = {u.x, u.y, u.z, u.w, v.x, v.y, v.z, v.w};
        const int pb = r / g.N1;
        if (g.NJG == 1) {
            if (w[0] | w[1] | w[2] | w[3] | w[4] | w[5] | w[6] | w[7]) atomicOr(g.flags + (pb >> 5), 1u << (pb & 31));
            continue;
        }
        const int q2lo = fdiv(pb * kSieveBlock, g.fn3);
        int seen = -1;                           // last group marked
#pragma unroll
        for (int x = 0; x < 8; ++x) {
            uint32_t b = w[x];
            while (b) {
                const int c = x * 32 + __ffs(b) - 1;
                const int jg = (fdiv(pb * kSieveBlock + c, g.fn3) - q2lo) / g.JQ;
                if (jg != seen) {
                    const int f = pb * g.NJG + jg;
                    atomicOr(g.flags + (f >> 5), 1u << (f & 31));
                    seen = jg;
                }
                // on to the group's end
                const int end = (q2lo + (jg + 1) * g.JQ) * g.N3 - pb * kSieveBlock - x * 32;
                b = end < 32 ? b & ~((1u << end) - 1u) : 0u;
            }
        }
    }
}

// The items {q1, N1 - q1} of a group that have pairs, by one warp; gl[nh], gl[nh + 1]: their number, next
// one to take.  The largest come first, in four classes of size, so that the warps that take
// them finish together.
__device__ __forceinline__ void list_items(const SfGroup &g, int N1, int *gl) {
    const int lane = threadIdx.x & 31, nh = N1 / 2 + 1, n2 = (N1 - 1) / 2;   // n2: items with two runs
    auto pairs = [&](int q1) -> int {
        const uint4 *w4 = reinterpret_cast<const uint4 *>(g.mpb) + 2 * q1;
        const uint4 x = __ldg(w4), y = __ldg(w4 + 1);
        const uint32_t w[8] = {x.x, x.y, x.z, x.w, y.x, y.y, y.z, y.w};
        int c = 0;
#pragma unroll
        for (int i = 0; i < 8; ++i) c += __popc(w[i] & g.bits(i));
        return c;
    };
    int cnt = 0;
    auto put = [&](int v, bool on) {
        const unsigned b = __ballot_sync(0xffffffffu, on);
        if (on) gl[cnt + __popc(b & ((1u << lane) - 1u))] = v;
        cnt += __popc(b);
    };
    // h: 1 .. n2, then 0, then N1 / 2
    auto item = [&](int h, int &size) -> int {
        const int q1 = h < n2 ? h + 1 : h == n2 ? 0 : h;
        size = h < nh ? pairs(q1) + (h < n2 ? pairs(N1 - q1) : 0) : 0;
        return q1;
    };
    if (nh <= 64) {
        int s0, s1 = 0, q0 = 0, q1 = 0;
        q0 = item(lane, s0);
        if (nh > 32) q1 = item(lane + 32, s1);
        const int top = max(__reduce_max_sync(0xffffffffu, max(s0, s1)), 1);
        const int c0 = min(4 * s0 / top, 3), c1 = min(4 * s1 / top, 3);
        for (int cls = 3; cls >= 0; --cls) {
            put(q0, s0 > 0 && c0 == cls);
            if (nh > 32) put(q1, s1 > 0 && c1 == cls);
        }
    } else {                                     // many items: their order matters little
        for (int h0 = 0; h0 < nh; h0 += 32) {
            int s;
            const int q = item(h0 + lane, s);
            put(q, s > 0);
        }
    }
    if (lane == 0) {
        gl[nh] = cnt;
        gl[nh + 1] = 0;
    }
}
