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
    s.bytes = 2 * real * (s.y + s.u) + real * (s.cs + s.rs) + sizeof(int) * (s.rs + 2 + s.flags) +
              kSfWarps * ((size_t)kSieveBlock + 64 * (size_t)W);
    return s;
}

struct SfPlan {
    int jq, njg, pbmax;
    size_t smem;
};

// q2 values per group (jq): Y of one group and two runs' U per warp within budgets that keep two or
// more CTAs per SM (FP32: three for 12 columns, 70 KB at jq = 7; FP64: two for 12 columns, 101 KB at
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

