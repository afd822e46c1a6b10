// Interpolated electrons and phonons on the full grid (Sec. II B, Eqs. 4-6; Sec. III A
// preprocessing): H(k) and D(q) Fourier sums with exact integer phase reduction, Jacobi
// eigensolvers with FP64 results (jacobi.cuh), band velocities and phonon displacement vectors.
//
// One thread owns one grid point (matrices of up to 8 rows; a warp beyond).  The FP64 units
// bind: per point the kernels form only the upper triangle of the Hermitian sums, and the
// launches use small blocks on small grids so that every SM's FP64 unit has work.  Measured on one
// GB300 against plain FP64 Jacobi sweeps (FP64 sweeps after an FP32 start for 8 and 6 rows), all
// eigensolves and velocities of a step: Si-like 100^3 (8 and 6 rows) 65 -> 27.8 ms, metal 48^3 (4 and
// 3 rows) 2.9 -> 0.6 ms, tiny 8^3 0.57 -> 0.15 ms.  Each point is diagonalised once (Nk + Nq solves); the
// scattering loops gather V(k+q), u(q) from these tables instead of re-diagonalising per
// pair.
#include <algorithm>

#include "epwi_internal.cuh"
#include "jacobi.cuh"

namespace {

__global__ void k_phase_tables(int L, double2 *ph64, float2 *ph32) {
    int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= L) return;
    double s, c;
    sincospi(2.0 * (double)m / (double)L, &s, &c);   // e^{2 pi i m / L}
    ph64[m] = make_double2(c, s);
    ph32[m] = make_float2((float)c, (float)s);
}

// Sum-factorised Fourier builds (Eqs. 4-5 reordered, exact in real arithmetic).  With the
// R-set embedded in its bounding cube [-r, r]^3 (absent vectors carry zero), e^{ik.R} =
// e1(k1, n1) e2(k2, n2) e3(k3, n3) and X(k) = sum_n1 e1 sum_n2 e2 sum_n3 e3 X(n) is done in
// three stages, each shared by every grid point that needs it: axis 3 per (n1, n2, k3), axis 2
// per (n1, k2, k3), axis 1 inside the eigensolve kernels per k.  For the band velocities the
// n_b-weighted sums sum_n n_b e^{ik.R} H(R) ride along (VEL): dH/dk_a = i sum_b A_ba S_b with
// R_cart = sum_b n_b a_b.  E = entries per matrix; all FP64.
//   T[s][n1][n2][k3][e]:  s = 0: sum_n3 e3 X;   s = 1 (VEL): sum_n3 n3 e3 X
//   U[s][n1][k2][k3][e]:  s = 0: sum_n2 e2 T0;  s = 1: sum_n2 n2 e2 T0;  s = 2: sum_n2 e2 T1
__device__ __forceinline__ double2 axis_ph(const double2 *ph, int n, int a, int L) {
    int t = (n * a) % L;
    if (t < 0) t += L;
    return ph[t];
}

template <bool VEL>
__global__ void k_fac_axis3(int D, int rc, int N3, int s3, int L, int E, const double2 *__restrict__ Xc,
                            const double2 *__restrict__ ph, double2 *__restrict__ T) {
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t total = (int64_t)D * D * N3 * E;
    if (idx >= total) return;
    const int e = (int)(idx % E);
    const int64_t t = idx / E;
    const int k3 = (int)(t % N3);
    const int r12 = (int)(t / N3);
    const int a3 = (int)((int64_t)k3 * s3 % L);
    double2 s0 = make_double2(0, 0), s1 = make_double2(0, 0);
    for (int j = 0; j < D; ++j) {
        const int n3 = j - rc;
        const double2 v = cmul(axis_ph(ph, n3, a3, L), Xc[((int64_t)r12 * D + j) * E + e]);
        s0 = cadd(s0, v);
        if (VEL) s1 = make_double2(fma((double)n3, v.x, s1.x), fma((double)n3, v.y, s1.y));
    }
    T[((int64_t)r12 * N3 + k3) * E + e] = s0;
    if (VEL) T[(((int64_t)D * D + r12) * N3 + k3) * E + e] = s1;
}

template <bool VEL>
__global__ void k_fac_axis2(int D, int rc, int N2, int N3, int s2, int L, int E, const double2 *__restrict__ T,
                            const double2 *__restrict__ ph, double2 *__restrict__ U) {
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t plane = (int64_t)N2 * N3;
    const int64_t total = (int64_t)D * plane * E;
    if (idx >= total) return;
    const int e = (int)(idx % E);
    int64_t t = idx / E;
    const int k3 = (int)(t % N3);
    t /= N3;
    const int k2 = (int)(t % N2);
    const int r1 = (int)(t / N2);
    const int a2 = (int)((int64_t)k2 * s2 % L);
    double2 u0 = make_double2(0, 0), u1 = make_double2(0, 0), u2 = make_double2(0, 0);
    for (int j = 0; j < D; ++j) {
        const int n2 = j - rc;
        const double2 p = axis_ph(ph, n2, a2, L);
        const double2 v = cmul(p, T[(((int64_t)r1 * D + j) * N3 + k3) * E + e]);
        u0 = cadd(u0, v);
        if (VEL) {
            u1 = make_double2(fma((double)n2, v.x, u1.x), fma((double)n2, v.y, u1.y));
            u2 = cadd(u2, cmul(p, T[((((int64_t)D + r1) * D + j) * N3 + k3) * E + e]));
        }
    }
    const int64_t o = ((int64_t)r1 * plane + (int64_t)k2 * N3 + k3) * E + e;
    U[o] = u0;
    if (VEL) {
        U[(int64_t)D * plane * E + o] = u1;
        U[2 * (int64_t)D * plane * E + o] = u2;
    }
}

// The axis-2 stage output U[s][n1][k2 k3][e] of a factorised build (sources s = 0, 1, 2).
struct FacDesc {
    const double2 *U = nullptr;      // NULL: direct sums over the R-set
    int D, rc;
    int64_t plane;                   // N2 N3
};
struct Lattice {
    double a[3][3];                  // rows a_1, a_2, a_3 (A)
};

// Electrons: eps (ascending), V (columns), velocities, FP32 copies.
// fac.U given: H(k) from the factorised stages (and no velocities); otherwise direct sums, with the
// velocities of every point when do_vel is set.
// Above four bands the matrices live in local memory (4.5 KB a thread): 48 registers and ten blocks per
// SM cover its latency better than 226 registers and two, and the FP64 pipe binds (Si-like 100^3, 8
// bands and 6 modes: 35.1 -> 28.3 ms).
template <int WMAX, bool FIXED>
__global__ void __launch_bounds__(128, WMAX > 4 ? 10 : 1) k_eig_el(GridInfo g, int64_t nk, int W_, int nR,
                                                const int *__restrict__ R,
                                                const double *__restrict__ Rcart,
                                                const double2 *__restrict__ Hw,
                                                const double2 *__restrict__ ph,
                                                double *__restrict__ eps, float *__restrict__ eps32,
                                                double2 *__restrict__ Vout,
                                                float2 *__restrict__ V32,
                                                double *__restrict__ vel, int *__restrict__ flag,
                                                FacDesc fac, Lattice lat, int do_vel) {
    int64_t ik = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (ik >= nk) return;
    const int W = FIXED ? WMAX : W_;
    constexpr int U = WMAX <= 4 ? WMAX : 1;
    int i1, i2, i3;
    grid_coords(g, ik, i1, i2, i3);
    const int a1 = (int)((int64_t)i1 * g.s1 % g.L), a2 = (int)((int64_t)i2 * g.s2 % g.L),
              a3 = (int)((int64_t)i3 * g.s3 % g.L);
    double2 A[WMAX * WMAX], Vm[WMAX * WMAX];      // A: upper triangle
    const int WW = W * W;
    const int64_t pp = (int64_t)i2 * g.n3 + i3;   // (k2, k3) of this point (factorised build)
#pragma unroll U
    for (int i = 0; i < W; ++i)
#pragma unroll U
        for (int j = i; j < W; ++j) A[i * WMAX + j] = make_double2(0, 0);
    auto add = [&](double2 p, const double2 *h) {
#pragma unroll U
        for (int i = 0; i < W; ++i)
#pragma unroll U
            for (int j = i; j < W; ++j) A[i * WMAX + j] = cfma(p, h[i * W + j], A[i * WMAX + j]);
    };
    if (fac.U) {
        for (int j = 0; j < fac.D; ++j)
            add(axis_ph(ph, j - fac.rc, a1, g.L), fac.U + ((int64_t)j * fac.plane + pp) * WW);
    } else {
        for (int r = 0; r < nR; ++r)
            add(ph[phase_index(a1, a2, a3, R[3 * r], R[3 * r + 1], R[3 * r + 2], g.L)], Hw + (size_t)r * WW);
    }
    double w[WMAX];
    if (!eig_hermitian<WMAX>(A, Vm, W, w)) atomicAdd(flag, 1);
#pragma unroll U
    for (int n = 0; n < W; ++n) {
        eps[ik * W + n] = w[n];
        eps32[ik * W + n] = (float)w[n];
    }
#pragma unroll U
    for (int i = 0; i < W; ++i)
#pragma unroll U
        for (int j = 0; j < W; ++j) {
            const double2 v = Vm[i * WMAX + j];
            Vout[ik * WW + i * W + j] = v;
            V32[ik * WW + i * W + j] = make_float2((float)v.x, (float)v.y);
        }
    if (!do_vel) return;                 // velocities later, for the k-points that need them
    // v_n,a = (1/hbar) Re[V^dag (sum_R w_R i R_a e^{ik.R} H(R)) V]_nn, one axis at a time (direct
    // sums: the factorised build leaves the velocities to k_vel_fac)
    for (int ax = 0; ax < 3; ++ax) {
        for (int i = 0; i < W; ++i)
            for (int j = i; j < W; ++j) A[i * WMAX + j] = make_double2(0, 0);
        for (int r = 0; r < nR; ++r) {
            const double2 p = ph[phase_index(a1, a2, a3, R[3 * r], R[3 * r + 1], R[3 * r + 2], g.L)];
            const double ra = Rcart[3 * r + ax];
            add(make_double2(-ra * p.y, ra * p.x), Hw + (size_t)r * WW);   // i R_a e^{ik.R}
        }
        for (int n = 0; n < W; ++n) {
            double acc = 0;
            for (int i = 0; i < W; ++i) {
                const double2 vi = Vm[i * WMAX + n];
                acc = fma(A[i * WMAX + i].x, fma(vi.x, vi.x, vi.y * vi.y), acc);
                for (int j = i + 1; j < W; ++j) {
                    const double2 c = cmulc(vi, Vm[j * WMAX + n]);
                    acc = fma(2.0, fma(A[i * WMAX + j].x, c.x, -A[i * WMAX + j].y * c.y), acc);
                }
            }
            vel[(ik * W + n) * 3 + ax] = acc / epc::kHbarEVs * 1e-10;
        }
    }
}

// Band velocities from the factorised stages and the stored eigenvectors for the listed grid points
// (all n of them when list is NULL): with S_b(k) = sum_R n_b e^{ik.R} H(R) from the three sources, dH/dk_a =
// i sum_b A_ba S_b, so the expectation values of the Hermitian i S_b are taken once per lattice axis
// b and combined at the end.  32 points per block and a warp per b: the work is FP64 latency
// for the few points of a window (a thread per grid point and all three b in it: 33 us at 8^3, 0.85 ms
// at Si-like 100^3, where 4 of 1000 points lie in the window; now 17 us and 0.20 ms).
template <int WMAX, bool FIXED>
__global__ void __launch_bounds__(96) k_vel_fac(GridInfo g, int64_t n, int W_, const int *__restrict__ list,
                                                const double2 *__restrict__ ph, const double2 *__restrict__ Vin,
                                                double *__restrict__ vel, FacDesc fac, Lattice lat) {
    __shared__ double ex[3][WMAX][32];            // <n| i S_b |n>
    const int lane = threadIdx.x & 31, b = threadIdx.x >> 5;
    const int64_t x = (int64_t)blockIdx.x * 32 + lane;
    const bool on = x < n;
    const int64_t ik = !on ? 0 : list ? list[x] : x;
    const int W = FIXED ? WMAX : W_;
    constexpr int U = WMAX <= 4 ? WMAX : 1;
    if (on) {
        int i1, i2, i3;
        grid_coords(g, ik, i1, i2, i3);
        const int a1 = (int)((int64_t)i1 * g.s1 % g.L);
        const int WW = W * W;
        const int64_t pp = (int64_t)i2 * g.n3 + i3;
        const int64_t src = (int64_t)fac.D * fac.plane * WW;
        const double2 *V = Vin + ik * WW;
        double2 M[WMAX * WMAX];                   // upper triangle of i S_b
#pragma unroll U
        for (int i = 0; i < W; ++i)
#pragma unroll U
            for (int j = i; j < W; ++j) M[i * WMAX + j] = make_double2(0, 0);
        for (int d = 0; d < fac.D; ++d) {
            const int n1 = d - fac.rc;
            const double2 p = axis_ph(ph, n1, a1, g.L);
            const double s = b == 0 ? (double)n1 : 1.0;                    // the axis-1 weight is applied here
            const double2 ip = make_double2(-s * p.y, s * p.x);            // i n_1 e1 or i e1
            const double2 *u = fac.U + b * src + ((int64_t)d * fac.plane + pp) * WW;
#pragma unroll U
            for (int i = 0; i < W; ++i)
#pragma unroll U
                for (int j = i; j < W; ++j) M[i * WMAX + j] = cfma(ip, u[i * W + j], M[i * WMAX + j]);
        }
#pragma unroll U
        for (int m = 0; m < W; ++m) {
            double acc = 0;
#pragma unroll U
            for (int i = 0; i < W; ++i) {
                const double2 vi = V[i * W + m];
                acc = fma(M[i * WMAX + i].x, fma(vi.x, vi.x, vi.y * vi.y), acc);
#pragma unroll U
                for (int j = i + 1; j < W; ++j) {
                    const double2 c = cmulc(vi, V[j * W + m]);             // conj(v_i) v_j
                    acc = fma(2.0, fma(M[i * WMAX + j].x, c.x, -M[i * WMAX + j].y * c.y), acc);
                }
            }
            ex[b][m][lane] = acc;
        }
    }
    __syncthreads();
    if (on)                                       // Cartesian component b
        for (int m = 0; m < W; ++m)
            vel[(ik * W + m) * 3 + b] =
                (lat.a[0][b] * ex[0][m][lane] + lat.a[1][b] * ex[1][m][lane] + lat.a[2][b] * ex[2][m][lane]) *
                (1e-10 / epc::kHbarEVs);
}

// The force constants are real, so D(-q) = conj D(q): the solves run over the planes i1 <= N1 / 2, where of
// two points of the same plane the one with the smaller index takes both, and write the same
// energies and the conjugate vectors to -q.  Halves the FP64 work of every grid (Si-like 100^3, 6 modes:
// 13.7 -> 7.0 ms).
__device__ __forceinline__ int64_t minus_q(const GridInfo &g, int i1, int i2, int i3) {
    return ((int64_t)(i1 ? g.n1 - i1 : 0) * g.n2 + (i2 ? g.n2 - i2 : 0)) * g.n3 + (i3 ? g.n3 - i3 : 0);
}


// Phonons: hbar*omega, u = e (hbar^2 / (2 m hbar omega))^{1/2}, FP32 copies; D(q) from the
// factorised stages when fac.U is given.
template <int NMAX, bool FIXED>
__global__ void __launch_bounds__(128, NMAX > 4 ? 10 : 1) k_eig_ph(GridInfo g, int64_t nq, int Nm_, int nR,
                                                const int *__restrict__ R,
                                                const double *__restrict__ Phiw,
                                                const double *__restrict__ mode_mass,
                                                const double2 *__restrict__ ph, double omega_min,
                                                double *__restrict__ hw, float *__restrict__ hwmax32,
                                                float *__restrict__ hw32,
                                                double2 *__restrict__ uout,
                                                float2 *__restrict__ u32, int *__restrict__ flag,
                                                FacDesc fac) {
    int64_t iq = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (iq >= nq) return;
    const int Nm = FIXED ? NMAX : Nm_;
    constexpr int U = NMAX <= 4 ? NMAX : 1;
    int i1, i2, i3;
    grid_coords(g, iq, i1, i2, i3);
    const int64_t im = minus_q(g, i1, i2, i3);
    if (im < iq) return;                          // solved by that point's thread
    const int a1 = (int)((int64_t)i1 * g.s1 % g.L), a2 = (int)((int64_t)i2 * g.s2 % g.L),
              a3 = (int)((int64_t)i3 * g.s3 % g.L);
    double2 A[NMAX * NMAX], E[NMAX * NMAX];       // A: upper triangle
    const int MM = Nm * Nm;
#pragma unroll U
    for (int i = 0; i < Nm; ++i)
#pragma unroll U
        for (int j = i; j < Nm; ++j) A[i * NMAX + j] = make_double2(0, 0);
    if (fac.U) {
        const int64_t pp = (int64_t)i2 * g.n3 + i3;
        for (int d = 0; d < fac.D; ++d) {
            const double2 p = axis_ph(ph, d - fac.rc, a1, g.L);
            const double2 *u = fac.U + ((int64_t)d * fac.plane + pp) * MM;
#pragma unroll U
            for (int i = 0; i < Nm; ++i)
#pragma unroll U
                for (int j = i; j < Nm; ++j) A[i * NMAX + j] = cfma(p, u[i * Nm + j], A[i * NMAX + j]);
        }
    } else {
        for (int r = 0; r < nR; ++r) {
            const double2 p = ph[phase_index(a1, a2, a3, R[3 * r], R[3 * r + 1], R[3 * r + 2], g.L)];
            const double *f = Phiw + (size_t)r * MM;
#pragma unroll U
            for (int i = 0; i < Nm; ++i)
#pragma unroll U
                for (int j = i; j < Nm; ++j) {
                    A[i * NMAX + j].x = fma(p.x, f[i * Nm + j], A[i * NMAX + j].x);
                    A[i * NMAX + j].y = fma(p.y, f[i * Nm + j], A[i * NMAX + j].y);
                }
        }
    }
    double lam[NMAX];
    if (!eig_hermitian<NMAX>(A, E, Nm, lam)) atomicAdd(flag, im == iq ? 1 : 2);
    float wmax = -1.f;
#pragma unroll U
    for (int nu = 0; nu < Nm; ++nu) {
        const double l = lam[nu];
        const double w = (l >= 0 ? 1.0 : -1.0) * sqrt(fabs(l) * epc::kHbar2AmuA2);
        hw[iq * Nm + nu] = hw[im * Nm + nu] = w;
        const bool keep = w >= omega_min;
        hw32[iq * Nm + nu] = hw32[im * Nm + nu] = keep ? (float)w : -1.0f;
        if (keep) wmax = fmaxf(wmax, (float)w);
        double amp = 0, mass = -1;                // one root and division per atom
#pragma unroll U
        for (int m = 0; m < Nm; ++m) {
            if (mode_mass[m] != mass) {
                mass = mode_mass[m];
                amp = keep ? sqrt(epc::kHbar2AmuA2 / (2.0 * mass * w)) : 0.0;
            }
            const double2 v = make_double2(E[m * NMAX + nu].x * amp, E[m * NMAX + nu].y * amp);
            uout[iq * MM + m * Nm + nu] = v;
            u32[iq * MM + m * Nm + nu] = make_float2((float)v.x, (float)v.y);
            if (im != iq) {
                uout[im * MM + m * Nm + nu] = make_double2(v.x, -v.y);
                u32[im * MM + m * Nm + nu] = make_float2((float)v.x, -(float)v.y);
            }
        }
    }
    hwmax32[iq] = hwmax32[im] = wmax;
}

// Warp-per-matrix variants for large matrices (W >= 16, Nm >= 12): the matrix lives in
// shared memory (row stride n + 1), lane r builds row r of the Fourier sum, and the
// warp-parallel Jacobi diagonalises it.  Outputs are those of the one-thread kernels.
constexpr int kWarpsPerBlock = 4;

struct WarpScratch {
    double2 *A, *V;
    float2 *f;
    double *w;
    int *perm;
    JRot *rot;
};

__host__ __device__ inline size_t warp_scratch_per(int n) {
    const size_t per = (sizeof(double2) * 2 + sizeof(float2)) * n * (n + 1) + sizeof(double) * 32 + sizeof(int) * 32 +
                       sizeof(JRot) * 16;
    return (per + 15) & ~size_t(15);
}

__device__ inline WarpScratch warp_scratch(uint8_t *base, int n) {
    const int ld = n + 1;
    WarpScratch ws;
    ws.A = reinterpret_cast<double2 *>(base + (threadIdx.x >> 5) * warp_scratch_per(n));
    ws.V = ws.A + n * ld;
    ws.f = reinterpret_cast<float2 *>(ws.V + n * ld);
    ws.w = reinterpret_cast<double *>(ws.f + n * ld);
    ws.perm = reinterpret_cast<int *>(ws.w + 32);
    ws.rot = reinterpret_cast<JRot *>(ws.perm + 32);
    return ws;
}

size_t warp_scratch_bytes(int n) { return kWarpsPerBlock * warp_scratch_per(n); }

// FAC: H(k) and dH/dk from the factorised stages (as in k_eig_el), each lane building its row.
template <bool FAC>
__global__ void __launch_bounds__(32 * kWarpsPerBlock) k_eig_el_warp(
    GridInfo g, int64_t nk, int W, int nR, const int *__restrict__ R, const double *__restrict__ Rcart,
    const double2 *__restrict__ Hw, const double2 *__restrict__ ph, double *__restrict__ eps,
    float *__restrict__ eps32, double2 *__restrict__ Vout, float2 *__restrict__ V32,
    double *__restrict__ vel, int *__restrict__ flag, FacDesc fac, Lattice lat) {
    extern __shared__ __align__(16) uint8_t wsm[];
    const int lane = threadIdx.x & 31;
    const int64_t ik = (int64_t)blockIdx.x * kWarpsPerBlock + (threadIdx.x >> 5);
    if (ik >= nk) return;                      // whole warps leave together
    WarpScratch S = warp_scratch(wsm, W);
    const int ld = W + 1;
    int i1, i2, i3;
    grid_coords(g, ik, i1, i2, i3);
    const int a1 = (int)((int64_t)i1 * g.s1 % g.L), a2 = (int)((int64_t)i2 * g.s2 % g.L),
              a3 = (int)((int64_t)i3 * g.s3 % g.L);
    const int64_t WW = (int64_t)W * W;
    const int64_t pp = (int64_t)i2 * g.n3 + i3;   // (k2, k3) of this point (factorised build)
    if (lane < W) {
        for (int j = 0; j < W; ++j) S.A[lane * ld + j] = make_double2(0, 0);
        if constexpr (FAC) {
            for (int j1 = 0; j1 < fac.D; ++j1) {
                const double2 p = axis_ph(ph, j1 - fac.rc, a1, g.L);
                const double2 *u = fac.U + ((int64_t)j1 * fac.plane + pp) * WW + lane * W;
                for (int j = 0; j < W; ++j) S.A[lane * ld + j] = cfma(p, u[j], S.A[lane * ld + j]);
            }
        } else {
            for (int r = 0; r < nR; ++r) {
                const double2 p = ph[phase_index(a1, a2, a3, R[3 * r], R[3 * r + 1], R[3 * r + 2], g.L)];
                const double2 *h = Hw + (size_t)r * W * W + lane * W;
                for (int j = 0; j < W; ++j) S.A[lane * ld + j] = cfma(p, h[j], S.A[lane * ld + j]);
            }
        }
    }
    __syncwarp();
    const int ok = eig_hermitian_warp(S.A, S.V, S.f, W, ld, S.w, S.rot, S.perm);
    if (lane == 0 && !ok) atomicAdd(flag, 1);
    if (lane < W) {
        eps[ik * W + lane] = S.w[lane];
        eps32[ik * W + lane] = (float)S.w[lane];
        for (int n = 0; n < W; ++n) {
            const double2 v = S.V[lane * ld + n];
            Vout[ik * W * W + lane * W + n] = v;
            V32[ik * W * W + lane * W + n] = make_float2((float)v.x, (float)v.y);
        }
    }
    // v_n,a = (1/hbar) Re[V^dag (sum_R w_R i R_a e^{ik.R} H(R)) V]_nn, one axis at a time;
    // the derivative matrix reuses A (lane = row), then lane n contracts column n
    for (int ax = 0; ax < 3; ++ax) {
        __syncwarp();
        if (lane < W) {
            for (int j = 0; j < W; ++j) S.A[lane * ld + j] = make_double2(0, 0);
            if constexpr (FAC) {
                // i R_a = i (n1 A_1a + n2 A_2a + n3 A_3a): U_0 weighted by n1, U_1 (n2 sums), U_2 (n3 sums)
                const int64_t src = (int64_t)fac.D * fac.plane * WW;
                for (int j1 = 0; j1 < fac.D; ++j1) {
                    const int n1 = j1 - fac.rc;
                    const double2 p = axis_ph(ph, n1, a1, g.L);
                    const double2 ip = make_double2(-p.y, p.x);   // i e1
                    const double c0 = n1 * lat.a[0][ax], c1 = lat.a[1][ax], c2 = lat.a[2][ax];
                    const double2 *u = fac.U + ((int64_t)j1 * fac.plane + pp) * WW + lane * W;
                    for (int j = 0; j < W; ++j) {
                        const double2 sr = make_double2(c0 * u[j].x + c1 * u[src + j].x + c2 * u[2 * src + j].x,
                                                        c0 * u[j].y + c1 * u[src + j].y + c2 * u[2 * src + j].y);
                        S.A[lane * ld + j] = cfma(ip, sr, S.A[lane * ld + j]);
                    }
                }
            } else {
                for (int r = 0; r < nR; ++r) {
                    const double2 p = ph[phase_index(a1, a2, a3, R[3 * r], R[3 * r + 1], R[3 * r + 2], g.L)];
                    const double ra = Rcart[3 * r + ax];
                    const double2 ip = make_double2(-ra * p.y, ra * p.x);
                    const double2 *h = Hw + (size_t)r * W * W + lane * W;
                    for (int j = 0; j < W; ++j) S.A[lane * ld + j] = cfma(ip, h[j], S.A[lane * ld + j]);
                }
            }
        }
        __syncwarp();
        if (lane < W) {
            const int n = lane;
            double acc = 0;
            for (int i = 0; i < W; ++i) {
                double2 t = make_double2(0, 0);
                for (int j = 0; j < W; ++j) t = cfma(S.A[i * ld + j], S.V[j * ld + n], t);
                acc += S.V[i * ld + n].x * t.x + S.V[i * ld + n].y * t.y;
            }
            vel[(ik * W + n) * 3 + ax] = acc / epc::kHbarEVs * 1e-10;
        }
    }
}

template <bool FAC>
__global__ void __launch_bounds__(32 * kWarpsPerBlock) k_eig_ph_warp(
    GridInfo g, int64_t nq, int Nm, int nR, const int *__restrict__ R, const double *__restrict__ Phiw,
    const double *__restrict__ mode_mass, const double2 *__restrict__ ph, double omega_min,
    double *__restrict__ hw, float *__restrict__ hwmax32, float *__restrict__ hw32,
    double2 *__restrict__ uout, float2 *__restrict__ u32, int *__restrict__ flag, FacDesc fac) {
    extern __shared__ __align__(16) uint8_t wsm[];
    const int lane = threadIdx.x & 31;
    const int64_t iq = (int64_t)blockIdx.x * kWarpsPerBlock + (threadIdx.x >> 5);
    if (iq >= nq) return;
    int i1, i2, i3;
    grid_coords(g, iq, i1, i2, i3);
    const int64_t im = minus_q(g, i1, i2, i3);
    if (im < iq) return;                       // solved by that point's warp
    WarpScratch S = warp_scratch(wsm, Nm);
    const int ld = Nm + 1;
    const int a1 = (int)((int64_t)i1 * g.s1 % g.L), a2 = (int)((int64_t)i2 * g.s2 % g.L),
              a3 = (int)((int64_t)i3 * g.s3 % g.L);
    if (lane < Nm) {
        for (int j = 0; j < Nm; ++j) S.A[lane * ld + j] = make_double2(0, 0);
        if constexpr (FAC) {
            const int64_t pp = (int64_t)i2 * g.n3 + i3;
            for (int j1 = 0; j1 < fac.D; ++j1) {
                const double2 p = axis_ph(ph, j1 - fac.rc, a1, g.L);
                const double2 *u = fac.U + ((int64_t)j1 * fac.plane + pp) * Nm * Nm + lane * Nm;
                for (int j = 0; j < Nm; ++j) S.A[lane * ld + j] = cfma(p, u[j], S.A[lane * ld + j]);
            }
        } else {
            for (int r = 0; r < nR; ++r) {
                const double2 p = ph[phase_index(a1, a2, a3, R[3 * r], R[3 * r + 1], R[3 * r + 2], g.L)];
                const double *f = Phiw + (size_t)r * Nm * Nm + lane * Nm;
                for (int j = 0; j < Nm; ++j) {
                    S.A[lane * ld + j].x = fma(p.x, f[j], S.A[lane * ld + j].x);
                    S.A[lane * ld + j].y = fma(p.y, f[j], S.A[lane * ld + j].y);
                }
            }
        }
    }
    __syncwarp();
    const int ok = eig_hermitian_warp(S.A, S.V, S.f, Nm, ld, S.w, S.rot, S.perm);
    if (lane == 0 && !ok) atomicAdd(flag, im == iq ? 1 : 2);
    // lane = mode nu
    float wmax = -1.f;
    if (lane < Nm) {
        const int nu = lane;
        const double l = S.w[nu];
        const double w = (l >= 0 ? 1.0 : -1.0) * sqrt(fabs(l) * epc::kHbar2AmuA2);
        hw[iq * Nm + nu] = hw[im * Nm + nu] = w;
        const bool keep = w >= omega_min;
        hw32[iq * Nm + nu] = hw32[im * Nm + nu] = keep ? (float)w : -1.0f;
        if (keep) wmax = (float)w;
        for (int m = 0; m < Nm; ++m) {
            const double amp = keep ? sqrt(epc::kHbar2AmuA2 / (2.0 * mode_mass[m] * w)) : 0.0;
            const double2 e = S.V[m * ld + nu];
            const double2 v = make_double2(e.x * amp, e.y * amp);
            uout[iq * Nm * Nm + m * Nm + nu] = v;
            u32[iq * Nm * Nm + m * Nm + nu] = make_float2((float)v.x, (float)v.y);
            if (im != iq) {
                uout[im * Nm * Nm + m * Nm + nu] = make_double2(v.x, -v.y);
                u32[im * Nm * Nm + m * Nm + nu] = make_float2((float)v.x, -(float)v.y);
            }
        }
    }
    for (int o = 16; o > 0; o >>= 1) wmax = fmaxf(wmax, __shfl_xor_sync(0xffffffffu, wmax, o));
    if (lane == 0) hwmax32[iq] = hwmax32[im] = wmax;
}

}  // namespace

GridInfo make_grid_info(const epwi_ctx *c) {
    GridInfo g;
    g.n1 = c->ng[0];
    g.n2 = c->ng[1];
    g.n3 = c->ng[2];
    g.L = c->L;
    g.s1 = c->L / c->ng[0];
    g.s2 = c->L / c->ng[1];
    g.s3 = c->L / c->ng[2];
    return g;
}

void launch_phase_tables(epwi_ctx *c) {
    c->ph64.ensure(sizeof(double2) * c->L);
    c->ph32.ensure(sizeof(float2) * c->L);
    k_phase_tables<<<(c->L + 127) / 128, 128, 0, c->stream>>>(c->L, c->ph64.as<double2>(),
                                                               c->ph32.as<float2>());
    EPWI_CHECK_LAUNCH();
}

// Threads per block of the thread-per-point kernels: an SM's FP64 unit takes 16 clocks per warp
// instruction, so a grid's points are spread over all SMs first (32-thread blocks up to 128 points
// per SM, 64 up to 256).
static int eig_block(const epwi_ctx *c, int64_t nk) {
    return nk <= c->sm_count * int64_t(128) ? 32 : nk <= c->sm_count * int64_t(256) ? 64 : 128;
}

// Velocities of the n listed points (NULL: all) from the electron stage output f.
static void launch_vel(epwi_ctx *c, const FacDesc &f, const Lattice &lat, const int *list, int64_t n) {
    if (n <= 0) return;
    const int W = c->nw;
    const GridInfo g = make_grid_info(c);
    const unsigned nb = (unsigned)((n + 31) / 32);
#define VEL_ARGS g, n, W, list, c->ph64.as<double2>(), c->V.as<double2>(), c->vel.as<double>(), f, lat
    if (W == 1) k_vel_fac<1, true><<<nb, 96, 0, c->stream>>>(VEL_ARGS);
    else if (W == 4) k_vel_fac<4, true><<<nb, 96, 0, c->stream>>>(VEL_ARGS);
    else if (W < 4) k_vel_fac<4, false><<<nb, 96, 0, c->stream>>>(VEL_ARGS);
    else if (W == 8) k_vel_fac<8, true><<<nb, 96, 0, c->stream>>>(VEL_ARGS);
    else k_vel_fac<8, false><<<nb, 96, 0, c->stream>>>(VEL_ARGS);
#undef VEL_ARGS
    EPWI_CHECK_LAUNCH();
}

void reserve_phonon_stages(epwi_ctx *c) {
    if (c->fac_rp_r < 0) return;
    const int64_t D = 2 * c->fac_rp_r + 1, E = (int64_t)c->nm * c->nm, n2 = c->ng[1], n3 = c->ng[2];
    c->fac_Tp.ensure(sizeof(double2) * D * D * n3 * E);
    c->fac_Up.ensure(sizeof(double2) * D * n2 * n3 * E);
}

void launch_eigs(epwi_ctx *c, cudaStream_t ph, cudaEvent_t fork, cudaEvent_t join) {
    const int64_t nk = c->nk;
    const int W = c->nw, Nm = c->nm;
    c->eps.ensure(sizeof(double) * nk * W);
    c->eps32.ensure(sizeof(float) * nk * W);
    c->V.ensure(sizeof(double2) * nk * W * W);
    c->V32.ensure(sizeof(float2) * nk * W * W);
    c->vel.ensure(sizeof(double) * nk * W * 3);
    c->hw.ensure(sizeof(double) * nk * Nm);
    c->hwmax32.ensure(sizeof(float) * nk);
    c->hw32.ensure(sizeof(float) * nk * Nm);
    c->u.ensure(sizeof(double2) * nk * Nm * Nm);
    c->u32.ensure(sizeof(float2) * nk * Nm * Nm);
    c->eig_flag.ensure(sizeof(int) * 2);
    EPWI_CUDA(cudaMemsetAsync(c->eig_flag.p, 0, sizeof(int) * 2, c->stream));
    const bool own = ph != nullptr;               // phonons on their own stream, with their own stage buffers
    if (own) {
        reserve_phonon_stages(c);
        EPWI_CUDA(cudaEventRecord(fork, c->stream));
        EPWI_CUDA(cudaStreamWaitEvent(ph, fork, 0));
    } else {
        ph = c->stream;
    }
    GridInfo g = make_grid_info(c);
    const int bs = eig_block(c, nk);
    const unsigned nb = (unsigned)((nk + bs - 1) / bs);
    const int64_t plane = (int64_t)g.n2 * g.n3;
    // factorised build: axis-3 and axis-2 stages into fac_U (sources 0..nsrc-1), axis 1 in the
    // eigensolve kernel
    auto fac_sizes = [&](int rc, int E, bool vel, int64_t &nT, int64_t &nU) {
        const int D = 2 * rc + 1;
        nT = (int64_t)(vel ? 2 : 1) * D * D * g.n3 * E;
        nU = (int64_t)(vel ? 3 : 1) * D * plane * E;
    };
    auto fac_stages = [&](const DevBuf &Xc, int rc, int E, bool vel, DevBuf &T, DevBuf &Uout, cudaStream_t st) {
        const int D = 2 * rc + 1;
        const int64_t t3 = (int64_t)D * D * g.n3 * E, t2 = (int64_t)D * plane * E;
        if (vel) {
            k_fac_axis3<true><<<(unsigned)((t3 + 255) / 256), 256, 0, st>>>(
                D, rc, g.n3, g.s3, g.L, E, Xc.as<double2>(), c->ph64.as<double2>(), T.as<double2>());
            EPWI_CHECK_LAUNCH();
            k_fac_axis2<true><<<(unsigned)((t2 + 255) / 256), 256, 0, st>>>(
                D, rc, g.n2, g.n3, g.s2, g.L, E, T.as<double2>(), c->ph64.as<double2>(), Uout.as<double2>());
        } else {
            k_fac_axis3<false><<<(unsigned)((t3 + 255) / 256), 256, 0, st>>>(
                D, rc, g.n3, g.s3, g.L, E, Xc.as<double2>(), c->ph64.as<double2>(), T.as<double2>());
            EPWI_CHECK_LAUNCH();
            k_fac_axis2<false><<<(unsigned)((t2 + 255) / 256), 256, 0, st>>>(
                D, rc, g.n2, g.n3, g.s2, g.L, E, T.as<double2>(), c->ph64.as<double2>(), Uout.as<double2>());
        }
        EPWI_CHECK_LAUNCH();
        FacDesc f;
        f.U = Uout.as<double2>();
        f.D = D;
        f.rc = rc;
        f.plane = plane;
        return f;
    };
    Lattice lat;
    for (int i = 0; i < 9; ++i) lat.a[i / 3][i % 3] = c->lattice[i];
    const bool fac_el = c->fac_re_r >= 0, fac_ph = c->fac_rp_r >= 0;
    {
        // on one stream both builds share the stage buffers: size them once, before any launch
        int64_t nT = 1, nU = 1, t, u;
        if (fac_el) {
            fac_sizes(c->fac_re_r, W * W, true, t, u);
            nT = std::max(nT, t);
            nU = std::max(nU, u);
        }
        if (fac_ph) {
            fac_sizes(c->fac_rp_r, Nm * Nm, false, t, u);
            if (!own) {
                nT = std::max(nT, t);
                nU = std::max(nU, u);
            }
        }
        if (fac_el || fac_ph) {
            c->fac_T.ensure(sizeof(double2) * nT);
            c->fac_U.ensure(sizeof(double2) * nU);
        }
    }
    // deferred velocities (thread-per-point solver with the factorised build): the electron
    // stage output stays in fac_Uel for ensure_velocities
    const bool defer = c->vel_defer && fac_el && W <= 8;
    if (defer) {
        int64_t t, u;
        fac_sizes(c->fac_re_r, W * W, true, t, u);
        c->fac_Uel.ensure(sizeof(double2) * u);
    }
    FacDesc fe{}, fp{};
    if (fac_el) fe = fac_stages(c->fac_Hc, c->fac_re_r, W * W, true, c->fac_T, defer ? c->fac_Uel : c->fac_U, c->stream);
    c->vel_state = defer ? 0 : 2;
#define EL_ARGS                                                                              \
    g, nk, W, c->nRe, c->Re.as<int>(), c->Rcart.as<double>(), c->Hw.as<double2>(),            \
        c->ph64.as<double2>(), c->eps.as<double>(), c->eps32.as<float>(), c->V.as<double2>(), \
        c->V32.as<float2>(), c->vel.as<double>(), c->eig_flag.as<int>()
    const unsigned nbw = (unsigned)((nk + kWarpsPerBlock - 1) / kWarpsPerBlock);
#define EL_LAUNCH(N, FIXED)                                                                  \
    do {                                                                                     \
        k_eig_el<N, FIXED><<<nb, bs, 0, c->stream>>>(EL_ARGS, fe, lat, fac_el ? 0 : 1);      \
    } while (0)
    if (W == 1) {
        EL_LAUNCH(1, true);
    } else if (W == 4) {
        EL_LAUNCH(4, true);
    } else if (W < 4) {
        EL_LAUNCH(4, false);
    } else if (W == 8) {
        EL_LAUNCH(8, true);
    } else if (W < 8) {
        EL_LAUNCH(8, false);
    } else {
        const size_t sm = warp_scratch_bytes(W);
        if (fac_el) {
            allow_smem(k_eig_el_warp<true>);
            k_eig_el_warp<true><<<nbw, 32 * kWarpsPerBlock, sm, c->stream>>>(EL_ARGS, fe, lat);
        } else {
            allow_smem(k_eig_el_warp<false>);
            k_eig_el_warp<false><<<nbw, 32 * kWarpsPerBlock, sm, c->stream>>>(EL_ARGS, fe, lat);
        }
    }
#undef EL_LAUNCH
#undef EL_ARGS
    EPWI_CHECK_LAUNCH();
    if (fac_el && W <= 8 && !defer) launch_vel(c, fe, lat, nullptr, nk);   // before the phonon stages reuse fac_U
    const int64_t nh = (g.n1 / 2 + 1) * plane;    // see minus_q
    const int bsh = eig_block(c, nh);
    const unsigned nbh = (unsigned)((nh + bsh - 1) / bsh), nbhw = (unsigned)((nh + kWarpsPerBlock - 1) / kWarpsPerBlock);
#define PH_ARGS                                                                             \
    g, nh, Nm, c->nRp, c->Rp.as<int>(), c->Phiw.as<double>(), c->mode_mass.as<double>(),     \
        c->ph64.as<double2>(), c->opt.omega_min_eV, c->hw.as<double>(), c->hwmax32.as<float>(), \
        c->hw32.as<float>(),                                                                   \
        c->u.as<double2>(), c->u32.as<float2>(), c->eig_flag.as<int>() + 1
    // on one stream the electron kernel above has read fac_U: the phonon stages reuse the buffers
    if (fac_ph)
        fp = fac_stages(c->fac_Pc, c->fac_rp_r, Nm * Nm, false, own ? c->fac_Tp : c->fac_T, own ? c->fac_Up : c->fac_U, ph);
    if (Nm == 3) {
        k_eig_ph<3, true><<<nbh, bsh, 0, ph>>>(PH_ARGS, fp);
    } else if (Nm == 6) {
        k_eig_ph<6, true><<<nbh, bsh, 0, ph>>>(PH_ARGS, fp);
    } else {
        const size_t sm = warp_scratch_bytes(Nm);
        if (fac_ph) {
            allow_smem(k_eig_ph_warp<true>);
            k_eig_ph_warp<true><<<nbhw, 32 * kWarpsPerBlock, sm, ph>>>(PH_ARGS, fp);
        } else {
            allow_smem(k_eig_ph_warp<false>);
            k_eig_ph_warp<false><<<nbhw, 32 * kWarpsPerBlock, sm, ph>>>(PH_ARGS, fp);
        }
    }
#undef PH_ARGS
    EPWI_CHECK_LAUNCH();
    if (own) {
        EPWI_CUDA(cudaEventRecord(join, ph));
        EPWI_CUDA(cudaStreamWaitEvent(c->stream, join, 0));
    }
}

void ensure_velocities(epwi_ctx *c, bool all) {
    if (c->vel_state == 2 || (!all && c->vel_state == 1)) return;
    GridInfo g = make_grid_info(c);
    FacDesc f;
    f.U = c->fac_Uel.as<double2>();
    f.rc = c->fac_re_r;
    f.D = 2 * f.rc + 1;
    f.plane = (int64_t)g.n2 * g.n3;
    Lattice lat;
    for (int i = 0; i < 9; ++i) lat.a[i / 3][i % 3] = c->lattice[i];
    // the window's k-points (build_window), or every grid point
    launch_vel(c, f, lat, all ? nullptr : c->kpts.as<int>(), all ? c->nk : c->nkp);
    c->vel_state = all ? 2 : 1;
}
