// Inference of the q-proposal network on the tensor cores (tcgen05).
//
// One CTA per SM, four groups of 128 threads; each group takes 128-row tiles of its own
// (persistent), thread r owning row r of the tile and TMEM lane r:
//   layer 1 (K = 9) on the CUDA cores in FP32: h1 = silu(W1 x + b1), rounded to BF16 and
//           written to shared memory as the A operand;
//   layer 2 h2 = silu(W2 h1 + b2): eight tcgen05.mma kind::f16 (BF16, M = N = 128, K = 16
//           each) with the FP32 accumulator in TMEM, read back by tcgen05.ld, bias and SiLU
//           in FP32, rounded to BF16 into the same A buffer;
//   layer 3 the same with W3, then y = w4 . silu(W3 h2 + b3) + b4 in FP32.
// The 384 SiLUs of a row (an exponential and a reciprocal each: 48 clocks of an SM's special-
// function units) and the FP32 arithmetic around them bound the kernel; the matrix products take
// a tenth of it.  Four groups share one copy of the weights (64 KB of W2 and W3), so that 16
// warps keep those units busy while others wait for their MMA or their barrier; a CTA with its
// own weights per tile left room for two tiles per SM.  Measured on one GB300, 3.0e7 proposal rows:
// 8.2 ms for the network and 6.8 ms for its input rows before, 7.1 ms together with tables and sums
// now.  The groups meet at named barriers of
// their own only.
// Operands use the no-swizzle K-major canonical layout (core matrices of 8 rows x 16 bytes;
// LBO = 128 bytes between core matrices along K, SBO = 2048 bytes between 8-row groups for
// K = 128).  Every mbarrier wait is bounded; on a timeout the group records the error and stops,
// and the CTA frees its TMEM when every group is done.
//
// The rows come from memory (k_mlp_infer_tc<false>) or are the proposal's rows of a chunk of
// states (true): the inputs of (state, cell, mode) are put together from tables of the grid's
// coordinates, the states and the modes, so that no row passes through memory.
#include <cuda_bf16.h>

#include <algorithm>

#include "mlp.cuh"
#include "tc_ptx.cuh"

namespace {
using namespace mlp;

constexpr int kRows = 128;
constexpr uint32_t kTileBytes = 128 * 128 * 2;      // one 128 x 128 BF16 operand
constexpr uint64_t kWaitNs = 2000000000ull;          // 2 s

__device__ __forceinline__ uint32_t cm_offset(int row, int k) {   // bytes, K = 128 BF16
    return (uint32_t)(((row >> 3) * 16 + (k >> 3)) * 128 + (row & 7) * 16 + (k & 7) * 2);
}

__device__ __forceinline__ float silu_fast(float z) { return __fdividef(z, 1.0f + __expf(-z)); }

__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const uint32_t *>(&v);
}

constexpr int kGroups = 4;                           // 128-thread groups (tiles in flight) per CTA
constexpr int kW1Row = 12;                           // floats per neuron of layer 1: 9 weights, bias, pad

struct MlpTcArgs {
    int64_t n;                   // rows
    const float *X;              // [n][9] (rows from memory)
    float *y;                    // [n]
    const uint16_t *wbf;         // BF16 parameters (storage order of mlp.cuh)
    const float *w;              // the same values as FP32 (biases, W1, w4)
    int *err;
    PropRows pr;                 // proposal rows
};

__device__ __forceinline__ void group_barrier(int g) {
    asm volatile("bar.sync %0, 128;" ::"r"(g + 1) : "memory");
}

template <bool PROP>
__global__ void __launch_bounds__(kRows * kGroups, 1) k_mlp_infer_tc(MlpTcArgs a) {
    extern __shared__ __align__(1024) uint8_t smem[];
    uint8_t *sW2 = smem;
    uint8_t *sW3 = smem + kTileBytes;
    const int grp = threadIdx.x / kRows, tid = threadIdx.x % kRows, warp = tid >> 5;
    uint8_t *sA = smem + (2 + grp) * kTileBytes;
    float *sW1 = reinterpret_cast<float *>(smem + (2 + kGroups) * kTileBytes);     // [128][kW1Row]
    float *sB2 = sW1 + kHid * kW1Row, *sB3 = sB2 + kHid, *sW4 = sB3 + kHid;
    uint64_t *bars = reinterpret_cast<uint64_t *>(sW4 + kHid);
    uint32_t *tslot = reinterpret_cast<uint32_t *>(bars + kGroups);
    volatile int *sfail = reinterpret_cast<volatile int *>(tslot + 1) + grp;
    uint64_t *bar = bars + grp;

    // weights into shared memory: W2, W3 as canonical BF16 tiles; the rest in FP32
    for (int e = threadIdx.x; e < kHid * kHid / 8; e += kRows * kGroups) {
        const int n = e / (kHid / 8), k8 = (e % (kHid / 8)) * 8;
        const uint4 v2 = *reinterpret_cast<const uint4 *>(a.wbf + oW2 + n * kHid + k8);
        const uint4 v3 = *reinterpret_cast<const uint4 *>(a.wbf + oW3 + n * kHid + k8);
        *reinterpret_cast<uint4 *>(sW2 + cm_offset(n, k8)) = v2;
        *reinterpret_cast<uint4 *>(sW3 + cm_offset(n, k8)) = v3;
    }
    for (int e = threadIdx.x; e < kHid * kW1Row; e += kRows * kGroups) {
        const int n = e / kW1Row, f = e % kW1Row;
        sW1[e] = f < kIn ? a.w[oW1 + n * kIn + f] : f == kIn ? a.w[ob1 + n] : 0.f;
    }
    for (int e = threadIdx.x; e < kHid; e += kRows * kGroups) {
        sB2[e] = a.w[ob2 + e];
        sB3[e] = a.w[ob3 + e];
        sW4[e] = a.w[ow4 + e];
    }
    const float b4 = a.w[ob4];
    if (tid == 0) {
        tc::mbar_init(bar, 1);
        *sfail = 0;
        tc::fence_mbar_init();
    }
    if (threadIdx.x < 32) {
        tc::tmem_alloc(tslot, 128 * kGroups);
        tc::tmem_relinquish();
    }
    tc::fence_proxy_async_smem();
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    const uint32_t tbase = *tslot;
    const uint32_t tmem = tbase + 128u * grp;                        // this group's accumulator columns
    const uint32_t trow = tmem + ((uint32_t)(warp * 32) << 16);
    const uint32_t idesc = tc::idesc(1, 128, 128, false);            // BF16 x BF16 -> FP32
    const uint32_t aA = tc::smem_u32(sA), aW2 = tc::smem_u32(sW2), aW3 = tc::smem_u32(sW3);
    uint32_t phase = 0;
    bool failed = false;
    const int64_t ntiles = (a.n + kRows - 1) / kRows;

    auto layer_mma = [&](uint32_t aB) -> bool {
        // all threads of the group: the A buffer is written and visible to the tensor core
        tc::fence_proxy_async_smem();
        tc::tc_fence_before();
        group_barrier(grp);
        if (tid == 0) {
            tc::tc_fence_after();
#pragma unroll
            for (int ks = 0; ks < kHid / 16; ++ks)
                tc::mma<false>(tmem, tc::sdesc(aA + ks * 256, 128, 2048),
                               tc::sdesc(aB + ks * 256, 128, 2048), idesc, ks > 0 ? 1u : 0u);
            tc::mma_commit(bar);
        }
        const bool ok = tc::mbar_wait_bounded(bar, phase, kWaitNs);
        phase ^= 1;
        tc::tc_fence_after();
        return ok;
    };

    for (int64_t t = blockIdx.x + (int64_t)grp * gridDim.x; t < ntiles && !failed; t += (int64_t)gridDim.x * kGroups) {
        const int64_t row = t * kRows + tid;
        // ---- layer 1 on the CUDA cores
        float x[kIn];
        if constexpr (PROP) {
            const uint32_t r = (uint32_t)min(row, a.n - 1);          // n < 2^31
            const uint32_t sc = r / (uint32_t)a.pr.Nm, nu = r - sc * a.pr.Nm;
            const uint32_t st = sc / (uint32_t)a.pr.ncell, cell = a.pr.cell0 + (sc - st * a.pr.ncell);
            const uint32_t c12 = cell / (uint32_t)a.pr.c3, c3 = cell - c12 * a.pr.c3;
            const uint32_t c1 = c12 / (uint32_t)a.pr.c2, c2 = c12 - c1 * a.pr.c2;
            const float *fs = a.pr.state + (size_t)st * 5, *ft = a.pr.tab;
            x[0] = fs[0];
            x[1] = fs[1];
            x[2] = fs[2];
            x[3] = ft[c1];
            x[4] = ft[a.pr.c1 + c2];
            x[5] = ft[a.pr.c1 + a.pr.c2 + c3];
            x[6] = fs[3];
            x[7] = fs[4];
            x[8] = ft[a.pr.c1 + a.pr.c2 + a.pr.c3 + nu];
        } else {
#pragma unroll
            for (int f = 0; f < kIn; ++f) x[f] = row < a.n ? a.X[row * kIn + f] : 0.f;
        }
#pragma unroll 1
        for (int k8 = 0; k8 < kHid; k8 += 8) {
            float h[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const float4 *wr = reinterpret_cast<const float4 *>(sW1 + (k8 + j) * kW1Row);
                const float4 w0 = wr[0], w1 = wr[1], w2 = wr[2];
                float z = w2.y;
                z = fmaf(w0.x, x[0], z);
                z = fmaf(w0.y, x[1], z);
                z = fmaf(w0.z, x[2], z);
                z = fmaf(w0.w, x[3], z);
                z = fmaf(w1.x, x[4], z);
                z = fmaf(w1.y, x[5], z);
                z = fmaf(w1.z, x[6], z);
                z = fmaf(w1.w, x[7], z);
                z = fmaf(w2.x, x[8], z);
                h[j] = silu_fast(z);
            }
            *reinterpret_cast<uint4 *>(sA + cm_offset(tid, k8)) =
                make_uint4(pack_bf16(h[0], h[1]), pack_bf16(h[2], h[3]), pack_bf16(h[4], h[5]),
                           pack_bf16(h[6], h[7]));
        }
        // ---- layers 2 and 3 on the tensor cores
        float out = b4;
        for (int layer = 0; layer < 2 && !failed; ++layer) {
            if (!layer_mma(layer == 0 ? aW2 : aW3)) *sfail = 1;
            group_barrier(grp);
            if (*sfail) {
                failed = true;
                break;
            }
            const float *bias = layer == 0 ? sB2 : sB3;
#pragma unroll 1
            for (int c0 = 0; c0 < kHid; c0 += 16) {
                float v[16];
                tc::tmem_ld16(trow + (uint32_t)c0, v);
                tc::tmem_wait_ld();
#pragma unroll
                for (int j = 0; j < 16; j += 4) {
                    const float4 b = *reinterpret_cast<const float4 *>(bias + c0 + j);
                    v[j] = silu_fast(v[j] + b.x);
                    v[j + 1] = silu_fast(v[j + 1] + b.y);
                    v[j + 2] = silu_fast(v[j + 2] + b.z);
                    v[j + 3] = silu_fast(v[j + 3] + b.w);
                }
                if (layer == 0) {
                    *reinterpret_cast<uint4 *>(sA + cm_offset(tid, c0)) =
                        make_uint4(pack_bf16(v[0], v[1]), pack_bf16(v[2], v[3]), pack_bf16(v[4], v[5]),
                                   pack_bf16(v[6], v[7]));
                    *reinterpret_cast<uint4 *>(sA + cm_offset(tid, c0 + 8)) =
                        make_uint4(pack_bf16(v[8], v[9]), pack_bf16(v[10], v[11]),
                                   pack_bf16(v[12], v[13]), pack_bf16(v[14], v[15]));
                } else {
#pragma unroll
                    for (int j = 0; j < 16; j += 4) {
                        const float4 w = *reinterpret_cast<const float4 *>(sW4 + c0 + j);
                        out = fmaf(w.x, v[j], out);
                        out = fmaf(w.y, v[j + 1], out);
                        out = fmaf(w.z, v[j + 2], out);
                        out = fmaf(w.w, v[j + 3], out);
                    }
                }
            }
            // the accumulator is read: the next MMA may overwrite it
            tc::tc_fence_before();
        }
        if (!failed && row < a.n) a.y[row] = out;
        group_barrier(grp);
    }
    if (failed) {
        // let the MMA whose wait gave up finish before the TMEM is released (its parity is
        // the one before the flip in layer_mma)
        tc::mbar_wait_bounded(bar, phase ^ 1u, kWaitNs);
        if (tid == 0) atomicAdd(a.err, 1);
    }
    tc::tc_fence_before();
    __syncthreads();
    if (threadIdx.x < 32) tc::tmem_dealloc(tbase, 128 * kGroups);
}

size_t infer_smem() {
    return (2 + kGroups) * (size_t)kTileBytes + sizeof(float) * (kHid * kW1Row + 3 * kHid) + 64;
}

template <bool PROP>
void launch_infer(epwi_ctx *c, const MlpTcArgs &a) {
    const size_t sm = infer_smem();
    allow_smem(k_mlp_infer_tc<PROP>);
    int nsm = 0;
    EPWI_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, c->device));
    // one CTA per SM; few tiles spread over the SMs first
    const int64_t ntiles = (a.n + kRows - 1) / kRows;
    const int grid = (int)std::min<int64_t>(ntiles, nsm);
    k_mlp_infer_tc<PROP><<<grid, kRows * kGroups, sm, c->stream>>>(a);
    EPWI_CHECK_LAUNCH();
}

}  // namespace

// y[n] = network(X[n][9]) on the tensor cores (BF16 activations between layers).  err_dev counts
// the groups that timed out.
void mlp_forward_tc(epwi_ctx *c, int64_t n, const float *X, float *y, int *err_dev) {
    if (n <= 0) return;
    MlpState &m = *c->mlp;
    launch_infer<false>(c, MlpTcArgs{n, X, y, m.wbf.as<uint16_t>(), m.w.as<float>(), err_dev, PropRows{}});
}

void mlp_proposal_tc(epwi_ctx *c, int64_t n, const PropRows &pr, float *y, int *err_dev) {
    if (n <= 0) return;
    MlpState &m = *c->mlp;
    launch_infer<true>(c, MlpTcArgs{n, nullptr, y, m.wbf.as<uint16_t>(), m.w.as<float>(), err_dev, pr});
}
