// Pieces the layer-by-layer FP32 gradients of the chain models share: the
// input code of a site and the two-way readout with its adjoint.
#pragma once

#include <cuda_runtime.h>

#include "psr_device.cuh"

namespace psr {

// input code of site t: 0 at the first site, 1 + s_{t-1} otherwise
__device__ __forceinline__ int code_at(const uint64_t *row, int t) {
    return t == 0 ? 0 : 1 + (int)((row[(t - 1) >> 6] >> ((t - 1) & 63)) & 1ull);
}

struct ReadoutArgs {
    int n, N, H, W, u1;
    const uint64_t *bits;
    const float *x;      // [n N][H] input of the readout
    const float *wd, *bd;  // logit-difference weights [H] and bias
    const float *dout;   // [n] weights or null
    float *g;            // [n N]
    float *wo, *bo;      // [2][H], [2] of sample 0, small_stride apart
    int64_t small_stride;
};

// Readout adjoint g_t = 1/2 (s_t - P(1 | s_<t)) dout and, through `top`, the
// adjoint of x: top.store(index, g wd, top.load(index)).  One warp per kSites
// sites, E = H / 32 units a lane; all the sites' rows are in flight together
// (bound by the arrays' bytes).
template <int E, class Top>
__global__ void __launch_bounds__(256) grad_readout_kernel(const __grid_constant__ ReadoutArgs A,
                                                           const __grid_constant__ Top top) {
    constexpr int kSites = 4;
    const int lane = threadIdx.x & 31;
    const int M = A.n * A.N, m0 = (int)(blockIdx.x * 8 + (threadIdx.x >> 5)) * kSites;
    if (m0 >= M) return;
    constexpr int H = 32 * E;
    float wd[E], x[kSites][E], d[kSites];
    typename Top::In in[kSites][E];
#pragma unroll
    for (int e = 0; e < E; ++e) wd[e] = A.wd[32 * e + lane];
#pragma unroll
    for (int i = 0; i < kSites; ++i) {
        const float *p = A.x + (size_t)min(m0 + i, M - 1) * H + lane;
#pragma unroll
        for (int e = 0; e < E; ++e) {
            x[i][e] = p[32 * e];
            in[i][e] = top.load((size_t)min(m0 + i, M - 1) * H + 32 * e + lane);
        }
    }
#pragma unroll
    for (int i = 0; i < kSites; ++i) {
        d[i] = 0.0f;
#pragma unroll
        for (int e = 0; e < E; ++e) d[i] = fmaf(wd[e], x[i][e], d[i]);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) d[i] += __shfl_xor_sync(0xffffffffu, d[i], o);
    }
    const float bd = A.bd[0];
#pragma unroll
    for (int i = 0; i < kSites; ++i) {
        const int m = m0 + i;
        if (m >= M) break;
        const int s = m / A.N, t = m - s * A.N;
        const uint64_t *row = A.bits + (int64_t)s * A.W;
        const int sv = (int)((row[t >> 6] >> (t & 63)) & 1ull);
        int forced = -1;  // forced sites carry no parameter dependence
        if (A.u1) {
            int up = 0;
            for (int w = lane; w < (t >> 6); w += 32) up += __popcll(row[w]);
            if (lane == 0 && (t & 63)) up += __popcll(row[t >> 6] & ((1ull << (t & 63)) - 1ull));
            forced = u1_forced(1, A.N, t, (int)__reduce_add_sync(0xffffffffu, (unsigned)up));
        }
        float g = forced >= 0 ? 0.0f : 0.5f * ((float)sv - 1.0f / (1.0f + expf(-(d[i] + bd))));
        if (A.dout) g *= A.dout[s];
        if (lane == 0) A.g[m] = g;
#pragma unroll
        for (int e = 0; e < E; ++e) top.store((size_t)m * H + 32 * e + lane, g * wd[e], in[i][e]);
    }
}

// gradient of the readout: per (sample, unit) the sum of g x over the sites
static __global__ void __launch_bounds__(128) grad_wo_kernel(const __grid_constant__ ReadoutArgs A) {
    const int H = A.H, N = A.N;
    const int64_t idx = (int64_t)blockIdx.x * 128 + threadIdx.x;
    const int64_t s = idx / H;
    const int j = (int)(idx % H);
    if (s >= A.n) return;
    const float *x = A.x + s * N * H + j, *g = A.g + s * N;
    float wo = 0.0f, bo = 0.0f;
    for (int t0 = 0; t0 < N; t0 += 16) {
        float xv[16], gv[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const bool in = t0 + i < N;
            xv[i] = in ? x[(int64_t)(t0 + i) * H] : 0.0f;
            gv[i] = in ? g[t0 + i] : 0.0f;
        }
        float sw = 0.0f, sb = 0.0f;
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            sw = fmaf(gv[i], xv[i], sw);
            sb += gv[i];
        }
        wo += sw;
        bo += sb;
    }
    float *w = A.wo + s * A.small_stride, *b = A.bo + s * A.small_stride;
    // logit difference d = (W_o[1] - W_o[0]) x + (b_o[1] - b_o[0])
    w[j] = -wo;
    w[H + j] = wo;
    if (j == 0) {
        b[0] = -bo;
        b[1] = bo;
    }
}

template <class Top>
inline cudaError_t launch_readout(const ReadoutArgs &A, const Top &top, cudaStream_t st) {
    const unsigned blocks = (unsigned)((A.n * A.N + 31) / 32);
    if (A.H == 32) grad_readout_kernel<1><<<blocks, 256, 0, st>>>(A, top);
    else if (A.H == 64) grad_readout_kernel<2><<<blocks, 256, 0, st>>>(A, top);
    else grad_readout_kernel<4><<<blocks, 256, 0, st>>>(A, top);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    grad_wo_kernel<<<(unsigned)(((int64_t)A.n * A.H + 127) / 128), 128, 0, st>>>(A);
    return cudaGetLastError();
}

}  // namespace psr
