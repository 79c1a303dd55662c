// Reverse-mode gradient d log psi / d theta of the 2D patched minGRU in FP32
// (Sec. II.F two-dimensional recurrences, Sec. II.G residual), layer by layer
// over a whole batch of samples.  Site-major arrays [patch row][sample][column]
// [unit], so that one patch row of all samples is a contiguous block of
// matrix rows and the patch above a site is the same row of the block before:
//   forward   z | c = [W_z; W_hx] u + b for all patches at once (layer 0: u is
//             the pair of one-hot inputs, 32 wide), then patch row by patch
//             row c += W_hv h(row above) and h_k = z h_{k-1} + (1 - z) c along
//             the path; then x = GELU(C h + D u [+ h of layer l-1]) for all
//   readout   16 logits, masked softmax, g = 1/2 ([o = v] - P(o)) dout
//   backward  gy = gx GELU'(y);  gh = C^T gy (+ gy of layer l+1) for all, then
//             row by row from the last: gh += W_hv^T dc(row below), the reverse
//             scan along the path, dz and dc; then gx of the layer below =
//             W_z^T dz + W_hx^T dc + D^T gy for all
//   weights   sums over patches of dz u^T, dc u^T, dc h(above)^T, gy h^T, gy u^T
// The products run on the engine the caller picks (psr_gemm_tc.cuh, split BF16
// operands on the tensor cores; psr_gemm.cuh, FP32 multiply-adds), the weight
// gradients on CUDA cores.  What bounds it: the weight gradients' FP32 rate (52
// TFLOP/s); the products of one patch row (n Lx / 2 sites) are the only ones
// that wait for each other.  Measured, hidden 256, 1600 samples of 10 x 10,
// weighted sum with log psi of the samples: 3.3 ms (5.3 ms with FP32
// multiply-adds throughout; the row-recompute kernel, psr_bwd2d.cu, a CTA per
// sample: 37.7 ms and two forwards of 4.3 ms).
#include <cuda_runtime.h>

#include "psr_device.cuh"
#include "psr_gemm_tc.cuh"
#include "psr_internal.cuh"

namespace psr {

namespace {

using namespace gemm;

__device__ __forceinline__ int sp2(int Lx, int i, int j) { return j * Lx + ((j & 1) ? Lx - 1 - i : i); }

__device__ __forceinline__ int patch_value(const uint64_t *row, int Lx, int pi, int pj) {
    int v = 0;
#pragma unroll
    for (int b = 0; b < 4; ++b) {
        const int t = sp2(Lx, 2 * pi + (b & 1), 2 * pj + (b >> 1));
        v |= (int)((row[t >> 6] >> (t & 63)) & 1ull) << b;
    }
    return v;
}

// the 32-wide one-hot input (v of the predecessor along the path, v above)
__global__ void __launch_bounds__(256) onehot2d_kernel(const __grid_constant__ Grad2dArgs A) {
    const int Px = A.Lx >> 1, M = A.n * Px * (A.Ly >> 1);
    for (int64_t q = (int64_t)blockIdx.x * 256 + threadIdx.x; q < (int64_t)M * 8; q += (int64_t)gridDim.x * 256) {
        const int m = (int)(q >> 3), e0 = (int)(q & 7) * 4;
        const int i = m % Px, js = m / Px, s = js % A.n, j = js / A.n;
        const uint64_t *row = A.bits + (int64_t)s * A.W;
        const int hi = (j & 1) ? i + 1 : i - 1;
        const int vh = hi >= 0 && hi < Px ? patch_value(row, A.Lx, hi, j) : -1;
        const int vv = j > 0 ? 16 + patch_value(row, A.Lx, i, j - 1) : -1;
        const auto on = [&](int e) { return e == vh || e == vv ? 1.0f : 0.0f; };
        st4(A.u0 + (size_t)m * 32 + e0, make_float4(on(e0), on(e0 + 1), on(e0 + 2), on(e0 + 3)));
    }
}

// W_o padded to 32 rows, and its transpose
__global__ void pad_wo_kernel(const float *__restrict__ wo, int H, float *__restrict__ w32, float *__restrict__ w32t) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < 32 * H; i += gridDim.x * blockDim.x) {
        const int o = i / H, k = i % H;
        const float v = o < 16 ? wo[i] : 0.0f;
        w32[i] = v;
        w32t[k * 32 + o] = v;
    }
}

struct EpiZC {  // a = sigmoid(z), c without its part from the row above
    using In = NoIn;
    const float *bz, *bh;
    float *a, *c;
    int H;
    __device__ NoIn load(int, int) const { return {}; }
    __device__ void store(int m, int u, float4 z, float4 cc, NoIn) const {
        const size_t i = (size_t)m * H + u;
        st4(a + i, map4(sigmoid_f, add4(z, ld4(bz + u))));
        st4(c + i, add4(cc, ld4(bh + u)));
    }
};

struct EpiAdd {  // out += product
    struct In {
        float4 v;
    };
    float *out;
    int H;
    __device__ In load(int m, int j) const { return {ld4(out + (size_t)m * H + j)}; }
    __device__ void store(int m, int j, float4 v, In in) const { st4(out + (size_t)m * H + j, add4(in.v, v)); }
};

struct EpiX {  // GELU and its derivative
    struct In {
        float4 r;
    };
    const float *h_below;  // residual, or null
    float *dy, *x;
    int H;
    __device__ In load(int m, int j) const {
        return {h_below ? ld4(h_below + (size_t)m * H + j) : make_float4(0.0f, 0.0f, 0.0f, 0.0f)};
    }
    __device__ void store(int m, int j, float4 v, In in) const {
        const size_t i = (size_t)m * H + j;
        v = add4(v, in.r);
        const float4 cdf = map4([](float t) { return 0.5f * (1.0f + erff(t * 0.70710678118654752f)); }, v);
        st4(x + i, mul4(v, cdf));
        st4(dy + i, fma4(map4([](float t) { return t * 0.39894228040143268f; }, v),
                         map4([](float t) { return expf(-0.5f * t * t); }, v), cdf));
    }
};

struct EpiGyOf {
    struct In {
        float4 dy;
    };
    const float *dy;
    float *gy;
    int H;
    __device__ In load(int m, int j) const { return {ld4(dy + (size_t)m * H + j)}; }
    __device__ void store(int m, int j, float4 v, In in) const { st4(gy + (size_t)m * H + j, mul4(v, in.dy)); }
};

struct EpiGyAcc {  // gy = (gy + product) GELU'(y): the last of several products
    struct In {
        float4 gy, dy;
    };
    const float *dy;
    float *gy;
    int H;
    __device__ In load(int m, int j) const {
        const size_t i = (size_t)m * H + j;
        return {ld4(gy + i), ld4(dy + i)};
    }
    __device__ void store(int m, int j, float4 v, In in) const {
        st4(gy + (size_t)m * H + j, mul4(add4(in.gy, v), in.dy));
    }
};

constexpr int kStep = 8;  // patches in flight per thread

// h of one patch row of layer l: thread = (sample, unit), along the path
__global__ void __launch_bounds__(128) scan_row_fwd_kernel(const __grid_constant__ Grad2dArgs A, int l, int pj) {
    const int H = A.H, Px = A.Lx >> 1;
    const int64_t idx = (int64_t)blockIdx.x * 128 + threadIdx.x;
    const int64_t s = idx / H;
    if (s >= A.n) return;
    const int64_t base = (((int64_t)pj * A.n + s) * Px + ((pj & 1) ? Px - 1 : 0)) * H + idx % H;
    const int64_t dir = (pj & 1) ? -(int64_t)H : H;
    const float *a = A.a[l] + base, *c = A.c[l] + base;
    float *hp = A.h[l] + base;
    float h = 0.0f;
    for (int k0 = 0; k0 < Px; k0 += kStep) {
        float av[kStep], cv[kStep];
#pragma unroll
        for (int i = 0; i < kStep; ++i) {
            const bool in = k0 + i < Px;
            av[i] = in ? a[(k0 + i) * dir] : 0.0f;
            cv[i] = in ? c[(k0 + i) * dir] : 0.0f;
        }
#pragma unroll
        for (int i = 0; i < kStep; ++i) {
            h = av[i] * h + (1.0f - av[i]) * cv[i];
            if (k0 + i < Px) hp[(k0 + i) * dir] = h;
        }
    }
}

// reverse scan of one patch row: dz in place of gh, and dc
template <bool kResid>
__global__ void __launch_bounds__(128) scan_row_bwd_kernel(const __grid_constant__ Grad2dArgs A, int l, int pj) {
    const int H = A.H, Px = A.Lx >> 1;
    const int64_t idx = (int64_t)blockIdx.x * 128 + threadIdx.x;
    const int64_t s = idx / H;
    if (s >= A.n) return;
    const int64_t base = (((int64_t)pj * A.n + s) * Px + ((pj & 1) ? Px - 1 : 0)) * H + idx % H;
    const int64_t dir = (pj & 1) ? -(int64_t)H : H;
    const float *a = A.a[l] + base, *c = A.c[l] + base, *h = A.h[l] + base, *r = A.gy[(l + 1) & 1] + base;
    float *dzp = A.gh + base, *dcp = A.dc + base;
    float lam = 0.0f, an = 0.0f;
    for (int k0 = Px - kStep; k0 > -kStep; k0 -= kStep) {
        float g[kStep], av[kStep], cv[kStep], hv[kStep];
#pragma unroll
        for (int i = 0; i < kStep; ++i) {
            const int k = k0 + i;
            g[i] = av[i] = cv[i] = hv[i] = 0.0f;
            if (k < 0) continue;
            g[i] = dzp[k * dir];
            if (kResid) g[i] += r[k * dir];
            av[i] = a[k * dir];
            cv[i] = c[k * dir];
            if (k > 0) hv[i] = h[(k - 1) * dir];
        }
#pragma unroll
        for (int i = kStep - 1; i >= 0; --i) {
            const int k = k0 + i;
            if (k < 0) continue;
            lam = g[i] + an * lam;
            dzp[k * dir] = lam * (hv[i] - cv[i]) * av[i] * (1.0f - av[i]);
            dcp[k * dir] = lam * (1.0f - av[i]);
            an = av[i];
        }
    }
}

// Masked 16-way softmax of every patch (one thread each): log P of the patch
// (if logp) and the adjoint of the logits (if grad), 32 wide.
__global__ void __launch_bounds__(128) softmax2d_kernel(const __grid_constant__ Grad2dArgs A, float *logp, bool grad) {
    const int Px = A.Lx >> 1, M = A.n * Px * (A.Ly >> 1), N = A.Lx * A.Ly;
    const int m = blockIdx.x * 128 + threadIdx.x;
    if (m >= M) return;
    const int i = m % Px, js = m / Px, s = js % A.n, j = js / A.n;
    const uint64_t *row = A.bits + (int64_t)s * A.W;
    const float *bo = A.theta + A.tl.bo;
    float lg[16];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const float4 v = ld4(A.logits + (size_t)m * 32 + 4 * q);
        lg[4 * q] = v.x + bo[4 * q];
        lg[4 * q + 1] = v.y + bo[4 * q + 1];
        lg[4 * q + 2] = v.z + bo[4 * q + 2];
        lg[4 * q + 3] = v.w + bo[4 * q + 3];
    }
    int up = 0, down = 0;
    if (A.u1) {
        up = count_up_before(row, 2 * j * A.Lx);
        down = 2 * j * A.Lx - up;
        const int k = (j & 1) ? Px - 1 - i : i;
        for (int q = 0; q < k; ++q) {
            const int pc = __popc(patch_value(row, A.Lx, (j & 1) ? Px - 1 - q : q, j));
            up += pc;
            down += 4 - pc;
        }
    }
    const int v = patch_value(row, A.Lx, i, j);
    unsigned allowed = 0;
    float mx = -INFINITY;
#pragma unroll
    for (int o = 0; o < 16; ++o) {
        const int pc = __popc(o);
        if (!A.u1 || (up + pc <= N / 2 && down + 4 - pc <= N / 2)) {
            allowed |= 1u << o;
            mx = fmaxf(mx, lg[o]);
        }
    }
    float sum = 0.0f, lv = -INFINITY;
#pragma unroll
    for (int o = 0; o < 16; ++o)
        if ((allowed >> o) & 1u) {
            if (o == v) lv = lg[o];
            lg[o] = expf(lg[o] - mx);
            sum += lg[o];
        }
    if (logp) logp[m] = lv - mx - logf(sum);
    if (!grad) return;
    const float sc = 0.5f * (A.dout ? A.dout[s] : 1.0f);
    float *g = A.g + (size_t)m * 32;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        float w[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int o = 4 * q + e;
            const float p = o < 16 && ((allowed >> (o & 15)) & 1u) ? lg[o & 15] / sum : 0.0f;
            w[e] = o < 16 ? sc * ((o == v ? 1.0f : 0.0f) - p) : 0.0f;
        }
        st4(g + 4 * q, make_float4(w[0], w[1], w[2], w[3]));
    }
}

// log psi = 1/2 sum of a sample's log P: one warp per sample
__global__ void __launch_bounds__(256) sum_logp_kernel(const float *__restrict__ logp, int n, int Px, int Py,
                                                       float *__restrict__ out) {
    const int s = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (s >= n) return;
    float acc = 0.0f;
    for (int t = lane; t < Px * Py; t += 32) acc += logp[((size_t)(t / Px) * n + s) * Px + t % Px];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) out[s] = 0.5f * acc;
}

}  // namespace

size_t grad2d_floats_per_site(int nL, int H) { return (size_t)(5 * nL + 4) * H + 3 * 32 + 1; }

cudaError_t launch_grad2d_fwd(const Grad2dArgs &A, float *logpsi, cudaStream_t st) {
    const int H = A.H, Px = A.Lx >> 1, Py = A.Ly >> 1, R = A.n * Px, M = R * Py, nL = A.nL;
    const T2Layout &tl = A.tl;
    const unsigned scan_blocks = (unsigned)(((int64_t)A.n * H + 127) / 128);
    cudaError_t e;
    onehot2d_kernel<<<(unsigned)(((int64_t)M * 8 + 255) / 256), 256, 0, st>>>(A);
    pad_wo_kernel<<<32, 256, 0, st>>>(A.theta + tl.Wo, H, A.wo32, A.wo32t);
    if ((e = cudaGetLastError())) return e;
    for (int l = 0; l < nL; ++l) {
        const int din = l ? H : 32, ldh = din + H;
        const float *u = l ? A.x[l - 1] : A.u0;
        const Args g1{M, H, 1, {{u, A.theta + tl.Wz[l], A.theta + tl.Wh[l], din, din, din, ldh}}};
        if ((e = launch<true>(g1, EpiZC{A.theta + tl.bz[l], A.theta + tl.bh[l], A.a[l], A.c[l], H}, A.en, st))) return e;
        for (int j = 0; j < Py; ++j) {
            if (j > 0) {
                const Args gv{R, H, 1, {{A.h[l] + (size_t)(j - 1) * R * H, A.theta + tl.Wh[l] + din, nullptr, H, H, ldh, 0}}};
                if ((e = launch<false>(gv, EpiAdd{A.c[l] + (size_t)j * R * H, H}, A.en, st))) return e;
            }
            scan_row_fwd_kernel<<<scan_blocks, 128, 0, st>>>(A, l, j);
            if ((e = cudaGetLastError())) return e;
        }
        const Args gy{M, H, 2,
                      {{A.h[l], A.theta + tl.C[l], nullptr, H, H, H, 0}, {u, A.theta + tl.D[l], nullptr, din, din, din, 0}}};
        if ((e = launch<false>(gy, EpiX{l >= 2 ? A.h[l - 1] : nullptr, A.dy[l], A.x[l], H}, A.en, st))) return e;
    }
    const Args go{M, 32, 1, {{A.x[nL - 1], A.wo32, nullptr, H, H, H, 0}}};
    if ((e = launch<false>(go, EpiStore{A.logits, 32}, A.en, st))) return e;
    if (logpsi) {
        softmax2d_kernel<<<(unsigned)((M + 127) / 128), 128, 0, st>>>(A, A.logp, false);
        sum_logp_kernel<<<(unsigned)((A.n + 7) / 8), 256, 0, st>>>(A.logp, A.n, Px, Py, logpsi);
    }
    return cudaGetLastError();
}

cudaError_t launch_grad2d_bwd(const Grad2dArgs &A, cudaStream_t st) {
    const int H = A.H, Px = A.Lx >> 1, Py = A.Ly >> 1, R = A.n * Px, M = R * Py, nL = A.nL;
    const T2Layout &tl = A.tl;
    const unsigned scan_blocks = (unsigned)(((int64_t)A.n * H + 127) / 128);
    const int top = nL - 1;
    cudaError_t e;
    WgArgs w0{};  // ranges of the weight gradients: a sample, or a few hundred sites
    if (A.sum_out) {
        w0.n_range = (M + A.range - 1) / A.range;
        w0.len = w0.step = w0.seg_len = w0.seg_stride = A.range;
    } else {
        w0.n_range = A.n;
        w0.len = Px * Py;
        w0.step = w0.seg_len = Px;
        w0.seg_stride = R;
    }
    w0.out = A.rows;
    w0.out_stride = tl.total;
    softmax2d_kernel<<<(unsigned)((M + 127) / 128), 128, 0, st>>>(A, nullptr, true);
    if ((e = cudaGetLastError())) return e;
    {
        WgArgs w = w0;
        w.n_pair = 1;
        w.p[0] = Pair{A.g, A.x[top], 32, H, 32, H, 16, M, tl.Wo, H, tl.bo};
        if ((e = launch_wgrad(w, A.enw, st))) return e;
        const Args gx{M, H, 1, {{A.g, A.wo32t, nullptr, 32, 32, 32, 0}}};
        if ((e = launch<false>(gx, EpiGyOf{A.dy[top], A.gy[top & 1], H}, A.en, st))) return e;
    }
    for (int l = top; l >= 0; --l) {
        const int din = l ? H : 32, ldh = din + H;
        const float *u = l ? A.x[l - 1] : A.u0;
        float *gy = A.gy[l & 1];
        const bool resid = l + 1 < nL && l + 1 >= 2;
        const Args gc{M, H, 1, {{gy, A.pk + A.f.CT[l], nullptr, H, H, H, 0}}};
        if ((e = launch<false>(gc, EpiStore{A.gh, H}, A.en, st))) return e;
        for (int j = Py - 1; j >= 0; --j) {
            if (j + 1 < Py) {
                const Args gv{R, H, 1, {{A.dc + (size_t)(j + 1) * R * H, A.pk + A.f.WhvT[l], nullptr, H, H, H, 0}}};
                if ((e = launch<false>(gv, EpiAdd{A.gh + (size_t)j * R * H, H}, A.en, st))) return e;
            }
            if (resid) scan_row_bwd_kernel<true><<<scan_blocks, 128, 0, st>>>(A, l, j);
            else scan_row_bwd_kernel<false><<<scan_blocks, 128, 0, st>>>(A, l, j);
            if ((e = cudaGetLastError())) return e;
        }
        // the pairs with the layer input (layer 0: 32 wide) and those with h
        WgArgs w = w0;
        w.n_pair = 3;
        w.p[0] = Pair{gy, u, H, din, H, din, H, M, tl.D[l], din, -1};
        w.p[1] = Pair{A.gh, u, H, din, H, din, H, M, tl.Wz[l], din, tl.bz[l]};
        w.p[2] = Pair{A.dc, u, H, din, H, din, H, M, tl.Wh[l], ldh, tl.bh[l]};
        WgArgs v = w0;
        v.n_pair = 2;
        v.p[0] = Pair{gy, A.h[l], H, H, H, H, H, M, tl.C[l], H, -1};
        // dc of row j with h of row j - 1, at the same column
        v.p[1] = Pair{A.dc + (size_t)R * H, A.h[l], H, H, H, H, H, M - R, tl.Wh[l] + din, ldh, -1};
        if (l) {
            for (int q = 0; q < 2; ++q) w.p[w.n_pair++] = v.p[q];
        } else if ((e = launch_wgrad(v, A.enw, st))) {
            return e;
        }
        if ((e = launch_wgrad(w, A.enw, st))) return e;
        if (l) {
            const Seg seg[3] = {{A.gh, A.pk + A.f.WzT[l], nullptr, H, H, H, 0},
                                {A.dc, A.pk + A.f.WhxT[l], nullptr, H, H, H, 0},
                                {gy, A.pk + A.f.DT[l], nullptr, H, H, H, 0}};
            float *to = A.gy[(l - 1) & 1];
            if (A.en.split) {
                // one product each, added in FP32: a tensor-core sum over 3 H
                // terms would round (toward zero) three times as often
                if ((e = launch<false>(Args{M, H, 1, {seg[0]}}, EpiStore{to, H}, A.en, st))) return e;
                if ((e = launch<false>(Args{M, H, 1, {seg[1]}}, EpiAdd{to, H}, A.en, st))) return e;
                if ((e = launch<false>(Args{M, H, 1, {seg[2]}}, EpiGyAcc{A.dy[l - 1], to, H}, A.en, st))) return e;
            } else {
                const Args gx{M, H, 3, {seg[0], seg[1], seg[2]}};
                if ((e = launch<false>(gx, EpiGyOf{A.dy[l - 1], to, H}, A.en, st))) return e;
            }
        }
    }
    if (!A.sum_out) return cudaSuccess;
    SumArgs sa{};
    sa.add = A.add;
    sa.out = A.sum_out;
    sa.n = 1;
    sa.s[0] = SumSeg{A.rows, tl.total, 0, w0.n_range, (int)tl.total};
    return launch_sum_rows(sa, st);
}

}  // namespace psr
