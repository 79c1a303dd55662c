// Reverse-mode gradient d log psi / d theta of the chain minGRU
// (derivative of Eq. minGRU and of the output map, Sec. II.F-G; the
// energy-gradient estimates of Sec. III.B), layer by layer over a whole batch
// of samples in site-major arrays [sample][site][unit]:
//   forward   z | c = [W_z; W_h] u + b (layer 0: lookups of the one-hot input),
//             a = sigmoid(z); h_t = a_t h_{t-1} + (1 - a_t) c_t;
//             y = C h + D u [+ h of layer l-1 for l >= 2], u of the next layer
//             = GELU(y); readout adjoint g_t = 1/2 (s_t - P(1 | s_<t)) dout
//   backward  gy = gx GELU'(y);  gh = C^T gy (+ gy of layer l+1, l+1 >= 2);
//             lambda_t = gh_t + a_{t+1} lambda_{t+1};
//             dz = lambda (h_{t-1} - c) a (1 - a),  dc = lambda (1 - a);
//             gx of layer l-1 = W_z^T dz + W_h^T dc + D^T gy
//   weights   dC = sum gy h^T, dD = sum gy u^T, dW_z = sum dz u^T, dW_h = sum dc u^T
// The products run on the engine the caller picks (psr_gemm_tc.cuh: split BF16
// operands on the tensor cores; psr_gemm.cuh: FP32 multiply-adds); the scans are
// one thread per (sample, unit), coalesced over units.
//
// What bounds it: HBM, for the arrays between the products (about 75 arrays of
// 4 H bytes a site; the products run at 0.5 to 0.8 of the measured rate for
// their bytes, the weight gradients at 0.4).  Measured, per-sample kernels of
// a CTA each with reductions in L2 (psr_bwd.cu) / FP32 multiply-adds / split
// operands: weighted sum, hidden 64, 4096 samples of 100 sites 11.3 / 2.9 / 2.1
// ms; O_k rows at BF16, hidden 128, 2048 samples of 100 sites 2.0 ms (two-part
// split; 5.7 ms in unit-major arrays with unpipelined products before).
#include <cuda_runtime.h>

#include "psr_device.cuh"
#include "psr_gemm_tc.cuh"
#include "psr_grad_common.cuh"
#include "psr_internal.cuh"

namespace psr {

namespace {

using namespace gemm;

struct EpiProj {  // a = sigmoid(z), c
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

struct EpiOut {  // the next layer's input u = GELU(y), and GELU'(y) for the way back
    struct In {
        float4 more;  // layer 0: D of the one-hot input; l >= 2: h of the layer below
    };
    const float *du0;      // layer 0: D of the one-hot input by code, else null
    const float *h_below;  // residual, or null
    const uint64_t *bits;
    float *dy, *u;
    int H, N, W;
    __device__ In load(int m, int j) const {
        if (du0) {
            const int s = m / N;
            return {ld4(du0 + code_at(bits + (int64_t)s * W, m - s * N) * H + j)};
        }
        return {h_below ? ld4(h_below + (size_t)m * H + j) : make_float4(0.0f, 0.0f, 0.0f, 0.0f)};
    }
    __device__ void store(int m, int j, float4 v, In in) const {
        const size_t i = (size_t)m * H + j;
        v = add4(v, in.more);
        const float4 cdf = map4([](float x) { return 0.5f * (1.0f + erff(x * 0.70710678118654752f)); }, v);
        st4(u + i, mul4(v, cdf));
        st4(dy + i, fma4(map4([](float x) { return x * 0.39894228040143268f; }, v),
                         map4([](float x) { return expf(-0.5f * x * x); }, v), cdf));
    }
};

struct EpiGy {  // adjoint of the pre-activation of the layer below
    struct In {
        float4 dy;
    };
    const float *dy;
    float *gy;
    int H;
    __device__ In load(int m, int j) const { return {ld4(dy + (size_t)m * H + j)}; }
    __device__ void store(int m, int j, float4 v, In in) const { st4(gy + (size_t)m * H + j, mul4(v, in.dy)); }
};

constexpr int kScanStep = 8;

// h of one layer; layer 0 takes a and b = (1 - a) c from the input code
__global__ void __launch_bounds__(128) grad_scan_fwd_kernel(const __grid_constant__ GradF32Args A, int l) {
    const int H = A.H, N = A.N;
    const int64_t idx = (int64_t)blockIdx.x * 128 + threadIdx.x;
    const int64_t s = idx / H;
    const int j = (int)(idx % H);
    if (s >= A.n) return;
    const int64_t base = s * N * H + j;
    float *hp = A.h[l] + base;
    float h = 0.0f;
    if (l == 0) {
        const uint64_t *row = A.bits + s * A.W;
        float ta[3], tb[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            ta[q] = A.pk[A.fl.A0 + q * H + j];
            tb[q] = A.pk[A.fl.B0 + q * H + j];
        }
        h = tb[0];
        hp[0] = h;
        for (int t = 1; t < N; ++t) {
            const bool up = (row[(t - 1) >> 6] >> ((t - 1) & 63)) & 1ull;
            h = (up ? ta[2] : ta[1]) * h + (up ? tb[2] : tb[1]);
            hp[(int64_t)t * H] = h;
        }
        return;
    }
    const float *ap = A.a[l] + base, *cp = A.c[l] + base;
    float na[kScanStep], nc[kScanStep];
    auto fetch = [&](int t) {
#pragma unroll
        for (int i = 0; i < kScanStep; ++i) {
            const bool in = t + i < N;
            na[i] = in ? ap[(int64_t)(t + i) * H] : 0.0f;
            nc[i] = in ? cp[(int64_t)(t + i) * H] : 0.0f;
        }
    };
    fetch(0);
    for (int t = 0; t < N; t += kScanStep) {
        float a[kScanStep], c[kScanStep];
#pragma unroll
        for (int i = 0; i < kScanStep; ++i) {
            a[i] = na[i];
            c[i] = nc[i];
        }
        fetch(t + kScanStep);  // in flight while this step is computed
#pragma unroll
        for (int i = 0; i < kScanStep; ++i) {
            h = a[i] * h + (1.0f - a[i]) * c[i];
            if (t + i < N) hp[(int64_t)(t + i) * H] = h;
        }
    }
}

struct TopGy {  // gy of the top layer from gx = g wd
    using In = float;
    const float *dy;
    float *gy;
    __device__ float load(size_t i) const { return dy[i]; }
    __device__ void store(size_t i, float gx, float d) const { gy[i] = gx * d; }
};

// reverse scan of a layer l >= 1: dz (in place of gh) and dc
template <bool kResid>
__global__ void __launch_bounds__(128) grad_scan_bwd_kernel(const __grid_constant__ GradF32Args A, int l) {
    const int H = A.H, N = A.N;
    const int64_t idx = (int64_t)blockIdx.x * 128 + threadIdx.x;
    const int64_t s = idx / H;
    if (s >= A.n) return;
    const int64_t base = s * N * H + idx % H;
    float *dzp = A.gh + base, *dcp = A.dc + base;
    const float *hp = A.h[l] + base, *ap = A.a[l] + base, *cp = A.c[l] + base;
    const float *rp = A.gy[(l + 1) & 1] + base;
    float lam = 0.0f, an = 0.0f;
    float g[kScanStep], a[kScanStep], c[kScanStep], h[kScanStep], r[kScanStep];
    auto fetch = [&](int t) {  // sites t .. t + kScanStep - 1; h one site earlier
#pragma unroll
        for (int i = 0; i < kScanStep; ++i) {
            const int64_t o = (int64_t)(t + i) * H;
            g[i] = a[i] = c[i] = h[i] = r[i] = 0.0f;
            if (t + i >= 0) {
                g[i] = dzp[o];
                a[i] = ap[o];
                c[i] = cp[o];
                if (kResid) r[i] = rp[o];
                if (t + i >= 1) h[i] = hp[o - H];
            }
        }
    };
    // steps end at the last site; the first one may reach before site 0
    fetch(N - kScanStep);
    for (int t = N - kScanStep; t > -kScanStep; t -= kScanStep) {
        float dz[kScanStep], dc[kScanStep];
#pragma unroll
        for (int i = kScanStep - 1; i >= 0; --i) {
            lam = (kResid ? g[i] + r[i] : g[i]) + an * lam;
            dz[i] = lam * (h[i] - c[i]) * a[i] * (1.0f - a[i]);
            dc[i] = lam * (1.0f - a[i]);
            an = a[i];
        }
        fetch(t - kScanStep);
#pragma unroll
        for (int i = 0; i < kScanStep; ++i) {
            if (t + i < 0) continue;
            const int64_t o = (int64_t)(t + i) * H;
            dzp[o] = dz[i];
            dcp[o] = dc[i];
        }
    }
}

// reverse scan of layer 0 (one-hot input): the sums of dz, dc and gy by input
// code, which are its W_z, W_h, D and bias gradients
__global__ void __launch_bounds__(128) grad_scan_bwd0_kernel(const __grid_constant__ GradF32Args A) {
    const int H = A.H, N = A.N;
    const int64_t idx = (int64_t)blockIdx.x * 128 + threadIdx.x;
    const int64_t s = idx / H;
    const int j = (int)(idx % H);
    if (s >= A.n) return;
    const int64_t base = s * N * H + j;
    const float *gp = A.gh + base, *hp = A.h[0] + base, *gyp = A.gy[0] + base;
    const uint64_t *row = A.bits + s * A.W;
    float ta[3], tc[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        ta[q] = A.pk[A.fl.A0 + q * H + j];
        tc[q] = A.pk[A.fl.CD0 + q * H + j];
    }
    // [0]: spin before the site down, [1]: up; a step's sums first, so that
    // their rounding grows with the square root of the steps
    float z[2] = {0, 0}, cs[2] = {0, 0}, ds[2] = {0, 0};
    float lam = 0.0f, an = 0.0f;
    float g[kScanStep], h[kScanStep], gy[kScanStep];
    unsigned up = 0;
    auto fetch = [&](int t) {
        up = 0;
#pragma unroll
        for (int i = 0; i < kScanStep; ++i) {
            const int64_t o = (int64_t)(t + i) * H;
            g[i] = h[i] = gy[i] = 0.0f;
            if (t + i >= 0) {
                g[i] = gp[o];
                gy[i] = gyp[o];
                if (t + i >= 1) {
                    h[i] = hp[o - H];
                    const int q = t + i - 1;
                    up |= (unsigned)((row[q >> 6] >> (q & 63)) & 1ull) << i;
                }
            }
        }
    };
    fetch(N - kScanStep);
    float dz0 = 0.0f, dc0 = 0.0f;
    for (int t = N - kScanStep; t > -kScanStep; t -= kScanStep) {
        float sz[2] = {0, 0}, sc[2] = {0, 0}, sd[2] = {0, 0};
#pragma unroll
        for (int i = kScanStep - 1; i >= 0; --i) {
            const bool first = t + i == 0, on = (up >> i) & 1u;
            const float a = first ? ta[0] : on ? ta[2] : ta[1];
            const float c = first ? tc[0] : on ? tc[2] : tc[1];
            lam = g[i] + an * lam;
            const float dz = lam * (h[i] - c) * a * (1.0f - a), dc = lam * (1.0f - a);
            an = a;
            if (t + i > 0) {
                sz[0] += on ? 0.0f : dz;
                sz[1] += on ? dz : 0.0f;
                sc[0] += on ? 0.0f : dc;
                sc[1] += on ? dc : 0.0f;
                sd[0] += on ? 0.0f : gy[i];
                sd[1] += on ? gy[i] : 0.0f;
            } else if (first) {  // no input there: the biases only
                dz0 = dz;
                dc0 = dc;
            }
        }
        fetch(t - kScanStep);
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            z[q] += sz[q];
            cs[q] += sc[q];
            ds[q] += sd[q];
        }
    }
    float *out = A.small + s * A.small_stride;
    const GradSmall &o = A.sm;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        out[o.Wz0 + 2 * j + q] = z[q];
        out[o.Wh0 + 2 * j + q] = cs[q];
        out[o.D0 + 2 * j + q] = ds[q];
    }
    out[o.bz0 + j] = dz0 + (z[0] + z[1]);
    out[o.bh0 + j] = dc0 + (cs[0] + cs[1]);
}

}  // namespace

// A range is one CTA's serial sum, so few sites take shorter ones, down to a
// stage of the kernels, while there are too few to fill the SMs (a range is four
// tiles at hidden 32, more at wider models, whose partial rows cost more to add).
// 64 samples of 16 sites, hidden 32: the gradient took 148 us with 256-site
// ranges, 139 us with 64-site ones.  At hidden 128, 6400 sites of the LRU stay at
// 512 (50 ranges instead of 13 took 2 % longer).
int grad_f32_range(int H, int64_t sites) {
    int r = H <= 64 ? 256 : 512;
    const int least = H == 32 ? 32 : 64, enough = H <= 64 ? 32 : 8;
    while (r > least && sites < enough * (int64_t)r) r /= 2;
    return r;
}

size_t grad_f32_floats_per_site(int nL, int H) { return (size_t)(5 * nL - 2 + 4) * H + 1; }

int64_t grad_f32_small_floats(int H) { return 10 * (int64_t)H + 2; }

cudaError_t launch_grad_f32(const GradF32Args &A, cudaStream_t st) {
    const int H = A.H, M = A.n * A.N, nL = A.nL;
    const ThetaLayout &tl = A.tl;
    const unsigned scan_blocks = (unsigned)(((int64_t)A.n * H + 127) / 128);
    cudaError_t e;
    // ------------------------------------------------ forward
    for (int l = 0; l < nL; ++l) {
        if (l > 0) {
            Args g{M, H, 1, {{A.u[l - 1], A.theta + tl.Wz[l], A.theta + tl.Wh[l], H, H, H, H}}};
            if ((e = launch<true>(g, EpiProj{A.pk + A.fl.bz[l], A.pk + A.fl.bh[l], A.a[l], A.c[l], H}, A.en, st))) return e;
        }
        grad_scan_fwd_kernel<<<scan_blocks, 128, 0, st>>>(A, l);
        if ((e = cudaGetLastError())) return e;
        Args g{M, H, l ? 2 : 1, {{A.h[l], A.theta + tl.C[l], nullptr, H, H, H, H}, {}}};
        if (l) g.seg[1] = Seg{A.u[l - 1], A.theta + tl.D[l], nullptr, H, H, H, H};
        const EpiOut eo{l ? nullptr : A.pk + A.fl.DU0, l >= 2 ? A.h[l - 1] : nullptr, A.bits, A.dy[l], A.u[l], H, A.N, A.W};
        if ((e = launch<false>(g, eo, A.en, st))) return e;
    }
    const ReadoutArgs ro{A.n, A.N, H, A.W, A.u1, A.bits, A.u[nL - 1], A.pk + A.fl.wd, A.pk + A.fl.bd, A.dout, A.g,
                         A.small + A.sm.Wo, A.small + A.sm.bo, A.small_stride};
    if ((e = launch_readout(ro, TopGy{A.dy[nL - 1], A.gy[(nL - 1) & 1]}, st))) return e;
    // ------------------------------------------------ backward, top down
    const int range = A.sum_out ? A.range : A.N;
    for (int l = nL - 1; l >= 0; --l) {
        float *gy = A.gy[l & 1];
        Args gc{M, H, 1, {{gy, A.pk + A.fl.CT[l], nullptr, H, H, H, H}}};
        if ((e = launch<false>(gc, EpiStore{A.gh, H}, A.en, st))) return e;
        if (l == 0) grad_scan_bwd0_kernel<<<scan_blocks, 128, 0, st>>>(A);
        else if (l + 1 < nL) grad_scan_bwd_kernel<true><<<scan_blocks, 128, 0, st>>>(A, l);
        else grad_scan_bwd_kernel<false><<<scan_blocks, 128, 0, st>>>(A, l);
        if ((e = cudaGetLastError())) return e;
        WgArgs w{};
        w.n_pair = l ? 4 : 1;
        w.p[0] = Pair{gy, A.h[l], H, H, H, H, H, M, tl.C[l], H, -1};
        if (l) {
            const float *u = A.u[l - 1];
            w.p[1] = Pair{gy, u, H, H, H, H, H, M, tl.D[l], H, -1};
            w.p[2] = Pair{A.gh, u, H, H, H, H, H, M, tl.Wz[l], H, tl.bz[l]};
            w.p[3] = Pair{A.dc, u, H, H, H, H, H, M, tl.Wh[l], H, tl.bh[l]};
        }
        w.n_range = A.sum_out ? (M + range - 1) / range : A.n;
        w.len = w.step = range;
        w.seg_len = range;
        w.seg_stride = range;
        w.out = A.rows;
        w.out_stride = tl.total;
        if ((e = launch_wgrad(w, A.en, st))) return e;
        if (l > 0) {
            // W^T as [input unit][output unit] rows: the packed transposes
            Args gx{M, H, 3,
                    {{A.gh, A.pk + A.fl.WzT[l], nullptr, H, H, H, H},
                     {A.dc, A.pk + A.fl.WhT[l], nullptr, H, H, H, H},
                     {gy, A.pk + A.fl.DT[l], nullptr, H, H, H, H}}};
            if ((e = launch<false>(gx, EpiGy{A.dy[l - 1], A.gy[(l - 1) & 1], H}, A.en, st))) return e;
        }
    }
    if (!A.sum_out) return cudaSuccess;
    SumArgs sa{};
    sa.add = A.add;
    sa.out = A.sum_out;
    const int n_range = (M + range - 1) / range;
    auto part = [&](int64_t off, int64_t len) { sa.s[sa.n++] = SumSeg{A.rows + off, tl.total, off, n_range, (int)len}; };
    auto small = [&](int64_t src, int64_t dst, int len) {
        sa.s[sa.n++] = SumSeg{A.small + src, A.small_stride, dst, A.n, len};
    };
    for (int l = 0; l < nL; ++l) {
        if (l) part(tl.Wz[l], 4 * (int64_t)H * H + 2 * H);
        else part(tl.C[0], (int64_t)H * H);
    }
    small(A.sm.Wz0, tl.Wz[0], 2 * H);
    small(A.sm.bz0, tl.bz[0], H);
    small(A.sm.Wh0, tl.Wh[0], 2 * H);
    small(A.sm.bh0, tl.bh[0], H);
    small(A.sm.D0, tl.D[0], 2 * H);
    small(A.sm.Wo, tl.Wo, 2 * H);
    small(A.sm.bo, tl.bo, 2);
    return launch_sum_rows(sa, st);
}

}  // namespace psr
