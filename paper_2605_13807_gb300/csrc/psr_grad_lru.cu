// Reverse-mode gradient d log psi / d theta of the deep 1D LRU in FP32
// (Sec. II.B Eq. lru, Sec. II.G 1D residual, Sec. III.B GLU blocks), layer by
// layer over a whole batch of samples in site-major arrays [sample][site][unit]
// (complex numbers as two arrays; the states' imaginary part is kept negated,
// as C uses it):
//   forward   Bu = B u (layer 0: lookups); h_t = lambda h_{t-1} + e^gamma Bu_t;
//             y = Re(C h) + D u;  x = a sigmoid(g) [+ u], a = W_a y + b_a,
//             g = W_g y + b_g;  kept: sigmoid(g) and a sigmoid(g) (1 - sigmoid(g))
//   backward  da, dg from gx;  dy = W_a^T da + W_g^T dg;
//             dh = (C_re^T dy, -C_im^T dy);  mu_t = dh_t + conj(lambda) mu_{t+1};
//             d(Bu) = e^gamma mu;  gx of the layer below = B_re^T d(Bu)_re +
//             B_im^T d(Bu)_im + D dy + gx (residual)
//   weights   sums over sites of da y^T, dg y^T, dy h^T, d(Bu) u^T; lambda,
//             gamma, D and the one-hot columns of layer 0 in the reverse scan
// The products run on the engine the caller picks (psr_gemm_tc.cuh, split BF16
// operands on the tensor cores; psr_gemm.cuh, FP32 multiply-adds).  What bounds
// it: HBM for about 110 arrays of 4 H bytes a site.  Measured, hidden 64, 1024
// samples of 256 sites, weighted sum: 2.3 ms (3.3 ms with FP32 multiply-adds;
// 10.7 ms for the chunk-recompute kernel, psr_bwd_lru.cu, and its forward).
#include <cuda_runtime.h>

#include "psr_device.cuh"
#include "psr_gemm_tc.cuh"
#include "psr_grad_common.cuh"
#include "psr_internal.cuh"

namespace psr {

namespace {

using namespace gemm;

struct EpiBu {
    using In = NoIn;
    float *br, *bi;
    int H;
    __device__ NoIn load(int, int) const { return {}; }
    __device__ void store(int m, int u, float4 vr, float4 vi, NoIn) const {
        const size_t i = (size_t)m * H + u;
        st4(br + i, vr);
        st4(bi + i, vi);
    }
};

struct EpiY {  // y = Re(C h) + D u
    struct In {
        float4 du;
    };
    const float *d;  // layer 0: D by input code [2][H]; above: diagonal [H]
    const float *u;  // layer input, null at layer 0
    const uint64_t *bits;
    float *y;
    int H, N, W;
    __device__ In load(int m, int j) const {
        if (u) return {mul4(ld4(d + j), ld4(u + (size_t)m * H + j))};
        const int s = m / N, code = code_at(bits + (int64_t)s * W, m - s * N);
        return {code ? ld4(d + (code - 1) * H + j) : make_float4(0.0f, 0.0f, 0.0f, 0.0f)};
    }
    __device__ void store(int m, int j, float4 v, In in) const { st4(y + (size_t)m * H + j, add4(v, in.du)); }
};

struct EpiGlu {
    struct In {
        float4 u;
    };
    const float *ba, *bg;
    const float *u;  // residual, or null
    float *p1, *p2, *x;
    int H;
    __device__ In load(int m, int j) const {
        return {u ? ld4(u + (size_t)m * H + j) : make_float4(0.0f, 0.0f, 0.0f, 0.0f)};
    }
    __device__ void store(int m, int j, float4 va, float4 vg, In in) const {
        const size_t i = (size_t)m * H + j;
        const float4 a = add4(va, ld4(ba + j)), sg = map4(sigmoid_f, add4(vg, ld4(bg + j)));
        st4(p1 + i, sg);
        st4(p2 + i, map4([](float x, float s) { return x * s * (1.0f - s); }, a, sg));
        st4(x + i, fma4(a, sg, in.u));
    }
};

struct EpiDh {
    using In = NoIn;
    float *re, *im;
    int H;
    __device__ NoIn load(int, int) const { return {}; }
    __device__ void store(int m, int j, float4 vr, float4 vi, NoIn) const {
        const size_t i = (size_t)m * H + j;
        st4(re + i, vr);
        st4(im + i, map4([](float x) { return -x; }, vi));
    }
};

// gx of a block's output turned into the adjoints of its GLU
struct TopGlu {
    struct In {
        float p1, p2;
    };
    const float *p1, *p2;
    float *gx, *da, *dg;
    __device__ In load(size_t i) const { return {p1[i], p2[i]}; }
    __device__ void store(size_t i, float v, In in) const {
        gx[i] = v;
        da[i] = v * in.p1;
        dg[i] = v * in.p2;
    }
};

struct EpiGx {  // through the residual and D, then the GLU of the layer below
    struct In {
        float4 dy, gx, p1, p2;
    };
    const float *d, *dy, *p1, *p2;
    float *gx, *da, *dg;
    int H;
    __device__ In load(int m, int j) const {
        const size_t i = (size_t)m * H + j;
        return {ld4(dy + i), ld4(gx + i), ld4(p1 + i), ld4(p2 + i)};
    }
    __device__ void store(int m, int j, float4 v, In in) const {
        const size_t i = (size_t)m * H + j;
        v = add4(fma4(ld4(d + j), in.dy, v), in.gx);
        st4(gx + i, v);
        st4(da + i, mul4(v, in.p1));
        st4(dg + i, mul4(v, in.p2));
    }
};

constexpr int kStep = 8;

__global__ void __launch_bounds__(128) lru_scan_fwd_kernel(const __grid_constant__ GradLruArgs A, int l) {
    const int H = A.H, N = A.N;
    const int64_t idx = (int64_t)blockIdx.x * 128 + threadIdx.x;
    const int64_t s = idx / H;
    const int j = (int)(idx % H);
    if (s >= A.n) return;
    const int64_t base = s * N * H + j;
    const float lr = A.pk[A.f.lre[l] + j], li = A.pk[A.f.lim[l] + j], ga = A.pk[A.f.gam[l] + j];
    float *hr = A.hr[l] + base, *hn = A.hn[l] + base;
    const float *brp = l ? A.br[l] + base : nullptr, *bip = l ? A.bi[l] + base : nullptr;
    const uint64_t *row = A.bits + s * A.W;
    float tr[2] = {0, 0}, ti[2] = {0, 0};
    if (l == 0) {
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            tr[q] = A.pk[A.f.BreT[0] + q * H + j];
            ti[q] = A.pk[A.f.BimT[0] + q * H + j];
        }
    }
    float nr[kStep], ni[kStep];
    auto fetch = [&](int t) {
#pragma unroll
        for (int i = 0; i < kStep; ++i) {
            nr[i] = ni[i] = 0.0f;
            const int tt = t + i;
            if (tt >= N) continue;
            if (l) {
                nr[i] = brp[(int64_t)tt * H];
                ni[i] = bip[(int64_t)tt * H];
            } else if (tt > 0) {
                const bool up = (row[(tt - 1) >> 6] >> ((tt - 1) & 63)) & 1ull;
                nr[i] = up ? tr[1] : tr[0];
                ni[i] = up ? ti[1] : ti[0];
            }
        }
    };
    float zr = 0.0f, zi = 0.0f;
    fetch(0);
    for (int t = 0; t < N; t += kStep) {
        float b[kStep], c[kStep];
#pragma unroll
        for (int i = 0; i < kStep; ++i) {
            b[i] = nr[i];
            c[i] = ni[i];
        }
        fetch(t + kStep);
#pragma unroll
        for (int i = 0; i < kStep; ++i) {
            const float r = fmaf(lr, zr, fmaf(-li, zi, ga * b[i]));
            const float m = fmaf(lr, zi, fmaf(li, zr, ga * c[i]));
            zr = r;
            zi = m;
            if (t + i < N) {
                hr[(int64_t)(t + i) * H] = zr;
                hn[(int64_t)(t + i) * H] = -zi;
            }
        }
    }
}

// Reverse scan: d(Bu) in place of dh; the sums for lambda and gamma, D, and at
// layer 0 the one-hot columns of B and D.
template <bool kFirst>
__global__ void __launch_bounds__(128) lru_scan_bwd_kernel(const __grid_constant__ GradLruArgs A, int l) {
    constexpr int S = 4;
    const int H = A.H, N = A.N;
    const int64_t idx = (int64_t)blockIdx.x * 128 + threadIdx.x;
    const int64_t s = idx / H;
    const int j = (int)(idx % H);
    if (s >= A.n) return;
    const int64_t base = s * N * H + j;
    const float lr = A.pk[A.f.lre[l] + j], li = A.pk[A.f.lim[l] + j], ga = A.pk[A.f.gam[l] + j];
    float *drp = A.dhr + base, *dip = A.dhi + base;
    const float *hrp = A.hr[l] + base, *hnp = A.hn[l] + base, *dyp = A.dy + base;
    const float *brp = kFirst ? nullptr : A.br[l] + base, *bip = kFirst ? nullptr : A.bi[l] + base;
    const float *up = kFirst ? nullptr : A.x[l - 1] + base;
    const uint64_t *row = A.bits + s * A.W;
    float tr[2] = {0, 0}, ti[2] = {0, 0};
    if (kFirst) {
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            tr[q] = A.pk[A.f.BreT[0] + q * H + j];
            ti[q] = A.pk[A.f.BimT[0] + q * H + j];
        }
    }
    float dr[S], di[S], hr[S], hn[S], dy[S], br[S], bi[S], u[S];
    unsigned on = 0;  // layer 0: spin before the site
    auto fetch = [&](int t) {
        on = 0;
#pragma unroll
        for (int i = 0; i < S; ++i) {
            const int tt = t + i;
            const int64_t o = (int64_t)tt * H;
            dr[i] = di[i] = hr[i] = hn[i] = dy[i] = br[i] = bi[i] = u[i] = 0.0f;
            if (tt < 0) continue;
            dr[i] = drp[o];
            di[i] = dip[o];
            dy[i] = dyp[o];
            if (!kFirst) {
                br[i] = brp[o];
                bi[i] = bip[o];
                u[i] = up[o];
            }
            if (tt >= 1) {
                hr[i] = hrp[o - H];
                hn[i] = hnp[o - H];
                if (kFirst) on |= (unsigned)((row[(tt - 1) >> 6] >> ((tt - 1) & 63)) & 1ull) << i;
            }
        }
    };
    float mr = 0.0f, mi = 0.0f;
    float sr = 0.0f, si = 0.0f, sg = 0.0f, sd[2] = {0, 0}, sbr[2] = {0, 0}, sbi[2] = {0, 0};
    fetch(N - S);
    for (int t = N - S; t > -S; t -= S) {
        float wr[S], wi[S];
        float pr = 0.0f, pi = 0.0f, pg = 0.0f, pd[2] = {0, 0}, pbr[2] = {0, 0}, pbi[2] = {0, 0};
#pragma unroll
        for (int i = S - 1; i >= 0; --i) {
            const float a = dr[i] + lr * mr + li * mi;
            const float b = di[i] - li * mr + lr * mi;
            mr = a;
            mi = b;
            // h_{t-1} = (hr, -hn)
            pr += mr * hr[i] - mi * hn[i];
            pi += mi * hr[i] + mr * hn[i];
            wr[i] = ga * mr;
            wi[i] = ga * mi;
            if (kFirst) {
                if (t + i < 1) continue;  // no input at the first site (nor before it)
                const bool w = (on >> i) & 1u;
                pg += mr * (w ? tr[1] : tr[0]) + mi * (w ? ti[1] : ti[0]);
                pd[0] += w ? 0.0f : dy[i];
                pd[1] += w ? dy[i] : 0.0f;
                pbr[0] += w ? 0.0f : wr[i];
                pbr[1] += w ? wr[i] : 0.0f;
                pbi[0] += w ? 0.0f : wi[i];
                pbi[1] += w ? wi[i] : 0.0f;
            } else {
                pg += mr * br[i] + mi * bi[i];
                pd[0] += dy[i] * u[i];
            }
        }
        fetch(t - S);
        if (!kFirst) {
#pragma unroll
            for (int i = 0; i < S; ++i) {
                if (t + i < 0) continue;
                drp[(int64_t)(t + i) * H] = wr[i];
                dip[(int64_t)(t + i) * H] = wi[i];
            }
        }
        sr += pr;
        si += pi;
        sg += pg;
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            sd[q] += pd[q];
            sbr[q] += pbr[q];
            sbi[q] += pbi[q];
        }
    }
    // lambda = exp(-e^nu) (cos e^theta + i sin e^theta)
    float *out = A.small + s * A.small_stride;
    const float enu = expf(A.theta[A.tl.nu[l] + j]), eth = expf(A.theta[A.tl.th[l] + j]);
    out[A.sm.nu[l] + j] = -enu * (sr * lr + si * li);
    out[A.sm.th[l] + j] = eth * (si * lr - sr * li);
    out[A.sm.ga[l] + j] = sg * ga;
    if (kFirst) {
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            out[A.sm.Bre0 + 2 * j + q] = sbr[q];
            out[A.sm.Bim0 + 2 * j + q] = sbi[q];
            out[A.sm.D[0] + 2 * j + q] = sd[q];
        }
    } else {
        out[A.sm.D[l] + j] = sd[0];
    }
}

}  // namespace

size_t grad_lru_floats_per_site(int nL, int H) { return (size_t)(8 * nL - 2 + 6) * H + 1; }

// compact places of the per-sample entries of a weighted sum
GradLruSmall grad_lru_small(int nL, int H, int64_t *floats) {
    GradLruSmall m{};
    int64_t off = 0;
    auto take = [&](int64_t k) {
        const int64_t o = off;
        off += k;
        return o;
    };
    for (int l = 0; l < nL; ++l) {
        m.nu[l] = take(H);
        m.th[l] = take(H);
        m.ga[l] = take(H);
        m.D[l] = take(l ? H : 2 * H);
    }
    m.Bre0 = take(2 * H);
    m.Bim0 = take(2 * H);
    m.Wo = take(2 * H);
    m.bo = take(2);
    *floats = off;
    return m;
}

cudaError_t launch_grad_lru(const GradLruArgs &A, cudaStream_t st) {
    const int H = A.H, M = A.n * A.N, nL = A.nL;
    const TLruLayout &tl = A.tl;
    const unsigned scan_blocks = (unsigned)(((int64_t)A.n * H + 127) / 128);
    cudaError_t e;
    // ------------------------------------------------ forward
    for (int l = 0; l < nL; ++l) {
        const float *u = l ? A.x[l - 1] : nullptr;
        if (l) {
            const Args g{M, H, 1, {{u, A.theta + tl.Bre[l], A.theta + tl.Bim[l], H, H, H, H}}};
            if ((e = launch<true>(g, EpiBu{A.br[l], A.bi[l], H}, A.en, st))) return e;
        }
        lru_scan_fwd_kernel<<<scan_blocks, 128, 0, st>>>(A, l);
        if ((e = cudaGetLastError())) return e;
        const Args gy{M, H, 2,
                      {{A.hr[l], A.theta + tl.Cre[l], nullptr, H, H, H, H}, {A.hn[l], A.theta + tl.Cim[l], nullptr, H, H, H, H}}};
        if ((e = launch<false>(gy, EpiY{A.pk + A.f.D[l], u, A.bits, A.y[l], H, A.N, A.W}, A.en, st))) return e;
        const Args gg{M, H, 1, {{A.y[l], A.theta + tl.Wa[l], A.theta + tl.Wg[l], H, H, H, H}}};
        if ((e = launch<true>(gg, EpiGlu{A.pk + A.f.ba[l], A.pk + A.f.bg[l], u, A.p1[l], A.p2[l], A.x[l], H}, A.en, st))) return e;
    }
    const int top = nL - 1;
    const ReadoutArgs ro{A.n, A.N, H, A.W, A.u1, A.bits, A.x[top], A.pk + A.f.wd, A.pk + A.f.bd, A.dout, A.g,
                         A.small + A.sm.Wo, A.small + A.sm.bo, A.small_stride};
    if ((e = launch_readout(ro, TopGlu{A.p1[top], A.p2[top], A.gx, A.da, A.dg}, st))) return e;
    // ------------------------------------------------ backward, top down
    const int range = A.sum_out ? A.range : A.N;
    const int n_range = A.sum_out ? (M + range - 1) / range : A.n;
    for (int l = top; l >= 0; --l) {
        const float *u = l ? A.x[l - 1] : nullptr;
        const Args gy{M, H, 2,
                      {{A.da, A.pk + A.f.WaT[l], nullptr, H, H, H, H}, {A.dg, A.pk + A.f.WgT[l], nullptr, H, H, H, H}}};
        if ((e = launch<false>(gy, EpiStore{A.dy, H}, A.en, st))) return e;
        const Args gh{M, H, 1, {{A.dy, A.pk + A.f.CreT[l], A.pk + A.f.CimT[l], H, H, H, H}}};
        if ((e = launch<true>(gh, EpiDh{A.dhr, A.dhi, H}, A.en, st))) return e;
        if (l) lru_scan_bwd_kernel<false><<<scan_blocks, 128, 0, st>>>(A, l);
        else lru_scan_bwd_kernel<true><<<scan_blocks, 128, 0, st>>>(A, l);
        if ((e = cudaGetLastError())) return e;
        WgArgs w{};
        w.n_pair = l ? 6 : 4;
        w.p[0] = Pair{A.da, A.y[l], H, H, H, H, H, M, tl.Wa[l], H, tl.ba[l]};
        w.p[1] = Pair{A.dg, A.y[l], H, H, H, H, H, M, tl.Wg[l], H, tl.bg[l]};
        w.p[2] = Pair{A.dy, A.hr[l], H, H, H, H, H, M, tl.Cre[l], H, -1};
        w.p[3] = Pair{A.dy, A.hn[l], H, H, H, H, H, M, tl.Cim[l], H, -1};
        if (l) {
            w.p[4] = Pair{A.dhr, u, H, H, H, H, H, M, tl.Bre[l], H, -1};
            w.p[5] = Pair{A.dhi, u, H, H, H, H, H, M, tl.Bim[l], H, -1};
        }
        w.n_range = n_range;
        w.len = w.step = w.seg_len = w.seg_stride = range;
        w.out = A.rows;
        w.out_stride = tl.total;
        if ((e = launch_wgrad(w, A.en, st))) return e;
        if (l) {
            const Args gx{M, H, 2,
                          {{A.dhr, A.pk + A.f.BreT[l], nullptr, H, H, H, H}, {A.dhi, A.pk + A.f.BimT[l], nullptr, H, H, H, H}}};
            const EpiGx ex{A.pk + A.f.D[l], A.dy, A.p1[l - 1], A.p2[l - 1], A.gx, A.da, A.dg, H};
            if ((e = launch<false>(gx, ex, A.en, st))) return e;
        }
    }
    if (!A.sum_out) return cudaSuccess;
    SumArgs sa{};
    sa.add = A.add;
    sa.out = A.sum_out;
    auto part = [&](int64_t off, int64_t len) { sa.s[sa.n++] = SumSeg{A.rows + off, tl.total, off, n_range, (int)len}; };
    auto small = [&](int64_t src, int64_t dst, int len) {
        sa.s[sa.n++] = SumSeg{A.small + src, A.small_stride, dst, A.n, len};
    };
    for (int l = 0; l < nL; ++l) {
        if (l) part(tl.Bre[l], 4 * (int64_t)H * H);
        else part(tl.Cre[0], 2 * (int64_t)H * H);
        part(tl.Wa[l], 2 * (int64_t)H * H + 2 * H);
        small(A.sm.nu[l], tl.nu[l], 3 * H);
        small(A.sm.D[l], tl.D[l], l ? H : 2 * H);
    }
    small(A.sm.Bre0, tl.Bre[0], 4 * H);
    small(A.sm.Wo, tl.Wo, 2 * H);
    small(A.sm.bo, tl.bo, 2);
    return launch_sum_rows(sa, st);
}

}  // namespace psr
