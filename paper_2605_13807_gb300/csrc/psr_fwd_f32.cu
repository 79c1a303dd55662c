// FP32 SIMT forward of the PSR-NQS ansatz (the plain path), parameter
// packing and spin bit-packing.
//
// One CTA of H threads evaluates one sequence at a time (thread j owns hidden
// unit j) and walks it chunk by chunk (32 sites).  Inside a chunk:
//   layer 0  : gates from lookup tables of the one-hot input onehot(s_{t-1})
//              (Sec. II.F: zero input at the first site), the recurrence
//              h_t = a_t h_{t-1} + b_t (Sec. II.C) carried in a register,
//              then x^(1) = GELU(C h + D u) (Sec. II.F-G);
//   layer l>0: z = W_z x + b_z, h~ = W_h x + b_h (FP32 FMA over a shared-memory
//              tile), a = sigmoid(z), b = (1 - a) h~, the same scan, and
//              x^(l+1) = GELU(C h + D x + [l >= 2] h^(l-1));
//   readout  : d_t = (W_o[1] - W_o[0]) x_t + (b_o[1] - b_o[0]) and
//              log P(s_t) = -softplus(-+d_t) (two-way softmax), summed over
//              sites; log psi = 1/2 sum_t log P (Sec. III.B).
// The scan carry of each layer crosses chunk boundaries in shared memory, so
// a sequence needs no inter-CTA communication; jobs are handed out by an
// atomic counter for load balance over ragged sequence lengths.
#include <cuda_runtime.h>

#include "psr_device.cuh"
#include "psr_internal.cuh"

namespace psr {

ThetaLayout theta_layout(int nL, int H) {
    ThetaLayout t{};
    t.nL = nL;
    t.H = H;
    int64_t off = 0;
    for (int l = 0; l < nL; ++l) {
        int64_t din = (l == 0) ? 2 : H;
        t.Wz[l] = off; off += H * din;
        t.bz[l] = off; off += H;
        t.Wh[l] = off; off += H * din;
        t.bh[l] = off; off += H;
        t.C[l] = off;  off += (int64_t)H * H;
        t.D[l] = off;  off += H * din;
    }
    t.Wo = off; off += 2 * H;
    t.bo = off; off += 2;
    t.total = off;
    return t;
}

F32Layout f32_layout(int nL, int H) {
    F32Layout f{};
    f.nL = nL;
    f.H = H;
    int64_t off = 0;
    for (int l = 0; l < nL; ++l) {
        int64_t din = (l == 0) ? 2 : H;
        f.WzT[l] = off; off += din * H;
        f.WhT[l] = off; off += din * H;
        f.CT[l] = off;  off += (int64_t)H * H;
        f.DT[l] = off;  off += din * H;
        f.bz[l] = off;  off += H;
        f.bh[l] = off;  off += H;
    }
    f.A0 = off;  off += 3 * H;
    f.B0 = off;  off += 3 * H;
    f.DU0 = off; off += 3 * H;
    f.CD0 = off; off += 3 * H;
    f.wd = off;  off += H;
    f.bd = off;  off += 4;
    f.total = off;
    return f;
}

// One thread per packed element, so that every read of theta is in flight at
// once (a loop over layers and tensors paid the latency of each: 9 us at any
// width, 3 us so).
__device__ __forceinline__ void pack_f32_element(const float *__restrict__ theta, const ThetaLayout &tl,
                                                 const F32Layout &fl, float *__restrict__ pk, int i) {
    const int H = tl.H;
    if (i >= fl.total) return;
    // tensors of a layer in packed order; the tables and readout follow
    if (i < fl.A0) {
        int l = 0;
        while (l + 1 < tl.nL && i >= fl.WzT[l + 1]) ++l;
        const int din = l == 0 ? 2 : H, m = din * H;
        int r = i - (int)fl.WzT[l];
        int64_t src = tl.Wz[l];
        int rows = din;
        if (r >= m) { r -= m; src = tl.Wh[l];
            if (r >= m) { r -= m; src = tl.C[l]; rows = H;
                if (r >= H * H) { r -= H * H; src = tl.D[l]; rows = din;
                    if (r >= m) { r -= m; rows = 0; src = tl.bz[l];
                        if (r >= H) { r -= H; src = tl.bh[l]; } } } } }
        pk[i] = rows == 0 ? theta[src + r] : theta[src + (int64_t)(r % H) * rows + r / H];
        return;
    }
    if (i < fl.wd) {
        int r = i - (int)fl.A0;
        const int table = r / (3 * H);  // A0, B0, DU0, CD0
        r %= 3 * H;
        const int code = r / H, j = r % H;
        float zp = theta[tl.bz[0] + j];
        float cd = theta[tl.bh[0] + j];
        float du = 0.0f;
        if (code > 0) {
            zp += theta[tl.Wz[0] + 2 * j + (code - 1)];
            cd += theta[tl.Wh[0] + 2 * j + (code - 1)];
            du = theta[tl.D[0] + 2 * j + (code - 1)];
        }
        const float a = sigmoid_f(zp);
        pk[i] = table == 0 ? a : table == 1 ? (1.0f - a) * cd : table == 2 ? du : cd;
        return;
    }
    if (i < fl.bd) {
        const int j = i - (int)fl.wd;
        pk[i] = theta[tl.Wo + H + j] - theta[tl.Wo + j];
    } else if (i == fl.bd) {
        pk[i] = theta[tl.bo + 1] - theta[tl.bo];
    }
}

__global__ void __launch_bounds__(256) pack_f32_kernel(const float *__restrict__ theta, ThetaLayout tl, F32Layout fl,
                                                       float *__restrict__ pk) {
    pack_f32_element(theta, tl, fl, pk, blockIdx.x * 256 + threadIdx.x);
}

cudaError_t launch_pack_theta_f32(const float *theta, const ThetaLayout &tl, const F32Layout &fl,
                                  float *packed, cudaStream_t stream) {
    pack_f32_kernel<<<(unsigned)((fl.total + 255) / 256), 256, 0, stream>>>(theta, tl, fl, packed);
    return cudaGetLastError();
}

// One warp per 64-bit word (two ballots over coalesced bytes); a byte other
// than 0/1 is reported as PSR_EDEVICE and treated as its lowest bit.  Words past
// N are zero.  The first thread also zeroes n_zero counters for a kernel that
// follows (a launch less than a memset).
__device__ __forceinline__ void bitpack_words(const uint8_t *__restrict__ spins, int64_t n, int N, int W,
                                              uint64_t *__restrict__ bits, int *status, unsigned long long *zero,
                                              int n_zero, int block, int blocks) {
    const int lane = threadIdx.x & 31;
    if (block == 0 && threadIdx.x < n_zero) zero[threadIdx.x] = 0;
    const int64_t total = n * W, warps = (int64_t)blocks * 8;
    for (int64_t i = (int64_t)block * 8 + (threadIdx.x >> 5); i < total; i += warps) {
        const int64_t s = i / W;
        const int t = (int)(i - s * W) * 64 + lane;
        const uint8_t *row = spins + s * N;
        const unsigned v0 = t < N ? row[t] : 0u, v1 = t + 32 < N ? row[t + 32] : 0u;
        const unsigned lo = __ballot_sync(0xffffffffu, v0 & 1u), hi = __ballot_sync(0xffffffffu, v1 & 1u);
        if ((v0 | v1) > 1u) set_status(status, PSR_EDEVICE);
        if (lane == 0) bits[i] = (uint64_t)lo | (uint64_t)hi << 32;
    }
}

__global__ void __launch_bounds__(256) bitpack_kernel(const uint8_t *__restrict__ spins, int64_t n, int N, int W,
                                                      uint64_t *__restrict__ bits, int *status,
                                                      unsigned long long *zero, int n_zero) {
    bitpack_words(spins, n, N, W, bits, status, zero, n_zero, blockIdx.x, gridDim.x);
}

static int bitpack_blocks(int64_t n, int W) {
    const int64_t blocks = (n * W + 7) / 8;
    return (int)(blocks > 65535 ? 65535 : blocks);
}

cudaError_t launch_bitpack(const uint8_t *spins, int64_t n, int N, int W, uint64_t *bits,
                           int *status, cudaStream_t stream, unsigned long long *zero, int n_zero) {
    bitpack_kernel<<<bitpack_blocks(n, W), 256, 0, stream>>>(spins, n, N, W, bits, status, zero, n_zero);
    return cudaGetLastError();
}

// Both packings in one launch: the first blocks take the parameters, the others
// the spins.  A small gradient is a row of launches of about 4 us, whatever they do.
__global__ void __launch_bounds__(256) pack_f32_bits_kernel(const float *__restrict__ theta, ThetaLayout tl,
                                                            F32Layout fl, float *__restrict__ pk, int theta_blocks,
                                                            const uint8_t *__restrict__ spins, int64_t n, int N, int W,
                                                            uint64_t *__restrict__ bits, int *status) {
    const int b = (int)blockIdx.x - theta_blocks;
    if (b < 0) pack_f32_element(theta, tl, fl, pk, blockIdx.x * 256 + threadIdx.x);
    else bitpack_words(spins, n, N, W, bits, status, nullptr, 0, b, gridDim.x - theta_blocks);
}

cudaError_t launch_pack_f32_bits(const float *theta, const ThetaLayout &tl, const F32Layout &fl, float *packed,
                                 const uint8_t *spins, int64_t n, int N, int W, uint64_t *bits, int *status,
                                 cudaStream_t stream) {
    const int tb = (int)((fl.total + 255) / 256);
    pack_f32_bits_kernel<<<tb + bitpack_blocks(n, W), 256, 0, stream>>>(theta, tl, fl, packed, tb, spins, n, N, W, bits,
                                                                       status);
    return cudaGetLastError();
}

// ------------------------------------------------------------- forward
// A job is one sequence; the threads of its CTA own one unit each and walk it in
// windows of 32 or 16 sites (CW).
//
// What bounds it: shared memory and the FP32 rate, about equally.  A thread
// keeps CW sums of both gates, so a row of the window (CW / 4 16-byte
// broadcasts) and two weights serve 2 CW multiply-adds, done in pairs of sites
// (fma.rn.f32x2, half the instructions).  A job's CTA is one warp per 32 units;
// seven jobs per SM overlap.  Two units a thread (measured, not kept) halve the
// shared-memory reads but leave half the warps: 7.8 ms against 6.7 ms at hidden 64, 2 to 4 % better
// to twice as slow at hidden 128 (few long sequences).
// Measured (E_loc of the 100-site periodic Heisenberg chain, hidden 64, 1024
// samples): 6.7 ms; 12.0 ms with 32-site windows counted from site 0, plain
// multiply-adds and unrolled gate functions.
//
// Windows.  Chunk boundaries lie on multiples of 16 sites counted from the END
// of the sequence (off = sites the first chunk starts before site 0), or from
// its start (align_start: the carries of the chunk-recompute gradient).  A
// connected configuration resumes at the boundary before its first flipped
// site: with 32-site windows from site 0, a 100-site chain evaluated 94 sites
// per configuration where 50 are needed (28 of them past the end, in the last
// window); boundaries from the end waste 8 on average.  An odd number of
// chunks starts with one window of 16 sites.
namespace {

__device__ __forceinline__ void ffma2(uint64_t &d, uint64_t a, uint64_t b) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}
__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
    uint64_t v;
    asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(lo), "f"(hi));
    return v;
}
__device__ __forceinline__ float lo2(uint64_t v) { return __uint_as_float((uint32_t)v); }
__device__ __forceinline__ float hi2(uint64_t v) { return __uint_as_float((uint32_t)(v >> 32)); }

// Bits of sites [t0, t0 + 32) and of site t0 - 1, flips p and q applied; t0
// may be negative or unaligned, sites outside [0, N) read as 0.
__device__ __forceinline__ void window_bits(const uint64_t *row, int N, int t0, int p, int q, uint32_t &cur,
                                            uint32_t &prev) {
    const int b = max(t0, 0);
    uint64_t v = row[b >> 6] >> (b & 63);
    if (b & 63) v |= row[(b >> 6) + 1] << (64 - (b & 63));  // rows end with a zero word
    cur = (uint32_t)v << (b - t0);
    if (t0 + 32 > N) cur &= t0 < N ? 0xffffffffu >> (t0 + 32 - N) : 0u;
    prev = t0 > 0 ? (uint32_t)(row[(t0 - 1) >> 6] >> ((t0 - 1) & 63)) & 1u : 0u;
#pragma unroll
    for (int f = 0; f < 2; ++f) {
        const int x = f ? q : p;
        if (x < 0) continue;
        if (x >= t0 && x < t0 + 32) cur ^= 1u << (x - t0);
        else if (x == t0 - 1) prev ^= 1u;
    }
}

struct FwdF32Job {
    const uint64_t *row;
    float *carries;  // of this job's chunk 0 (mode 0, or null): [nch][nL][H]
    float *logp_out;
    const float *logp_ref;
    int N, u1, p, q;
};

constexpr int LD = 36;  // row of a tile: 32 sites, 16-byte aligned

// a job is one CTA of H threads
template <int H>
__device__ __forceinline__ void job_sync() {
    if constexpr (H == 32) __syncwarp();
    else __syncthreads();
}

// y += w[k][this thread's unit] x[k] over a window's pairs of sites, k = 0 .. H - 1,
// for NM (weights, tile, sums) triples at once; the weights (coalesced over units)
// of the next K inner units are fetched while K are used.
template <int H, int CW, int NM>
__device__ __forceinline__ void products(const float *const (&w)[NM], const float *const (&tile)[NM],
                                         uint64_t *const (&y)[NM]) {
    constexpr int P = CW / 2;
    // K = 4 leaves the code of the narrow model small enough for jobs out of step
    constexpr int K = H == 32 ? 4 : 8;
    float nw[NM][K];
    auto fetch = [&](int k0) {
#pragma unroll
        for (int m = 0; m < NM; ++m)
#pragma unroll
            for (int k = 0; k < K; ++k) nw[m][k] = w[m][(k0 + k) * H];
    };
    fetch(0);
#pragma unroll 1
    for (int k0 = 0; k0 < H; k0 += K) {
        uint64_t cw[NM][K];
#pragma unroll
        for (int m = 0; m < NM; ++m)
#pragma unroll
            for (int k = 0; k < K; ++k) cw[m][k] = pack2(nw[m][k], nw[m][k]);
        if (k0 + K < H) fetch(k0 + K);
#pragma unroll
        for (int k = 0; k < K; ++k) {
#pragma unroll
            for (int q = 0; q < P / 2; ++q) {
                ulonglong2 v;
#pragma unroll
                for (int m = 0; m < NM; ++m) {
                    if (m == 0 || tile[m] != tile[0])
                        v = *reinterpret_cast<const ulonglong2 *>(tile[m] + (k0 + k) * LD + 4 * q);
                    ffma2(y[m][2 * q], cw[m][k], v.x);
                    ffma2(y[m][2 * q + 1], cw[m][k], v.y);
                }
            }
        }
    }
}

// One window of CW sites starting at t0 (chunk c): x of the last layer's sites
// through the readout; returns this thread's share of the sum of log P.
template <int H, int CW>
__device__ __forceinline__ float window(const FwdF32Job &J, const float *__restrict__ pk, const F32Layout &fl,
                                        float *xs, float *hs, float *zs, float *hcar, int t0, int c,
                                        int &n_up) {
    constexpr int P = CW / 2;
    const int j = threadIdx.x, nL = fl.nL;  // j: this thread's unit
    uint32_t cur, prev;
    window_bits(J.row, J.N, t0, J.p, J.q, cur, prev);
    if (CW < 32) cur &= (1u << CW) - 1u;
    const uint32_t prevbits = (cur << 1) | prev;  // bit t = s_{t0+t-1}
    const int first = max(0, -t0);                // sites before the sequence: no input, no state

    uint64_t y[P];
    // scan of the unit: h_t from a_t and c_t (or b_t), written to its row of
    // hs; y starts from the unit's old row (the layer below's states) if kept
    auto put_carry = [&](int l, int chunk, float h) {
        if (J.carries) J.carries[((int64_t)chunk * nL + l) * H + j] = h;
    };
    // ---------------- layer 0: gates by lookup of the one-hot input
    {
        float a[3], b[3], d[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            a[q] = pk[fl.A0 + q * H + j];
            b[q] = pk[fl.B0 + q * H + j];
            d[q] = pk[fl.DU0 + q * H + j];
        }
        float h = hcar[j];
        put_carry(0, c, h);
#pragma unroll
        for (int t = 0; t < CW; t += 4) {
            float hv[4], dv[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int tt = t + e;
                if (CW == 32 && tt == 16) put_carry(0, c + 1, h);
                const bool up = (prevbits >> tt) & 1u;
                const bool start = t0 + tt == 0;
                const float hn = (start ? a[0] : up ? a[2] : a[1]) * h + (start ? b[0] : up ? b[2] : b[1]);
                h = tt < first ? 0.0f : hn;
                hv[e] = h;
                dv[e] = start ? d[0] : up ? d[2] : d[1];
            }
            *reinterpret_cast<float4 *>(hs + j * LD + t) = make_float4(hv[0], hv[1], hv[2], hv[3]);
            y[t / 2] = pack2(dv[0], dv[1]);
            y[t / 2 + 1] = pack2(dv[2], dv[3]);
        }
        hcar[j] = h;
    }
    job_sync<H>();
    products<H, CW, 1>({pk + fl.CT[0] + j}, {hs}, {y});
    // The element-wise functions run in rolled loops over the thread's own row
    // in shared memory: unrolled over the register arrays their code (some 40
    // instructions a site) outgrew the instruction cache as soon as the jobs of
    // an SM were out of step (connected configurations: 13.4 against 7 ms).
    auto put_row = [&](float *tile, const uint64_t (&v)[P]) {
#pragma unroll
        for (int q = 0; q < P / 2; ++q)
            *reinterpret_cast<ulonglong2 *>(tile + j * LD + 4 * q) = make_ulonglong2(v[2 * q], v[2 * q + 1]);
    };
    auto map_row = [&](float *tile, auto f) {
#pragma unroll 1
        for (int i = 0; i < CW / 4; ++i) {
            float4 *p = reinterpret_cast<float4 *>(tile + j * LD + 4 * i);
            const float4 v = *p;
            *p = make_float4(f(v.x), f(v.y), f(v.z), f(v.w));
        }
    };
    auto store_x = [&]() {
        put_row(xs, y);
        map_row(xs, [](float v) { return gelu_f(v); });
    };
    store_x();
    job_sync<H>();

    for (int l = 1; l < nL; ++l) {
        uint64_t z[P];
        const float bz = pk[fl.bz[l] + j], bh = pk[fl.bh[l] + j];
#pragma unroll
        for (int q = 0; q < P; ++q) {
            z[q] = pack2(bz, bz);
            y[q] = pack2(bh, bh);
        }
        products<H, CW, 2>({pk + fl.WzT[l] + j, pk + fl.WhT[l] + j}, {xs, xs}, {z, y});
        put_row(zs, z);
        map_row(zs, [](float v) { return sigmoid_f(v); });
        // scan: this unit's row of hs turns from h of the layer below (the
        // residual of l >= 2, which y starts from) into h of this layer
        {
            float h = hcar[l * H + j];
            put_carry(l, c, h);
            float *row = hs + j * LD;
#pragma unroll
            for (int t = 0; t < CW; t += 4) {
                const float4 below = *reinterpret_cast<const float4 *>(row + t);
                const float4 gate = *reinterpret_cast<const float4 *>(zs + j * LD + t);
                const float av[4] = {gate.x, gate.y, gate.z, gate.w};
                float hv[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int tt = t + e;
                    if (CW == 32 && tt == 16) put_carry(l, c + 1, h);
                    const uint64_t c2 = y[tt / 2];
                    const float a = av[e];
                    const float hn = a * h + (1.0f - a) * (tt & 1 ? hi2(c2) : lo2(c2));
                    h = tt < first ? 0.0f : hn;
                    hv[e] = h;
                }
                *reinterpret_cast<float4 *>(row + t) = make_float4(hv[0], hv[1], hv[2], hv[3]);
                y[t / 2] = l >= 2 ? pack2(below.x, below.y) : 0;
                y[t / 2 + 1] = l >= 2 ? pack2(below.z, below.w) : 0;
            }
            hcar[l * H + j] = h;
        }
        job_sync<H>();
        products<H, CW, 2>({pk + fl.CT[l] + j, pk + fl.DT[l] + j}, {hs, xs}, {y, y});
        job_sync<H>();
        store_x();
        job_sync<H>();
    }

    // readout: lane t of the first warp handles site t0 + t
    float v = 0.0f;
    if (j < CW) {
        const int t = j, tt = t0 + t;
        if (tt >= 0 && tt < J.N) {
            float d[4] = {pk[fl.bd], 0.0f, 0.0f, 0.0f};  // four chains: the sum is latency-bound
            const float *wd = pk + fl.wd;
#pragma unroll 2
            for (int k = 0; k < H; k += 4)
#pragma unroll
                for (int e = 0; e < 4; ++e) d[e] = fmaf(wd[k + e], xs[(k + e) * LD + t], d[e]);
            const int s = (cur >> t) & 1u;
            const int nu = n_up + __popc(cur & ((1u << t) - 1u));
            const float lp = site_logp((d[0] + d[1]) + (d[2] + d[3]), s, u1_forced(J.u1, J.N, tt, nu));
            if (J.logp_out) J.logp_out[tt] = lp;
            v = J.logp_ref ? lp - J.logp_ref[tt] : lp;
        }
    }
    n_up += __popc(cur);
    job_sync<H>();
    return v;
}

}  // namespace

// kWide: windows of 32 sites (after one of 16 if the chunks are odd in
// number); else 16.
template <int H, bool kWide>
__global__ void __launch_bounds__(H) fwd_f32_kernel(const __grid_constant__ FwdJobs jb,
                                                                    const float *__restrict__ pk, F32Layout fl,
                                                                    bool align_start) {
    constexpr int CH = kChunkGrad;
    extern __shared__ __align__(16) float smem[];
    float *xs = smem;              // [H][LD] layer input / output
    float *hs = xs + H * LD;       // [H][LD] hidden states of the window
    float *zs = hs + H * LD;       // [H][LD] gates of the window
    float *hcar = zs + H * LD;     // [nL][H] scan carries
    __shared__ long long s_job;
    const int j = threadIdx.x, nL = fl.nL;
    long long base[kMaxGroups + 1];
    base[0] = 0;
    for (int i = 0; i < jb.n_groups; ++i)
        base[i + 1] = base[i] + (jb.mode == 1 ? (long long)*jb.g[i].n_jobs_dev : (long long)jb.g[i].n_jobs);
    for (;;) {
        job_sync<H>();
        if (j == 0) s_job = (long long)atomicAdd((unsigned long long *)jb.job_counter, 1ull);
        job_sync<H>();
        const long long job = s_job;
        if (job >= base[jb.n_groups]) break;
        int gi = 0;
        while (gi + 1 < jb.n_groups && job >= base[gi + 1]) ++gi;
        const FwdGroup &G = jb.g[gi];
        const long long lj = job - base[gi];
        const int N = G.N, nch = (N + CH - 1) / CH;
        const int off = align_start ? 0 : nch * CH - N;

        int sample, c0 = 0;
        FwdF32Job J{};
        J.p = J.q = -1;
        if (jb.mode == 0) {
            sample = (int)lj;
        } else {
            const int32_t *e = G.entries + 3 * lj;
            sample = e[0];
            J.p = e[1];
            J.q = e[2];
            c0 = (J.p + off) / CH;
        }
        J.row = G.bits + (int64_t)sample * G.W;
        J.N = N;
        J.u1 = G.u1;
        J.carries = G.carries_out ? G.carries_out + (int64_t)sample * nch * nL * H : nullptr;
        J.logp_out = G.logp_out ? G.logp_out + (int64_t)sample * N : nullptr;
        J.logp_ref = jb.mode == 1 ? G.logp_ref + (int64_t)sample * N : nullptr;
        for (int l = 0; l < nL; ++l)
            hcar[l * H + j] = c0 == 0 ? 0.0f : G.carries_in[(((int64_t)sample * nch + c0) * nL + l) * H + j];
        int n_up = G.u1 ? count_up_before(J.row, max(c0 * CH - off, 0)) : 0;
        float acc = 0.0f;
        int c = c0;
        if (!kWide || ((nch - c) & 1)) {
            do {
                acc += window<H, 16>(J, pk, fl, xs, hs, zs, hcar, c * CH - off, c, n_up);
                ++c;
            } while (!kWide && c < nch);
        }
        if constexpr (kWide)
            for (; c < nch; c += 2) acc += window<H, 32>(J, pk, fl, xs, hs, zs, hcar, c * CH - off, c, n_up);
        if (j < 32) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
            if (j == 0) G.out[lj] = 0.5f * acc;
        }
    }
}

template <int H, bool kWide>
static cudaError_t launch_fwd_f32_h(const FwdJobs &jobs, const float *packed, const F32Layout &fl,
                                    int num_sms, cudaStream_t stream, bool align_start) {
    const size_t smem = (size_t)(3 * H * LD + fl.nL * H) * sizeof(float);
    cudaError_t e = cudaFuncSetAttribute(fwd_f32_kernel<H, kWide>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fwd_f32_kernel<H, kWide>, H, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) per_sm = 1;
    int64_t grid = (int64_t)num_sms * per_sm;
    const int64_t nj = max_jobs(jobs);
    if (nj < grid) grid = nj;
    if (grid < 1) grid = 1;
    fwd_f32_kernel<H, kWide><<<(int)grid, H, smem, stream>>>(jobs, packed, fl, align_start);
    return cudaGetLastError();
}

cudaError_t launch_fwd_f32(const FwdJobs &jobs, const float *packed, const F32Layout &fl, int num_sms,
                           cudaStream_t stream, int chunk, bool align_start) {
    if (chunk != kChunkF32 && chunk != kChunkGrad) return cudaErrorInvalidValue;
    const bool wide = chunk == kChunkF32;
    switch (fl.H) {
        case 32:
            return wide ? launch_fwd_f32_h<32, true>(jobs, packed, fl, num_sms, stream, align_start)
                        : launch_fwd_f32_h<32, false>(jobs, packed, fl, num_sms, stream, align_start);
        case 64:
            return wide ? launch_fwd_f32_h<64, true>(jobs, packed, fl, num_sms, stream, align_start)
                        : launch_fwd_f32_h<64, false>(jobs, packed, fl, num_sms, stream, align_start);
        case 128:
            return wide ? launch_fwd_f32_h<128, true>(jobs, packed, fl, num_sms, stream, align_start)
                        : launch_fwd_f32_h<128, false>(jobs, packed, fl, num_sms, stream, align_start);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace psr
