// Matrix products of the layer-by-layer gradients with FP32 multiply-adds (CUDA
// cores): the site-major arrays [site][unit] of a whole batch of samples
// against weight matrices, and the weight gradients as products over the sites.
// They serve the FP32 O_k rows, width 32 and the 2D weight gradients;
// psr_gemm_tc.cuh holds the tensor-core form of the same contract.
//
// Why this form: a thread that owns one hidden unit of a few sites (the shape
// of a kernel that walks one sample per CTA) reads one shared-memory float for
// every one or two multiply-adds, which bounds it by shared memory at a fifth
// of the FP32 rate.  Here a thread owns 8 x 8 outputs and reads 16 floats for
// 64 multiply-adds, and a CTA tile of 128 sites serves every weight it loads
// to 128 sites: 33 to 45 TFLOP/s for the products, 47 to 52 for the weight
// gradients, of 80.  Neither the FP32 pipe (57 %) nor shared memory (50 %) is
// full; pairs of multiply-adds (fma.rn.f32x2), a third stage and 4 x 8 outputs
// a thread measured the same or slower.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace psr {
namespace gemm {

constexpr int BM = 128;        // sites per CTA tile
constexpr int BK = 32;         // inner elements per stage; every inner size is a multiple of it
constexpr int LDT = BK + 4;    // shared row: 9 x 16 bytes, so 8 consecutive rows hit 8 bank groups
constexpr int kMaxSeg = 3;

__device__ __forceinline__ void cp16(void *dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
// 16 bytes of src, or zeros
__device__ __forceinline__ void cp16_or_zero(void *dst, const void *src, bool take) {
    const int n = take ? 16 : 0;
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)),
                 "l"(src), "r"(n)
                 : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int K>
__device__ __forceinline__ void cp_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(K) : "memory");
}

// out[m][n] = sum over segments sum_k A[m][k] W[n][k]: both operands with the
// inner index contiguous (16-byte aligned rows).  With pairs, output unit u
// has two rows, W0[u] and W1[u], and one thread ends with both.
struct Seg {
    const float *A, *W0, *W1;
    int K, lda, ldw, ldw1;
};
struct Args {
    int M;      // sites
    int units;  // output units (columns, or pairs of columns)
    int n_seg;
    Seg seg[kMaxSeg];
};

// two stages; the epilogue's tile of BM x (BN + 8) floats reuses them
constexpr size_t smem_bytes(int BN) { return (size_t)2 * (BM + BN) * LDT * sizeof(float); }
constexpr int threads(int BN) { return BN == 128 ? 256 : 128; }

// BN columns per tile (a pair is two).  A warp covers 4 x 8 lanes; lane
// (ty, tx) of warp (wm, wn) owns sites 16 i + 4 wm + ty and columns 64 wn + tx
// + 8 j.  Epi: load(m, u) -> what the four units u .. u + 3 of site m need
// from memory, then store(m, u, values[, second values], loaded).
template <int BN, bool kPair, class Epi>
__global__ void __launch_bounds__(threads(BN), BN == 128 ? 2 : 4)
    gemm_kernel(const __grid_constant__ Args g, const __grid_constant__ Epi epi) {
    constexpr int T = threads(BN);
    constexpr int TN = BN == 32 ? 4 : 8;
    extern __shared__ __align__(16) float smem[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int tx = lane & 7, ty = lane >> 3;
    const int wn = BN == 128 ? (warp & 1) : 0, wm = BN == 128 ? (warp >> 1) : warp;
    const int nblk = g.units * (kPair ? 2 : 1) / BN;
    const int m0 = (int)(blockIdx.x / nblk) * BM;
    const int u0 = (int)(blockIdx.x % nblk) * (kPair ? BN / 2 : BN);
    const int lrow = tid >> 3, lcol = (tid & 7) * 4;  // copies: 8 lanes cover 32 floats of a row

    float acc[8][TN];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j] = 0.0f;

    int s_next = 0, k_next = 0;  // the stage to be requested next
    auto request = [&](int slot) {
        if (s_next < g.n_seg) {
            const Seg &s = g.seg[s_next];
            float *as = smem + (size_t)slot * (BM + BN) * LDT, *ws = as + BM * LDT;
#pragma unroll
            for (int r = 0; r < BM; r += T / 8) {
                const int m = min(m0 + lrow + r, g.M - 1);  // rows past the end repeat the last (not stored)
                cp16(as + (lrow + r) * LDT + lcol, s.A + (size_t)m * s.lda + k_next + lcol);
            }
#pragma unroll
            for (int r = 0; r < BN; r += T / 8) {
                const int n = lrow + r;
                if (BN < T / 8 && n >= BN) break;
                const float *w = s.W0 + (size_t)(u0 + n) * s.ldw;
                if constexpr (kPair) {
                    const size_t u = u0 + (n & 7) + 8 * (n >> 4);
                    w = n & 8 ? s.W1 + u * s.ldw1 : s.W0 + u * s.ldw;
                }
                cp16(ws + n * LDT + lcol, w + k_next + lcol);
            }
            k_next += BK;
            if (k_next >= s.K) {
                k_next = 0;
                ++s_next;
            }
        }
        cp_commit();
    };
    int stages = 0;
    for (int s = 0; s < g.n_seg; ++s) stages += g.seg[s].K / BK;
    request(0);
    for (int st = 0; st < stages; ++st) {
        request((st + 1) & 1);
        cp_wait<1>();
        __syncthreads();
        const float *as = smem + (size_t)(st & 1) * (BM + BN) * LDT + (4 * wm + ty) * LDT;
        const float *ws = smem + (size_t)(st & 1) * (BM + BN) * LDT + BM * LDT + (64 * wn + tx) * LDT;
#pragma unroll 2
        for (int k = 0; k < BK; k += 4) {
            float4 b[TN];
#pragma unroll
            for (int j = 0; j < TN; ++j) b[j] = *reinterpret_cast<const float4 *>(ws + 8 * j * LDT + k);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const float4 a = *reinterpret_cast<const float4 *>(as + 16 * i * LDT + k);
#pragma unroll
                for (int j = 0; j < TN; ++j) {
                    acc[i][j] = fmaf(a.x, b[j].x, acc[i][j]);
                    acc[i][j] = fmaf(a.y, b[j].y, acc[i][j]);
                    acc[i][j] = fmaf(a.z, b[j].z, acc[i][j]);
                    acc[i][j] = fmaf(a.w, b[j].w, acc[i][j]);
                }
            }
        }
        __syncthreads();
    }
    // The tile goes through shared memory, so that the epilogue reads and
    // writes whole rows (16 bytes a lane) and the reads of kRows rows are in
    // flight together; straight from the registers (32-byte pieces, one row
    // after another) the epilogues that read arrays took up to twice as long.
    constexpr int C = kPair ? BN / 2 : BN;  // units of the tile
    constexpr int LDC = BN + 8;             // 8 x 4 lanes of a store hit 32 banks
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        float *row = smem + (16 * i + 4 * wm + ty) * LDC;
#pragma unroll
        for (int j = 0; j < TN; ++j) {
            if constexpr (kPair) row[(j & 1) * C + 32 * wn + 8 * (j >> 1) + tx] = acc[i][j];
            else row[64 * wn + 8 * j + tx] = acc[i][j];
        }
    }
    __syncthreads();
    constexpr int kQuads = C / 4, kStep = T / kQuads, kRows = 4;
    static_assert(BM % (kStep * kRows) == 0, "whole groups of rows");
    const int q = (tid % kQuads) * 4, r0 = tid / kQuads;
    const int u = u0 + q;
#pragma unroll 1
    for (int r = r0; r < BM; r += kStep * kRows) {
        typename Epi::In in[kRows];
#pragma unroll
        for (int k = 0; k < kRows; ++k) in[k] = epi.load(min(m0 + r + k * kStep, g.M - 1), u);
#pragma unroll
        for (int k = 0; k < kRows; ++k) {
            const int m = m0 + r + k * kStep;
            if (m >= g.M) break;
            const float *row = smem + (r + k * kStep) * LDC + q;
            const float4 v = *reinterpret_cast<const float4 *>(row);
            if constexpr (kPair) epi.store(m, u, v, *reinterpret_cast<const float4 *>(row + C), in[k]);
            else epi.store(m, u, v, in[k]);
        }
    }
}

// element-wise helpers of the epilogues, four units at a time
__device__ __forceinline__ float4 ld4(const float *p) { return *reinterpret_cast<const float4 *>(p); }
__device__ __forceinline__ void st4(float *p, float4 v) { *reinterpret_cast<float4 *>(p) = v; }
template <class F>
__device__ __forceinline__ float4 map4(F f, float4 a) {
    return make_float4(f(a.x), f(a.y), f(a.z), f(a.w));
}
template <class F>
__device__ __forceinline__ float4 map4(F f, float4 a, float4 b) {
    return make_float4(f(a.x, b.x), f(a.y, b.y), f(a.z, b.z), f(a.w, b.w));
}
__device__ __forceinline__ float4 add4(float4 a, float4 b) {
    return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w);
}
__device__ __forceinline__ float4 mul4(float4 a, float4 b) {
    return make_float4(a.x * b.x, a.y * b.y, a.z * b.z, a.w * b.w);
}
__device__ __forceinline__ float4 fma4(float4 a, float4 b, float4 c) {
    return make_float4(fmaf(a.x, b.x, c.x), fmaf(a.y, b.y, c.y), fmaf(a.z, b.z, c.z), fmaf(a.w, b.w, c.w));
}

struct NoIn {};

struct EpiStore {  // out = the product
    using In = NoIn;
    float *out;
    int H;
    __device__ NoIn load(int, int) const { return {}; }
    __device__ void store(int m, int j, float4 v, NoIn) const { st4(out + (size_t)m * H + j, v); }
};

template <int BN, bool kPair, class Epi>
inline cudaError_t launch_bn(const Args &g, const Epi &epi, cudaStream_t st) {
    cudaError_t e = cudaFuncSetAttribute(gemm_kernel<BN, kPair, Epi>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem_bytes(BN));
    if (e != cudaSuccess) return e;
    const unsigned blocks = (unsigned)((g.M + BM - 1) / BM) * (unsigned)(g.units * (kPair ? 2 : 1) / BN);
    gemm_kernel<BN, kPair, Epi><<<blocks, threads(BN), smem_bytes(BN), st>>>(g, epi);
    return cudaGetLastError();
}

// The same products on tiles of 32 sites x 32 columns (16 pairs), 2 x 4 outputs
// a thread.  A product of few sites is one wave of tiles, and its time is one
// tile's latency: the wide tile does 64 multiply-adds a thread for 16 floats
// read, this one 8 for 6 (a chain of 3 x 128 inner elements: 53 us wide, 10 us
// so).  Every output is the same chain of multiply-adds over the inner index,
// so both give the same bits, whatever the number of sites.
constexpr int SB = 32;       // sites and columns of a tile
constexpr int SStages = 4;   // cp.async ring
template <bool kPair, class Epi>
__global__ void __launch_bounds__(128) gemm_small_kernel(const __grid_constant__ Args g, const __grid_constant__ Epi epi) {
    constexpr int C = kPair ? SB / 2 : SB;  // units of the tile
    __shared__ __align__(16) float ring[SStages * 2 * SB * LDT];
    const int tid = threadIdx.x, tx = tid & 7, ty = tid >> 3;
    const int nblk = g.units / C;
    const int m0 = (int)(blockIdx.x / nblk) * SB, u0 = (int)(blockIdx.x % nblk) * C;
    const int lcol = tx * 4;

    int s_next = 0, k_next = 0;  // the stage to be requested next
    auto request = [&](int slot) {
        if (s_next < g.n_seg) {
            const Seg &s = g.seg[s_next];
            float *as = ring + (size_t)slot * 2 * SB * LDT, *ws = as + SB * LDT;
#pragma unroll
            for (int r = ty; r < SB; r += 16) {
                const int m = min(m0 + r, g.M - 1);  // rows past the end repeat the last (not stored)
                cp16(as + r * LDT + lcol, s.A + (size_t)m * s.lda + k_next + lcol);
                const float *w = !kPair || r < C ? s.W0 + (size_t)(u0 + r) * s.ldw : s.W1 + (size_t)(u0 + r - C) * s.ldw1;
                cp16(ws + r * LDT + lcol, w + k_next + lcol);
            }
            k_next += BK;
            if (k_next >= s.K) {
                k_next = 0;
                ++s_next;
            }
        }
        cp_commit();
    };
    int stages = 0;
    for (int s = 0; s < g.n_seg; ++s) stages += g.seg[s].K / BK;
#pragma unroll
    for (int st = 0; st < SStages - 1; ++st) request(st);
    float acc[2][4] = {};
    for (int st = 0; st < stages; ++st) {
        cp_wait<SStages - 2>();
        __syncthreads();  // this stage has landed, and the slot requested next has been read
        request((st + SStages - 1) % SStages);
        const float *as = ring + (size_t)(st % SStages) * 2 * SB * LDT + ty * LDT;
        const float *ws = ring + (size_t)(st % SStages) * 2 * SB * LDT + (SB + tx) * LDT;
#pragma unroll
        for (int k = 0; k < BK; k += 4) {
            float4 a[2], b[4];
#pragma unroll
            for (int i = 0; i < 2; ++i) a[i] = *reinterpret_cast<const float4 *>(as + 16 * i * LDT + k);
#pragma unroll
            for (int j = 0; j < 4; ++j) b[j] = *reinterpret_cast<const float4 *>(ws + 8 * j * LDT + k);
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    acc[i][j] = fmaf(a[i].x, b[j].x, acc[i][j]);
                    acc[i][j] = fmaf(a[i].y, b[j].y, acc[i][j]);
                    acc[i][j] = fmaf(a[i].z, b[j].z, acc[i][j]);
                    acc[i][j] = fmaf(a[i].w, b[j].w, acc[i][j]);
                }
        }
    }
    __syncthreads();  // the ring has been read: the tile goes through it, as in gemm_kernel
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) ring[(ty + 16 * i) * LDT + tx + 8 * j] = acc[i][j];
    __syncthreads();
    constexpr int kQuads = C / 4, kStep = 128 / kQuads;
    const int q = (tid % kQuads) * 4, u = u0 + q;
#pragma unroll
    for (int r = tid / kQuads; r < SB; r += kStep) {
        const int m = m0 + r;
        if (m >= g.M) break;
        const typename Epi::In in = epi.load(m, u);
        const float4 v = *reinterpret_cast<const float4 *>(ring + r * LDT + q);
        if constexpr (kPair) epi.store(m, u, v, *reinterpret_cast<const float4 *>(ring + r * LDT + C + q), in);
        else epi.store(m, u, v, in);
    }
}

// units: 32, 64 or a multiple of 128 (32 pairs make a 64-column tile).
// The small tile while the wide ones would not fill two thirds of the SMs: at
// 32, 64 and 96 wide tiles it takes 0.42 to 0.91, 0.64 to 0.95 and 0.70 to 1.09
// of the wide form's time (32 to 128 columns, 32 to 384 inner elements), at 128
// tiles 0.83 to 1.17, at 256 up to 1.24.  O_k rows of 64 samples of 16 sites,
// hidden 32 / 64 / 128: 131 / 200 / 395 us wide, 109 / 121 / 163 us small.
template <bool kPair, class Epi>
inline cudaError_t launch(const Args &g, const Epi &epi, int num_sms, cudaStream_t st) {
    const int cols = g.units * (kPair ? 2 : 1);
    const int BN = cols % 128 == 0 ? 128 : cols % 64 == 0 ? 64 : 32;
    if (cols % SB == 0 && 3 * ((int64_t)(g.M + BM - 1) / BM) * (cols / BN) <= 2 * (int64_t)num_sms) {
        const unsigned blocks = (unsigned)((g.M + SB - 1) / SB) * (unsigned)(cols / SB);
        gemm_small_kernel<kPair, Epi><<<blocks, 128, 0, st>>>(g, epi);
        return cudaGetLastError();
    }
    if (cols % 128 == 0) return launch_bn<128, kPair>(g, epi, st);
    if (cols % 64 == 0) return launch_bn<64, kPair>(g, epi, st);
    if constexpr (!kPair) {
        if (cols % 32 == 0) return launch_bn<32, kPair>(g, epi, st);
    }
    return cudaErrorInvalidValue;
}

// Weight gradients over a range of sites: out[j][k] = sum_m A[m][j] B[m][k],
// and (bias_off >= 0) the column sums of A.  Range x of a launch covers `len`
// sites at first x * step, in pieces of seg_len sites seg_stride apart; the
// result goes to out + x * out_stride.  Per-sample rows: a range is a sample.
// Sums over all samples: ranges of a few hundred sites, whose partial rows are
// summed in FP64 afterwards, so the rounding of a long FP32 sum never builds
// up (error of a range about 2.4e-8 sqrt(len) of its spread).
constexpr int kMaxPair = 6;
struct Pair {
    const float *A, *B;
    int lda, ldb, nj, nk, j_valid;  // rows j >= j_valid are not stored
    int M;                          // sites of this pair
    int64_t off;                    // of out[0][0]
    int ldo;
    int64_t bias_off;               // of the column sums of A, or -1
};
struct WgArgs {
    int n_pair, tiles[kMaxPair + 1];  // first tile of each pair
    Pair p[kMaxPair];
    int n_range, len, step, seg_len;
    int seg_stride;
    float *out;
    int64_t out_stride;
};

constexpr int WS = 32;  // sites per stage
constexpr size_t wg_smem_bytes(int BT) { return (size_t)2 * 2 * WS * BT * sizeof(float); }
constexpr int wg_threads(int BT) { return BT == 128 ? 256 : 64; }

template <int BT>
__global__ void __launch_bounds__(wg_threads(BT), BT == 128 ? 2 : 6) wgrad_kernel(const __grid_constant__ WgArgs g) {
    constexpr int T = wg_threads(BT);
    constexpr int TT = BT == 32 ? 4 : 8;  // outputs per thread: TT x TT
    extern __shared__ __align__(16) float smem[];
    const int tid = threadIdx.x;
    const int tk = tid % (BT / TT), tj = tid / (BT / TT);
    const int n_tiles = g.tiles[g.n_pair];
    const int x = (int)(blockIdx.x / n_tiles);
    const int tile = (int)(blockIdx.x % n_tiles);
    int pi = 0;
    while (tile >= g.tiles[pi + 1]) ++pi;
    const Pair &P = g.p[pi];
    const int kt = P.nk / BT;
    const int j0 = (tile - g.tiles[pi]) / kt * BT, k0 = (tile - g.tiles[pi]) % kt * BT;
    const int64_t base = (int64_t)x * g.step;
    // sites of the range that this pair has
    int cnt = g.len;
    if (g.seg_len >= g.len) cnt = (int)max((int64_t)0, min((int64_t)g.len, (int64_t)P.M - base));
    else cnt = min(g.len, P.M / g.seg_stride * g.seg_len);
    const bool bias = P.bias_off >= 0 && k0 == 0;

    float acc[TT][TT];
#pragma unroll
    for (int i = 0; i < TT; ++i)
#pragma unroll
        for (int k = 0; k < TT; ++k) acc[i][k] = 0.0f;
    float bsum[(BT + T - 1) / T];
#pragma unroll
    for (int i = 0; i < (BT + T - 1) / T; ++i) bsum[i] = 0.0f;

    constexpr int kChunks = BT / 4;  // 16-byte pieces of a row
    auto request = [&](int i0, int slot) {
        if (i0 < cnt) {
            float *as = smem + (size_t)slot * 2 * WS * BT, *bs = as + WS * BT;
#pragma unroll
            for (int q = tid; q < WS * kChunks; q += T) {
                const int r = q / kChunks, c = (q % kChunks) * 4;
                const int i = i0 + r;
                const bool in = i < cnt;
                const int ii = in ? i : 0;
                const int64_t m = base + (int64_t)(ii / g.seg_len) * g.seg_stride + ii % g.seg_len;
                cp16_or_zero(as + r * BT + c, P.A + (size_t)m * P.lda + j0 + c, in);
                cp16_or_zero(bs + r * BT + c, P.B + (size_t)m * P.ldb + k0 + c, in);
            }
        }
        cp_commit();
    };
    request(0, 0);
    int slot = 0;
    for (int i0 = 0; i0 < cnt; i0 += WS, slot ^= 1) {
        request(i0 + WS, slot ^ 1);
        cp_wait<1>();
        __syncthreads();
        const float *as = smem + (size_t)slot * 2 * WS * BT, *bs = as + WS * BT;
#pragma unroll 4
        for (int r = 0; r < WS; ++r) {
            float a[TT], b[TT];
#pragma unroll
            for (int q = 0; q < TT; q += 4) {
                const float4 va = *reinterpret_cast<const float4 *>(as + r * BT + tj * 4 + q / 4 * (BT / 2));
                const float4 vb = *reinterpret_cast<const float4 *>(bs + r * BT + tk * 4 + q / 4 * (BT / 2));
                a[q] = va.x; a[q + 1] = va.y; a[q + 2] = va.z; a[q + 3] = va.w;
                b[q] = vb.x; b[q + 1] = vb.y; b[q + 2] = vb.z; b[q + 3] = vb.w;
            }
#pragma unroll
            for (int i = 0; i < TT; ++i)
#pragma unroll
                for (int k = 0; k < TT; ++k) acc[i][k] = fmaf(a[i], b[k], acc[i][k]);
        }
        if (bias) {
#pragma unroll
            for (int q = 0; q < (BT + T - 1) / T; ++q) {
                const int j = tid + q * T;
                if (j >= BT) break;
                float s = 0.0f;
                for (int r = 0; r < WS; ++r) s += as[r * BT + j];
                bsum[q] += s;
            }
        }
        __syncthreads();
    }
    float *out = g.out + (int64_t)x * g.out_stride;
#pragma unroll
    for (int i = 0; i < TT; ++i) {
        const int j = j0 + tj * 4 + (i & 3) + i / 4 * (BT / 2);
        if (j >= P.j_valid) continue;
        float *row = out + P.off + (int64_t)j * P.ldo + k0 + tk * 4;
#pragma unroll
        for (int k = 0; k < TT; ++k) row[(k & 3) + k / 4 * (BT / 2)] = acc[i][k];
    }
    if (bias) {
#pragma unroll
        for (int q = 0; q < (BT + T - 1) / T; ++q) {
            const int j = j0 + tid + q * T;
            if (tid + q * T < BT && j < P.j_valid) out[P.bias_off + j] = bsum[q];
        }
    }
}

template <int BT>
inline cudaError_t launch_wgrad_bt(WgArgs g, cudaStream_t st) {
    g.tiles[0] = 0;
    for (int i = 0; i < g.n_pair; ++i) g.tiles[i + 1] = g.tiles[i] + (g.p[i].nj / BT) * (g.p[i].nk / BT);
    cudaError_t e = cudaFuncSetAttribute(wgrad_kernel<BT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)wg_smem_bytes(BT));
    if (e != cudaSuccess) return e;
    wgrad_kernel<BT><<<(unsigned)g.n_range * (unsigned)g.tiles[g.n_pair], wg_threads(BT), wg_smem_bytes(BT), st>>>(g);
    return cudaGetLastError();
}

// Tile by the pairs' sizes (all multiples of 32).
inline cudaError_t launch_wgrad(const WgArgs &g, cudaStream_t st) {
    bool by128 = true, by64 = true;
    for (int i = 0; i < g.n_pair; ++i) {
        by128 = by128 && g.p[i].nj % 128 == 0 && g.p[i].nk % 128 == 0;
        by64 = by64 && g.p[i].nj % 64 == 0 && g.p[i].nk % 64 == 0;
    }
    if (by128) return launch_wgrad_bt<128>(g, st);
    if (by64) return launch_wgrad_bt<64>(g, st);
    return launch_wgrad_bt<32>(g, st);
}

// out[dst + i] (+)= sum_r src[r * stride + i], i < len, in FP64 over groups of
// eight rows
constexpr int kMaxSum = 64;
struct SumSeg {
    const float *src;
    int64_t stride, dst;
    int rows, len;
};
struct SumArgs {
    int n;
    bool add;
    float *out;
    SumSeg s[kMaxSum];
};

static __global__ void __launch_bounds__(512) sum_rows_kernel(const __grid_constant__ SumArgs g) {
    __shared__ double part[8][64];
    const SumSeg &S = g.s[blockIdx.y];
    for (int64_t c0 = (int64_t)blockIdx.x * 64; c0 < S.len; c0 += (int64_t)gridDim.x * 64) {
        const int64_t i = c0 + threadIdx.x;
        double acc = 0.0;
        if (i < S.len) {
            // eight rows at a time in FP32: FP64 adds run at a fraction of the rate
            int r = threadIdx.y;
            for (; r + 56 < S.rows; r += 64) {
                float v = 0.0f;
#pragma unroll
                for (int q = 0; q < 8; ++q) v += S.src[(r + 8 * q) * S.stride + i];
                acc += (double)v;
            }
            for (; r < S.rows; r += 8) acc += (double)S.src[r * S.stride + i];
        }
        part[threadIdx.y][threadIdx.x] = acc;
        __syncthreads();
        if (threadIdx.y == 0 && i < S.len) {
            double t = 0.0;
#pragma unroll
            for (int y = 0; y < 8; ++y) t += part[y][threadIdx.x];
            if (g.add) t += (double)g.out[S.dst + i];
            g.out[S.dst + i] = (float)t;
        }
        __syncthreads();
    }
}

inline cudaError_t launch_sum_rows(const SumArgs &g, cudaStream_t st) {
    int longest = 1;
    for (int i = 0; i < g.n; ++i) longest = g.s[i].len > longest ? g.s[i].len : longest;
    int bx = (longest + 63) / 64;
    if (bx > 1024) bx = 1024;
    sum_rows_kernel<<<dim3((unsigned)bx, (unsigned)g.n), dim3(64, 8), 0, st>>>(g);
    return cudaGetLastError();
}

}  // namespace gemm
}  // namespace psr
