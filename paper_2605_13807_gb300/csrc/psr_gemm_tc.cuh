// The products of the layer-by-layer gradients on the tensor cores (tcgen05,
// BF16 operands, FP32 accumulation) with FP32 operands split into BF16 parts:
//   SPLIT = 2: x = hi + lo,        hi.hi + (hi.lo + lo.hi)
//   SPLIT = 3: x = hi + mid + lo,  hi.hi + (hi.mid + mid.hi + mid.mid + hi.lo + lo.hi)
// Two parts keep 16 mantissa bits (the 16-bit precision path), three keep all
// 24, so that only products below 2^-24 of the result are left out.  hi.hi and
// the corrections have accumulators of their own, added in FP32 at the end:
// the corrections (six times as many additions) then never round against the
// large sum.
//
// Same contract as psr_gemm.cuh's products (Args, Epi): out[m][n] = sum_k
// A[m][k] W[n][k].  A CTA tile is 128 sites (the 128 lanes of tensor memory) x
// BN columns; per 64 inner elements the threads read A and W as FP32, split
// them into 128-byte-swizzled K-major shared tiles, and one thread issues the
// MMAs.  The next 64 elements (of the next tile, at the end) are fetched into
// registers meanwhile; two CTAs per SM (99 KB and half of tensor memory each)
// overlap one's conversion and epilogue with the other's MMAs and loads.
//
// What bounds it: HBM at widths of 64 and 128 (K = 64, 128 columns, 409600 sites:
// 118 us for 315 MB; 202 us with FP32 multiply-adds), the MMAs and conversions
// at 256 (40000 x 256 x 256: 54 us = 97 TFLOP/s of the FP32 work; 144 us).
#pragma once

#include <cuda_bf16.h>

#include "psr_device.cuh"
#include "psr_gemm.cuh"
#include "psr_internal.cuh"
#include "psr_tc.cuh"

namespace psr {
namespace gemm {

constexpr uint32_t kTcA = 128 * 128;  // one part of a 128-row x 64-element BF16 tile

struct TcBlock {
    uint64_t mbar;
    uint32_t tmem_base;
    int abort_flag;
};

__host__ __device__ constexpr uint32_t tc_stage_bytes(int split, int BN) {
    return (uint32_t)split * (kTcA + (uint32_t)BN * 128u);
}
__host__ __device__ constexpr uint32_t tc_tile_bytes(int BN) { return 128u * (uint32_t)(BN + 4) * 4u; }
__host__ __device__ constexpr uint32_t tc_body_bytes(int split, int BN) {
    return tc_stage_bytes(split, BN) > tc_tile_bytes(BN) ? tc_stage_bytes(split, BN) : tc_tile_bytes(BN);
}
constexpr uint32_t tc_smem_bytes(int split, int BN) { return tc_body_bytes(split, BN) + (uint32_t)sizeof(TcBlock) + 1024; }

// kind::f16, D = F32, A = B = BF16, both K-major, M = 128, N = BN
template <int BN>
constexpr uint32_t kTcIdesc =
    (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);

// K-major tile: rows of 64 BF16 (128 bytes, swizzled), 8-row groups 1024 bytes apart
__device__ __forceinline__ uint64_t tc_desc(uint32_t addr) { return tc::sdesc(addr, 1024, 1024); }

// Eight consecutive inner elements of row r (16-byte chunk c) into the parts
// of a tile, `part` bytes apart.
template <int SPLIT>
__device__ __forceinline__ void split_store(uint8_t *tile, uint32_t part, int r, int c, const float (&v)[8]) {
    uint32_t w[SPLIT][4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        float x0 = v[2 * i], x1 = v[2 * i + 1];
#pragma unroll
        for (int s = 0; s < SPLIT; ++s) {
            const __nv_bfloat162 h = __floats2bfloat162_rn(x0, x1);
            w[s][i] = *reinterpret_cast<const uint32_t *>(&h);
            if (s + 1 < SPLIT) {
                x0 -= __uint_as_float(w[s][i] << 16);
                x1 -= __uint_as_float(w[s][i] & 0xFFFF0000u);
            }
        }
    }
    uint8_t *p = tile + (uint32_t)r * 128u + ((uint32_t)(c ^ (r & 7)) << 4);
#pragma unroll
    for (int s = 0; s < SPLIT; ++s)
        *reinterpret_cast<uint4 *>(p + s * part) = make_uint4(w[s][0], w[s][1], w[s][2], w[s][3]);
}

// MMAs of one 64-element stage (4 K steps): main += hi.hi, corr += the rest.
template <int SPLIT, uint32_t IDESC>
__device__ __forceinline__ void split_mma(uint32_t main, uint32_t corr, uint32_t a, uint32_t a_part, uint32_t b,
                                          uint32_t b_part, bool first) {
    auto run = [&](uint32_t d, int pa, int pb, bool fresh) {
        const uint64_t da = tc_desc(a + pa * a_part), db = tc_desc(b + pb * b_part);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)
            tc::mma_ss<IDESC>(d, da + (uint64_t)(2 * kk), db + (uint64_t)(2 * kk), (fresh && kk == 0) ? 0u : 1u);
    };
    if (SPLIT == 3) {
        run(corr, 2, 0, first);
        run(corr, 0, 2, false);
        run(corr, 1, 1, false);
    }
    run(corr, 1, 0, SPLIT == 2 && first);
    run(corr, 0, 1, false);
    run(main, 0, 0, first);
}

template <int SPLIT, int BN, bool kPair, class Epi>
__global__ void __launch_bounds__(256, 2)
    gemm_tc_kernel(const __grid_constant__ Args g, const __grid_constant__ Epi epi, int *status) {
    constexpr int C = kPair ? BN / 2 : BN, NB = BN / 32;  // NB: 8-element pieces of W per thread and stage
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    TcBlock &B = *reinterpret_cast<TcBlock *>(smem + tc_body_bytes(SPLIT, BN));
    uint8_t *tile_a = smem, *tile_b = smem + SPLIT * kTcA;
    constexpr uint32_t kPartB = (uint32_t)BN * 128u;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc::smem_u32(&B.tmem_base)),
                     "r"(2u * BN)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        tc::mbar_init(tc::smem_u32(&B.mbar), 1);
        B.abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    tc::tc_before();
    __syncthreads();
    tc::tc_after();
    const uint32_t tmem = B.tmem_base, bar = tc::smem_u32(&B.mbar);
    const uint32_t sa = tc::smem_u32(tile_a), sb = tc::smem_u32(tile_b);
    uint32_t phase = 0;

    const int nblk = g.units / C;
    const int64_t tiles = (int64_t)((g.M + 127) / 128) * nblk;
    const int row0 = tid >> 3, c0 = tid & 7;  // pieces: rows row0 + 32 i, chunk c0
    float ra[4][8], rb[NB][8];
    // the stage to be fetched next
    int64_t ft = blockIdx.x;
    int fs = 0, fk = 0;
    auto fetch = [&]() {
        if (ft >= tiles) return;
        const Seg &s = g.seg[fs];
        const int m0 = (int)(ft / nblk) * 128, u0 = (int)(ft % nblk) * C;
        const int k = fk + 8 * c0;
        const bool in = k < s.K;  // K is a multiple of 32; the rest of a stage is zero
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float *p = s.A + (size_t)min(m0 + row0 + 32 * i, g.M - 1) * s.lda + k;
            const float4 x = in ? ld4(p) : make_float4(0, 0, 0, 0), y = in ? ld4(p + 4) : make_float4(0, 0, 0, 0);
            ra[i][0] = x.x; ra[i][1] = x.y; ra[i][2] = x.z; ra[i][3] = x.w;
            ra[i][4] = y.x; ra[i][5] = y.y; ra[i][6] = y.z; ra[i][7] = y.w;
        }
#pragma unroll
        for (int i = 0; i < NB; ++i) {
            const int n = row0 + 32 * i;
            const float *p = (!kPair || n < C) ? s.W0 + (size_t)(u0 + n) * s.ldw + k
                                               : s.W1 + (size_t)(u0 + n - C) * s.ldw1 + k;
            const float4 x = in ? ld4(p) : make_float4(0, 0, 0, 0), y = in ? ld4(p + 4) : make_float4(0, 0, 0, 0);
            rb[i][0] = x.x; rb[i][1] = x.y; rb[i][2] = x.z; rb[i][3] = x.w;
            rb[i][4] = y.x; rb[i][5] = y.y; rb[i][6] = y.z; rb[i][7] = y.w;
        }
        fk += 64;
        if (fk >= s.K) {
            fk = 0;
            if (++fs == g.n_seg) {
                fs = 0;
                ft += gridDim.x;
            }
        }
    };
    int stages = 0;
    for (int s = 0; s < g.n_seg; ++s) stages += (g.seg[s].K + 63) / 64;
    fetch();
    bool stop = false;
    for (int64_t t = blockIdx.x; t < tiles && !stop; t += gridDim.x) {
        for (int st = 0; st < stages; ++st) {
#pragma unroll
            for (int i = 0; i < 4; ++i) split_store<SPLIT>(tile_a, kTcA, row0 + 32 * i, c0, ra[i]);
#pragma unroll
            for (int i = 0; i < NB; ++i) split_store<SPLIT>(tile_b, kPartB, row0 + 32 * i, c0, rb[i]);
            tc::fence_proxy_async();
            tc::tc_before();
            __syncthreads();
            tc::tc_after();
            if (B.abort_flag) {
                stop = true;
                break;
            }
            if (tid == 0) {
                split_mma<SPLIT, kTcIdesc<BN>>(tmem, tmem + BN, sa, kTcA, sb, kPartB, st == 0);
                tc::mma_commit(bar);
            }
            fetch();
            if (!tc::mbar_wait(bar, phase)) {
                B.abort_flag = 1;
                set_status(status, PSR_ETIMEOUT);
            }
            phase ^= 1u;
            tc::tc_after();
        }
        if (stop) break;
        // accumulators -> shared tile (whole rows for the epilogue)
        constexpr int LDC = BN + 4;
        float *tile = reinterpret_cast<float *>(smem);
        {
            const int r = (warp & 3) * 32 + lane;
            const uint32_t lane_off = (uint32_t)((warp & 3) * 32) << 16;
#pragma unroll
            for (int c = 0; c < BN / 2; c += 16) {
                const int col = (warp >> 2) * (BN / 2) + c;
                uint32_t x[16], y[16];
                tc::tmem_ld16(tmem + lane_off + col, x);
                tc::tmem_ld16(tmem + lane_off + BN + col, y);
                tc::tmem_wait_ld16x2(x, y);
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    st4(tile + r * LDC + col + 4 * q,
                        make_float4(__uint_as_float(x[4 * q]) + __uint_as_float(y[4 * q]),
                                    __uint_as_float(x[4 * q + 1]) + __uint_as_float(y[4 * q + 1]),
                                    __uint_as_float(x[4 * q + 2]) + __uint_as_float(y[4 * q + 2]),
                                    __uint_as_float(x[4 * q + 3]) + __uint_as_float(y[4 * q + 3])));
            }
        }
        tc::tc_before();
        __syncthreads();
        tc::tc_after();
        const int m0 = (int)(t / nblk) * 128;
        constexpr int kQuads = C / 4, kStep = 256 / kQuads, kRows = 4;
        static_assert(128 % (kStep * kRows) == 0, "whole groups of rows");
        const int q = (tid % kQuads) * 4, r0 = tid / kQuads;
        const int u = (int)(t % nblk) * C + q;
#pragma unroll 1
        for (int r = r0; r < 128; r += kStep * kRows) {
            typename Epi::In in[kRows];
#pragma unroll
            for (int k = 0; k < kRows; ++k) in[k] = epi.load(min(m0 + r + k * kStep, g.M - 1), u);
#pragma unroll
            for (int k = 0; k < kRows; ++k) {
                const int m = m0 + r + k * kStep;
                if (m >= g.M) break;
                const float *row = tile + (r + k * kStep) * LDC + q;
                if constexpr (kPair) epi.store(m, u, ld4(row), ld4(row + C), in[k]);
                else epi.store(m, u, ld4(row), in[k]);
            }
        }
        __syncthreads();  // the tile is free for the next stage
    }
    // after a wait that ran out, MMAs may still be reading the tiles: wait once
    // more (bounded too) before the tensor memory is given back
    if (B.abort_flag) tc::mbar_wait(bar, phase ^ 1u);
    tc::tc_before();
    __syncthreads();
    if (warp == 0) {
        tc::tc_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2u * BN) : "memory");
    }
}

template <int SPLIT, int BN, bool kPair, class Epi>
inline cudaError_t launch_tc(const Args &g, const Epi &epi, const Engine &en, cudaStream_t st) {
    constexpr int C = kPair ? BN / 2 : BN;
    cudaError_t e = cudaFuncSetAttribute(gemm_tc_kernel<SPLIT, BN, kPair, Epi>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tc_smem_bytes(SPLIT, BN));
    if (e != cudaSuccess) return e;
    const int64_t tiles = (int64_t)((g.M + 127) / 128) * (g.units / C);
    const int64_t grid = tiles < 2 * en.num_sms ? tiles : 2 * en.num_sms;
    gemm_tc_kernel<SPLIT, BN, kPair, Epi><<<(unsigned)grid, 256, tc_smem_bytes(SPLIT, BN), st>>>(g, epi, en.status);
    return cudaGetLastError();
}

// (two parts: hidden 128 only, so whole tiles of 128 columns)
template <bool kPair, class Epi>
inline cudaError_t launch(const Args &g, const Epi &epi, const Engine &en, cudaStream_t st) {
    const int cols = g.units * (kPair ? 2 : 1);
    if (en.split == 2 && cols % 128 == 0) return launch_tc<2, 128, kPair>(g, epi, en, st);
    if (en.split == 3 && cols % 128 == 0) return launch_tc<3, 128, kPair>(g, epi, en, st);
    if (en.split == 3 && cols % 64 == 0) return launch_tc<3, 64, kPair>(g, epi, en, st);
    return launch<kPair>(g, epi, en.num_sms, st);
}

// Weight gradients on the tensor cores: out[j][k] = sum_m A[m][j] B[m][k] over
// the sites of a range.  A job is a 128 x 128 block of outputs made of 64 x 64
// quadrants (row block rb from A[rb], column block cb from B[cb]; widths of 64
// stack two arrays, wider ones take neighbouring units), each stored at
// off[rb][cb] (-1: not wanted), plus column sums of A at bias[rb] (or -1).
// Both operands go to shared memory with the sites contiguous: a thread reads
// eight sites of one unit (coalesced over units) and splits them into 16 bytes
// of each part.
constexpr int kMaxJob = 24;
struct WgJob {
    const float *A[2], *B[2];
    int lda, ldb, M;
    int ldo[2][2];
    int64_t off[2][2], bias[2];
};
struct WgTcArgs {
    int n_job, n_range, len;  // range x: sites x len .. (x + 1) len - 1
    WgJob job[kMaxJob];
    float *out;
    int64_t out_stride;
};

template <int SPLIT>
__global__ void __launch_bounds__(256, 2) wgrad_tc_kernel(const __grid_constant__ WgTcArgs g, int *status) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    TcBlock &B = *reinterpret_cast<TcBlock *>(smem + tc_body_bytes(SPLIT, 128));
    uint8_t *tile_a = smem, *tile_b = smem + SPLIT * kTcA;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc::smem_u32(&B.tmem_base)),
                     "r"(256u)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        tc::mbar_init(tc::smem_u32(&B.mbar), 1);
        B.abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    tc::tc_before();
    __syncthreads();
    tc::tc_after();
    const uint32_t tmem = B.tmem_base, bar = tc::smem_u32(&B.mbar);
    const uint32_t sa = tc::smem_u32(tile_a), sb = tc::smem_u32(tile_b);
    uint32_t phase = 0;

    const int j = tid & 127, rb = j >> 6, c0 = tid >> 7;  // unit row of both tiles; site chunks c0 + 2 i
    const unsigned n_job = g.n_job, items = g.n_range * n_job;
    float ra[4][8], rbv[4][8];
    unsigned fi = blockIdx.x;  // the stage to be fetched next: item, first site in its range
    int f0 = 0;
    // sites of an item; an empty one still runs a stage, of zeros
    auto sites_of = [&](unsigned it) {
        const long long left = (long long)g.job[it % n_job].M - (long long)(it / n_job) * g.len;
        return left <= 0 ? 0 : left < g.len ? (int)left : g.len;
    };
    auto fetch = [&]() {
        if (fi >= items) return;
        const WgJob &J = g.job[fi % n_job];
        const int cnt = sites_of(fi), t = f0 + 8 * c0;
        const long long m = (long long)(fi / n_job) * g.len + t;
        const float *pa = J.A[rb] + (j & 63) + m * J.lda, *pb = J.B[rb] + (j & 63) + m * J.ldb;
        if (f0 + 64 <= cnt) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float *qa = pa + (long long)(16 * i) * J.lda, *qb = pb + (long long)(16 * i) * J.ldb;
#pragma unroll
                for (int e = 0; e < 8; ++e, qa += J.lda, qb += J.ldb) {
                    ra[i][e] = *qa;
                    rbv[i][e] = *qb;
                }
            }
        } else {
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const int d = 16 * i + e;
                    const bool in = t + d < cnt;
                    ra[i][e] = in ? pa[(long long)d * J.lda] : 0.0f;
                    rbv[i][e] = in ? pb[(long long)d * J.ldb] : 0.0f;
                }
        }
        f0 += 64;
        if (f0 >= cnt) {
            f0 = 0;
            fi += gridDim.x;
        }
    };
    fetch();
    bool stop = false;
    for (unsigned it = blockIdx.x; it < items && !stop; it += gridDim.x) {
        const WgJob &J = g.job[it % n_job];
        const int stages = max(1, (sites_of(it) + 63) / 64);
        float bsum = 0.0f;
        for (int st = 0; st < stages; ++st) {
            float s8 = 0.0f;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                split_store<SPLIT>(tile_a, kTcA, j, c0 + 2 * i, ra[i]);
                split_store<SPLIT>(tile_b, kTcA, j, c0 + 2 * i, rbv[i]);
#pragma unroll
                for (int e = 0; e < 8; ++e) s8 += ra[i][e];
            }
            bsum += s8;
            tc::fence_proxy_async();
            tc::tc_before();
            __syncthreads();
            tc::tc_after();
            if (B.abort_flag) {
                stop = true;
                break;
            }
            if (tid == 0) {
                split_mma<SPLIT, kTcIdesc<128>>(tmem, tmem + 128, sa, kTcA, sb, kTcA, st == 0);
                tc::mma_commit(bar);
            }
            fetch();
            if (!tc::mbar_wait(bar, phase)) {
                B.abort_flag = 1;
                set_status(status, PSR_ETIMEOUT);
            }
            phase ^= 1u;
            tc::tc_after();
        }
        if (stop) break;
        constexpr int LDC = 132;
        float *tile = reinterpret_cast<float *>(smem);
        {
            const int r = (warp & 3) * 32 + lane;
            const uint32_t lane_off = (uint32_t)((warp & 3) * 32) << 16;
#pragma unroll
            for (int c = 0; c < 64; c += 16) {
                const int col = (warp >> 2) * 64 + c;
                uint32_t x[16], y[16];
                tc::tmem_ld16(tmem + lane_off + col, x);
                tc::tmem_ld16(tmem + lane_off + 128 + col, y);
                tc::tmem_wait_ld16x2(x, y);
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    st4(tile + r * LDC + col + 4 * q,
                        make_float4(__uint_as_float(x[4 * q]) + __uint_as_float(y[4 * q]),
                                    __uint_as_float(x[4 * q + 1]) + __uint_as_float(y[4 * q + 1]),
                                    __uint_as_float(x[4 * q + 2]) + __uint_as_float(y[4 * q + 2]),
                                    __uint_as_float(x[4 * q + 3]) + __uint_as_float(y[4 * q + 3])));
            }
        }
        if (c0) tile[j * LDC + 128] = bsum;  // the padding of row j
        tc::tc_before();
        __syncthreads();
        tc::tc_after();
        float *out = g.out + (int64_t)(it / n_job) * g.out_stride;
        if (c0 == 0 && J.bias[rb] >= 0) out[J.bias[rb] + (j & 63)] = bsum + tile[j * LDC + 128];
        // rows warp, warp + 8, ...: 32 consecutive floats an instruction (a row
        // of P floats need not start 16-byte aligned)
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            const int64_t off = J.off[h >> 1][h & 1];
            if (off < 0) continue;
            const int ldo = J.ldo[h >> 1][h & 1];
            float *p = out + off + (int64_t)warp * ldo + lane;
            const float *q = tile + (64 * (h >> 1) + warp) * LDC + 64 * (h & 1) + lane;
#pragma unroll
            for (int r = 0; r < 64; r += 8, p += 8 * (int64_t)ldo, q += 8 * LDC) {
                p[0] = q[0];
                p[32] = q[32];
            }
        }
        __syncthreads();
    }
    // after a wait that ran out, MMAs may still be reading the tiles: wait once
    // more (bounded too) before the tensor memory is given back
    if (B.abort_flag) tc::mbar_wait(bar, phase ^ 1u);
    tc::tc_before();
    __syncthreads();
    if (warp == 0) {
        tc::tc_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(256u) : "memory");
    }
}

template <int SPLIT>
inline cudaError_t launch_wgrad_tc(const WgTcArgs &g, const Engine &en, cudaStream_t st) {
    cudaError_t e = cudaFuncSetAttribute(wgrad_tc_kernel<SPLIT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)tc_smem_bytes(SPLIT, 128));
    if (e != cudaSuccess) return e;
    const int64_t items = (int64_t)g.n_range * g.n_job;
    const int64_t grid = items < 2 * en.num_sms ? items : 2 * en.num_sms;
    wgrad_tc_kernel<SPLIT><<<(unsigned)grid, 256, tc_smem_bytes(SPLIT, 128), st>>>(g, en.status);
    return cudaGetLastError();
}

// The pairs of WgArgs on the engine: tensor cores for contiguous ranges and
// widths that are multiples of 64, else the CUDA-core form.
inline cudaError_t launch_wgrad(const WgArgs &g, const Engine &en, cudaStream_t st) {
    bool ok = en.split != 0 && g.seg_len >= g.len && g.step == g.len;
    int blocks = 0;
    for (int i = 0; i < g.n_pair; ++i) {
        const Pair &p = g.p[i];
        ok = ok && p.nj % 64 == 0 && p.nk % 64 == 0 && p.j_valid == p.nj &&
             (p.nj == 64 && p.nk == 64 || p.nj % 128 == 0 && p.nk % 128 == 0);
        blocks += p.nj >= 128 ? (p.nj / 128) * (p.nk / 128) : 1;
    }
    if (!ok || blocks > kMaxJob) return launch_wgrad(g, st);
    WgTcArgs w{};
    w.n_range = g.n_range;
    w.len = g.len;
    w.out = g.out;
    w.out_stride = g.out_stride;
    bool done[kMaxPair] = {};
    for (int i = 0; i < g.n_pair; ++i) {
        if (done[i]) continue;
        const Pair &p = g.p[i];
        if (p.nj >= 128) {
            for (int jt = 0; jt < p.nj; jt += 128)
                for (int kt = 0; kt < p.nk; kt += 128) {
                    WgJob &J = w.job[w.n_job++];
                    J.lda = p.lda;
                    J.ldb = p.ldb;
                    J.M = p.M;
                    for (int r = 0; r < 2; ++r) {
                        J.A[r] = p.A + jt + 64 * r;
                        J.B[r] = p.B + kt + 64 * r;
                        J.bias[r] = p.bias_off >= 0 && kt == 0 ? p.bias_off + jt + 64 * r : -1;
                        for (int c = 0; c < 2; ++c) {
                            J.off[r][c] = p.off + (int64_t)(jt + 64 * r) * p.ldo + kt + 64 * c;
                            J.ldo[r][c] = p.ldo;
                        }
                    }
                }
            continue;
        }
        // width 64: stack a second A array and a second B array of other
        // pairs over the same sites, and take every pair the four quadrants hold
        WgJob &J = w.job[w.n_job++];
        J.lda = p.lda;
        J.ldb = p.ldb;
        J.M = p.M;
        J.A[0] = J.A[1] = p.A;
        J.B[0] = J.B[1] = p.B;
        int na = 1, nb = 1;
        for (int q = i + 1; q < g.n_pair; ++q) {
            const Pair &o = g.p[q];
            if (done[q] || o.M != p.M || o.lda != p.lda || o.ldb != p.ldb) continue;
            const bool has_a = o.A == J.A[0] || (na == 2 && o.A == J.A[1]);
            const bool has_b = o.B == J.B[0] || (nb == 2 && o.B == J.B[1]);
            if (!has_a && !has_b) continue;
            if (!has_a && na == 1) J.A[na++] = o.A;
            if (!has_b && nb == 1) J.B[nb++] = o.B;
        }
        for (int r = 0; r < 2; ++r) {
            J.bias[r] = -1;
            for (int c = 0; c < 2; ++c) {
                J.off[r][c] = -1;
                J.ldo[r][c] = 0;
                if (r >= na || c >= nb) continue;
                for (int q = i; q < g.n_pair; ++q) {
                    const Pair &o = g.p[q];
                    if (done[q] || o.M != p.M || o.lda != p.lda || o.ldb != p.ldb || o.A != J.A[r] || o.B != J.B[c]) continue;
                    J.off[r][c] = o.off;
                    J.ldo[r][c] = o.ldo;
                    if (o.bias_off >= 0) J.bias[r] = o.bias_off;
                    done[q] = true;
                    break;
                }
            }
        }
    }
    return en.split == 2 ? launch_wgrad_tc<2>(w, en, st) : launch_wgrad_tc<3>(w, en, st);
}

}  // namespace gemm
}  // namespace psr
