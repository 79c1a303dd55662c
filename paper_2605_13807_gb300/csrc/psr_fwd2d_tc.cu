// Forward of the paper's two-dimensional patched minGRU (Sec. II.F,
// two-dimensional recurrences; Sec. II.G residual and GELU) on the tensor
// cores: BF16 operands, FP32 accumulation in tensor memory, FP32 gates,
// scan, GELU and softmax.
//
// The model is the one psr_fwd2d.cu evaluates in FP32 (2 x 2 patches along
// the zigzag path of the patch lattice, row by row: within a patch row the
// gates and candidates of all sites are one batched projection, the h_V part
// acting on the previous row's states, followed by the scan
// h = a h_H + (1 - a) h~ along the row).  Here every contraction of a row is
// a tcgen05 MMA with the weights as the A operand (M = 128 hidden units, one
// or two halves) and the row's sites as B (N = 128 columns):
//   z = W_z x,  c = W_hx x + W_hv h_V,  y = D x + C h,  logits = W_o x.
// Layer 0's input is the one-hot pair (v_H, v_V) of 32 entries, zero-padded
// to one 64-wide K chunk.
//
// Work layout.  One persistent CTA per SM holds 128 site columns cut into S
// slots of W = 8 ceil(P_x / 8) columns; each slot evaluates one job
// (configuration) and advances one patch row per step, so all slots share
// every weight fetch.  A slot whose job has finished takes the next job from
// a counter.  The weights (about 1.7 MB per row step at d_h = 256) do not fit
// in shared memory: they are stored once, in MMA order, as 16 KB slices
// (128 rows x 64 BF16, 128-byte swizzle) and streamed through a ring of
// slices by bulk copies, from L2, where every CTA's stream hits.
//
// Roles: 512 epilogue threads (a thread's tensor-memory lane holds one hidden
// unit's accumulators for all 128 columns), one producer thread (the weight
// stream), one MMA thread and one image warp (the h_V images: up to S H / 64
// bulk copies per layer each way, two a lane; issued by single threads of the
// MMA and epilogue roles they held up every other thread, 20 % of a row step
// at 16 slots).  Per row step and layer:
//   MMA  z, c (needs x, then h_V)  ->  epilogue: gates and scan, h -> smem
//   MMA  y = D x + C h             ->  epilogue: GELU(y + residual) -> x
// then the readout MMA and the masked 16-way softmax of every patch.
// The next row's h_V is this row's h, path-reversed (consecutive rows run in
// opposite directions); the image warp writes it to global memory as a 16-bit
// image in the tile layout, and the next row bulk-copies it into the h tile.  In
// mode 0 these images are the row checkpoints that mode 1 (connected
// configurations, resumed at the patch row of the first flipped spin) reads.
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include "psr_bf16_math.cuh"
#include "psr_device.cuh"
#include "psr_internal.cuh"
#include "psr_tc.cuh"

namespace psr {

namespace {

using namespace tc;
using namespace bf16m;

constexpr int kCols = 128;          // site columns per CTA (MMA N)
constexpr uint32_t kSlice = 16384;  // 128 rows x 64 BF16
constexpr int kMaxSlots = 16;
constexpr int kMaxRing = 10;

// kind::f16, D = F32, A = B = FP16 (F16) or BF16, both K-major, M = 128,
// N = 128.
template <bool F16>
constexpr uint32_t idesc2() {
    return (1u << 4) | ((F16 ? 0u : 1u) << 7) | ((F16 ? 0u : 1u) << 10) | (0u << 15) | (0u << 16) |
           ((uint32_t)(kCols >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
}

// Descriptor of a K-major, 128-byte-swizzled operand: 8-row atoms of 1024
// bytes stacked along M (or N); K = 16 step kk is 32 bytes along the row.
__device__ __forceinline__ uint64_t kdesc(uint32_t addr) {
    return (uint64_t)((addr >> 4) & 0x3FFFu) | ((uint64_t)(1024u >> 4) << 16) |
           ((uint64_t)(1024u >> 4) << 32) | (1ull << 46) | (2ull << 61);
}
__device__ __forceinline__ uint64_t kstep(int kk) { return (uint64_t)((kk * 32) >> 4); }

constexpr int kEpi = 512;             // epilogue threads: 512 / H per hidden unit
constexpr int kThreads2 = kEpi + 96;  // + producer, MMA and image warps

struct Slot2 {
    int job;              // -1: needs a job, -2: none left, else a job is running
    int64_t out;          // its place in A.out
    int sample, p, q;     // configuration (p, q: flipped sites or -1)
    int row, r0, n_up;    // current patch row, first row, up spins before it
    // sum of log P (mode 0) or of its differences (mode 1) over the rows before the
    // one whose sums (part, per 8-column chunk) are still to be added: its job's
    // last row or not, and that job's place in A.out
    float acc, part[4];
    int pend, pend_last;
    int64_t pend_out;
    uint8_t v[32];        // patch values of the current row, by column
    uint8_t vprev[32];    // previous row's values, by column
};

struct Misc2 {
    uint64_t full[kMaxRing], empty[kMaxRing];
    uint64_t e2m[2], m2e[2], go[2];  // e2m, m2e: per unit half
    // image warp: a row step's slots are set, the h tile is written (MMA thread),
    // its last reader is done (MMA commit), h_V has landed in it
    uint64_t slots, hset, hfree, hv;
    uint32_t tmem_base;
    int abort_flag;
    int go_flag[2];
    Slot2 slot[kMaxSlots];
};

// Bounded wait that also gives up once another role has aborted.
__device__ __forceinline__ bool wait_ab(uint32_t bar, uint32_t parity, const volatile int *ab) {
    if (mbar_try_wait(bar, parity)) return true;
    const uint64_t t0 = globaltimer();
    for (uint32_t it = 0; it < (1u << 30); ++it) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((it & 255u) == 255u && (*ab || globaltimer() - t0 > kWaitNs)) return false;
    }
    return false;
}

__device__ __forceinline__ int seq_pos2d(int Lx, int i, int j) {
    return j * Lx + ((j & 1) ? (Lx - 1 - i) : i);
}

// Value (0..15) of patch (pi, pj): spin (2 pi + dx, 2 pj + dy) is bit
// 2 dy + dx, with sites p and q flipped.
__device__ __forceinline__ int patch_value(const uint8_t *s, int Lx, int pi, int pj, int p, int q) {
    int v = 0;
#pragma unroll
    for (int b = 0; b < 4; ++b) {
        const int pos = seq_pos2d(Lx, 2 * pi + (b & 1), 2 * pj + (b >> 1));
        v |= ((int)(s[pos] & 1u) ^ (pos == p) ^ (pos == q)) << b;
    }
    return v;
}

// Named barrier `id` of `n` threads.
__device__ __forceinline__ void named_bar(uint32_t id, uint32_t n) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory");
}

// Named barrier that also ORs a flag over its threads, so that they all
// take the same exit.
__device__ __forceinline__ bool named_bar_or(uint32_t id, uint32_t n, bool v) {
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.u32 p, %1, 0;\n\t"
        "bar.red.or.pred q, %2, %3, p;\n\t"
        "selp.u32 %0, 1, 0, q;\n\t}"
        : "=r"(r)
        : "r"((uint32_t)v), "r"(id), "r"(n)
        : "memory");
    return r != 0;
}
// all epilogue threads (barrier 1)
__device__ __forceinline__ bool epi_bar_or(bool v) { return named_bar_or(1, kEpi, v); }

// Bulk copy shared -> global (bulk-group completion).
__device__ __forceinline__ void bulk_s2g(void *dst, uint32_t src, uint32_t bytes) {
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(src), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

// Operand bits of an FP32 value, rounded to nearest: FP16 (values beyond the
// largest finite FP16 saturate to it) or BF16.
template <bool F16>
__device__ __forceinline__ uint16_t op_bits(float x) {
    uint16_t h;
    if (F16) asm("cvt.rn.satfinite.f16.f32 %0, %1;" : "=h"(h) : "f"(x));
    else asm("cvt.rn.bf16.f32 %0, %1;" : "=h"(h) : "f"(x));
    return h;
}
template <bool F16>
__device__ __forceinline__ uint32_t op_pack(float lo, float hi) {
    return (uint32_t)op_bits<F16>(lo) | ((uint32_t)op_bits<F16>(hi) << 16);
}

template <int H, bool F16>
__global__ void __launch_bounds__(kThreads2, 1) fwd2d_tc_kernel(const __grid_constant__ Fwd2TcArgs A) {
    constexpr int NH = H / 128;     // unit halves (M tiles)
    constexpr int KC = H / 64;      // K chunks of a hidden-size input
    constexpr int CG = kEpi / H;    // epilogue threads per unit (column groups)
    constexpr int NW = kEpi / 32;   // epilogue warps
    constexpr uint32_t kTileBytes = KC * 16384u;
    extern __shared__ __align__(16) uint8_t smem_raw[];
    Misc2 &M = *reinterpret_cast<Misc2 *>(smem_raw);
    uint8_t *tiles = reinterpret_cast<uint8_t *>(
        (reinterpret_cast<uintptr_t>(smem_raw) + sizeof(Misc2) + 1023) & ~uintptr_t(1023));
    uint8_t *xt = tiles;                    // layer input x (K-major rows = site columns)
    uint8_t *ht = tiles + kTileBytes;       // h_V, then the layer's states h
    uint8_t *ring = tiles + 2 * kTileBytes; // weight slices
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int R = A.R, S = A.S, W = A.W, Lx = A.Lx, Ly = A.Ly, Px = Lx >> 1, Py = Ly >> 1;
    const int nL = A.tl.nL, N = Lx * Ly, Np = Px * Py;
    const int nch = W >> 3;  // 8-column chunks of a slot
    const uint32_t img_bytes = (uint32_t)KC * (uint32_t)W * 128u;  // one layer's h_V image of a slot
    const volatile int *ab = &M.abort_flag;
    uint8_t *scratch = A.scratch + (size_t)blockIdx.x * S * nL * img_bytes;

    // h_V image of layer l for slot s's current row (source) and for its next
    // row (destination; null after the job's last row)
    auto img_src = [&](const Slot2 &st, int s, int l) -> const uint8_t * {
        if (st.row == st.r0) {
            if (st.r0 == 0) return A.zero_img;
            return A.img_in + (((size_t)st.sample * Py + st.r0) * nL + l) * img_bytes;
        }
        if (A.img_out) return A.img_out + (((size_t)st.sample * Py + st.row) * nL + l) * img_bytes;
        return scratch + ((size_t)s * nL + l) * img_bytes;
    };
    auto img_dst = [&](const Slot2 &st, int s, int l) -> uint8_t * {
        if (st.row + 1 >= Py) return nullptr;
        if (A.img_out) return A.img_out + (((size_t)st.sample * Py + st.row + 1) * nL + l) * img_bytes;
        return scratch + ((size_t)s * nL + l) * img_bytes;
    };

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(&M.tmem_base))
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        for (int i = 0; i < R; ++i) {
            mbar_init(smem_u32(&M.full[i]), 1);
            mbar_init(smem_u32(&M.empty[i]), 1);
        }
        for (int g = 0; g < 2; ++g) {
            mbar_init(smem_u32(&M.e2m[g]), 1);
            mbar_init(smem_u32(&M.m2e[g]), 1);
        }
        mbar_init(smem_u32(&M.slots), 1);
        mbar_init(smem_u32(&M.hset), 1);
        mbar_init(smem_u32(&M.hfree), 1);
        mbar_init(smem_u32(&M.hv), 1);
        mbar_init(smem_u32(&M.go[0]), 1);
        mbar_init(smem_u32(&M.go[1]), 1);
        M.abort_flag = 0;
        M.go_flag[0] = 1;
        M.go_flag[1] = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    for (int s = tid; s < kMaxSlots; s += blockDim.x) {
        M.slot[s].job = -1;
        M.slot[s].acc = 0.0f;
        M.slot[s].pend = 0;
    }
    tc_before();
    __syncthreads();
    tc_after();
    const uint32_t tmem = M.tmem_base;
    if (tmem != 0) {  // all 512 columns are needed from column 0
        if (tid == 0) set_status(A.status, PSR_EDEVICE);
        M.abort_flag = 1;
    }
    if (tid == 0) mbar_arrive(smem_u32(&M.go[0]));  // row step 0 runs
    __syncthreads();
    const long long per_set = A.mode == 1 ? (long long)*A.n_jobs_dev : (long long)A.n_jobs;
    const long long njobs = A.images > 1 ? per_set * A.images : per_set;
    const uint32_t hvb = smem_u32(&M.hv);

    if (warp == NW) {
        // ------------------------------------------------ producer: weight stream
        if (lane == 0 && !M.abort_flag) {
            uint32_t q = 0, slot = 0, round = 0;  // slices issued; ring slot and pass over the ring
            const uint32_t fb = smem_u32(&M.full[0]), ebar = smem_u32(&M.empty[0]), rb = smem_u32(ring);
            for (uint32_t row = 0;; ++row) {
                if (!wait_ab(smem_u32(&M.go[row & 1]), (row >> 1) & 1, ab)) break;
                if (!*(volatile int *)&M.go_flag[row & 1]) break;
                bool ok = true;
                const uint8_t *src = A.wimg;
                for (int i = 0; i < A.n_slices; ++i, ++q, src += kSlice) {
                    if (round > 0 && !wait_ab(ebar + 8 * slot, (round - 1) & 1, ab)) {
                        ok = false;
                        break;
                    }
                    mbar_arrive_tx(fb + 8 * slot, kSlice);
                    bulk_g2s(rb + slot * kSlice, src, kSlice, fb + 8 * slot);
                    if (++slot == (uint32_t)R) {
                        slot = 0;
                        ++round;
                    }
                }
                if (!ok) break;
            }
            // copies still in flight land before the CTA may exit
            const uint32_t last = q < (uint32_t)R ? q : (uint32_t)R;
            for (uint32_t t = 0; t < last; ++t) {
                const uint32_t qq = q - 1 - t;
                if (!mbar_wait(smem_u32(&M.full[qq % R]), (qq / R) & 1)) set_status(A.status, PSR_ETIMEOUT);
            }
            if (*ab) set_status(A.status, PSR_ETIMEOUT);
        }
    } else if (warp == NW + 1) {
        // ------------------------------------------------ MMA issue
        if (!M.abort_flag) {
            // Issuing a slice's four MMAs (256 cycles of the tensor core) must not
            // take longer than they do.  So the order of the slices
            // (fwd2d_tc_schedule) is in loops, and the whole warp walks them with
            // every value uniform, electing a lane for the MMAs and commits only:
            // descriptors then stay in uniform registers, where the MMA takes them.
            // E_loc of the 16 x 16 model: 9.31 ms with one thread reading a list of
            // operations from the kernel's parameters (730 cycles a slice), 8.60 with
            // one thread in loops, 7.79 so.
            auto wait_u = [&](uint32_t bar, uint32_t parity) {
                return __all_sync(0xffffffffu, wait_ab(bar, parity, ab)) != 0;
            };
            // slices consumed; ring slot and the full barriers' phase; e2m and
            // h_V barrier phases
            uint32_t q = 0, slot = 0, fph = 0, pe = 0, ph = 0;
            const uint32_t e2m = smem_u32(&M.e2m[0]), m2e = smem_u32(&M.m2e[0]);
            const uint32_t hset = smem_u32(&M.hset), hfree = smem_u32(&M.hfree);
            const uint32_t fb = smem_u32(&M.full[0]), ebar = smem_u32(&M.empty[0]);
            const uint64_t xd = kdesc(smem_u32(xt)), hd = kdesc(smem_u32(ht)), rd = kdesc(smem_u32(ring));
            constexpr int HL = NH - 1;  // last unit half
            bool ok = true;
            // the next nk slices: accumulator columns d, K chunks of tile b, added to
            // the accumulator from the first K step if acc
            auto run = [&](uint32_t d, uint64_t b, int nk, uint32_t acc) {
#pragma unroll 1
                for (int kc = 0; kc < nk && ok; ++kc) {
                    // the weight slice has landed (bulk-copy transactions)
                    if (!wait_u(fb + 8 * slot, fph)) { ok = false; break; }
                    const uint64_t ad = rd + (uint64_t)(slot * (kSlice >> 4));
                    if (elect1()) {
                        mma_ss<idesc2<F16>()>(d, ad, b, acc);
                        mma_ss<idesc2<F16>()>(d, ad + kstep(1), b + kstep(1), 1u);
                        mma_ss<idesc2<F16>()>(d, ad + kstep(2), b + kstep(2), 1u);
                        mma_ss<idesc2<F16>()>(d, ad + kstep(3), b + kstep(3), 1u);
                        mma_commit(ebar + 8 * slot);
                    }
                    __syncwarp();
                    acc = 1u;
                    b += 16384u >> 4;
                    ++q;
                    if (++slot == (uint32_t)R) {
                        slot = 0;
                        fph ^= 1u;
                    }
                }
            };
            // half g's epilogue has arrived
            auto wait_e = [&](int g) {
                ok = ok && wait_u(e2m + 8 * g, (pe >> g) & 1u);
                pe ^= 1u << g;
                tc_after();
            };
            auto commit = [&](int g) {
                if (ok && elect1()) mma_commit(m2e + 8 * g);
                __syncwarp();
            };
            for (uint32_t row = 0; ok; ++row) {
                if (!wait_u(smem_u32(&M.go[row & 1]), (row >> 1) & 1)) {
                    ok = false;
                    break;
                }
                if (!*(volatile int *)&M.go_flag[row & 1]) break;
#pragma unroll 1
                for (int l = 0; l < nL && ok; ++l) {
                    const int kin = l == 0 ? 1 : KC;
                    // W_hv h_V needs only the h_V image of the layer: above layer 0 it
                    // runs while the epilogue computes the layer input
                    if (l > 0) {
                        commit(HL);         // the last half's output map of layer l - 1
                        if (elect1()) mma_commit(hfree);  // and the last MMAs on the h tile
                    }
                    ok = ok && wait_u(hvb, ph);
                    ph ^= 1u;
                    tc_after();
#pragma unroll 1
                    for (int g = 0; g < NH; ++g) run(tmem + 128u * (NH + g), hd, KC, 0u);
                    // W_z x, W_hx x once x is complete; half g's projections are
                    // committed (its scan may start) before half g + 1's are issued
                    for (int g = 0; g < NH; ++g) wait_e(g);
#pragma unroll 1
                    for (int g = 0; g < NH; ++g) {
                        if (g > 0) commit(g - 1);
                        run(tmem + 128u * g, xd, kin, 0u);
                        run(tmem + 128u * (NH + g), xd, kin, 1u);
                    }
                    commit(HL);
                    // D x of half g once half g's scan has consumed z; C h once every
                    // half's scan has written h (then h is also stored as the next
                    // row's h_V); half g's output map committed before half g + 1's C
#pragma unroll 1
                    for (int g = 0; g < NH; ++g) {
                        wait_e(g);
                        if (g == HL && ok && lane == 0) mbar_arrive(hset);
                        run(tmem + 128u * g, xd, kin, 0u);
                    }
#pragma unroll 1
                    for (int g = 0; g < NH; ++g) {
                        if (g > 0) commit(g - 1);
                        run(tmem + 128u * g, hd, KC, 1u);
                    }
                }
                // readout once both halves' layer input of the readout (x) is complete
                commit(HL);
                for (int g = 0; g < NH; ++g) wait_e(g);
                run(tmem, xd, KC, 0u);
                for (int g = 0; g < NH; ++g) commit(g);  // logits of the row
            }
            // the MMAs of the last slices complete before the CTA may exit
            const uint32_t last = q < (uint32_t)R ? q : (uint32_t)R;
            for (uint32_t t = 0; t < last; ++t) {
                const uint32_t qq = q - 1 - t;
                if (!mbar_wait(smem_u32(&M.empty[qq % R]), (qq / R) & 1)) set_status(A.status, PSR_ETIMEOUT);
            }
            if (!ok && lane == 0) {
                M.abort_flag = 1;
                set_status(A.status, PSR_ETIMEOUT);
            }
        }
    } else if (warp == NW + 2) {
        // ------------------------------------------------ h_V images
        // Lane pairs (slot, K chunk): loads of the row's h_V of each layer, then
        // stores of the layer's h as the next row's h_V.
        if (!M.abort_flag) {
            static_assert(kMaxSlots * KC <= 64, "two (slot, K chunk) pairs a lane");
            const uint32_t ha = smem_u32(ht), piece = (uint32_t)W * 128u;
            uint32_t armed = 0, nh = 0, nf = 0;  // loads, hset and hfree phases so far
            auto wait_w = [&](uint32_t bar, uint32_t parity) {
                bool w = false;
                if (lane == 0) w = wait_ab(bar, parity, ab);
                w = __shfl_sync(0xffffffffu, w ? 1 : 0, 0) != 0;
                __syncwarp();
                return w;
            };
            for (uint32_t row = 0;; ++row) {
                if (!wait_w(smem_u32(&M.go[row & 1]), (row >> 1) & 1)) break;
                if (!*(volatile int *)&M.go_flag[row & 1]) break;
                if (!wait_w(smem_u32(&M.slots), row & 1)) break;
                const uint8_t *src[2] = {nullptr, nullptr};
                uint8_t *dst[2] = {nullptr, nullptr};
                uint32_t sstep[2] = {0, 0}, at[2] = {0, 0}, bytes = 0;
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    const int id = lane + 32 * k, s = id / KC, kc = id - s * KC;
                    if (s >= S || M.slot[s].job < 0) continue;
                    const Slot2 &st = M.slot[s];
                    const size_t o = (size_t)kc * piece;
                    src[k] = img_src(st, s, 0) + o;
                    sstep[k] = (st.row == 0) ? 0u : img_bytes;  // one zero image for all layers
                    dst[k] = img_dst(st, s, 0);
                    if (dst[k]) dst[k] += o;
                    at[k] = ha + (uint32_t)kc * 16384u + (uint32_t)s * piece;
                    bytes += piece;
                }
                bytes = __reduce_add_sync(0xffffffffu, bytes);
                auto load = [&](int l) {
                    if (lane == 0) mbar_arrive_tx(hvb, bytes);
                    ++armed;
                    __syncwarp();
#pragma unroll
                    for (int k = 0; k < 2; ++k)
                        if (src[k]) bulk_g2s(at[k], src[k] + (size_t)l * sstep[k], piece, hvb);
                };
                load(0);
                bool ok = true;
                for (int l = 0; l < nL && ok; ++l) {
                    // the scan has written h: it is the next row's h_V of layer l
                    ok = wait_w(smem_u32(&M.hset), nh++ & 1);
                    if (!ok) break;
#pragma unroll
                    for (int k = 0; k < 2; ++k)
                        if (dst[k]) bulk_s2g(dst[k] + (size_t)l * img_bytes, at[k], piece);
                    bulk_commit();
                    if (l + 1 < nL) {
                        // h_V of layer l + 1 lands in the h tile once the stores and
                        // the output map's MMAs have read it
                        bulk_wait_read();
                        ok = wait_w(smem_u32(&M.hfree), nf++ & 1);
                        if (ok) load(l + 1);
                    }
                }
                // the row's image stores are complete before its successor reads them
                bulk_wait_all();
                __syncwarp();
                if (!ok) break;
            }
            bulk_wait_all();
            // loads still in flight land before the CTA may exit
            if (lane == 0 && armed > 0 && !mbar_wait(hvb, (armed - 1) & 1)) set_status(A.status, PSR_ETIMEOUT);
        }
    } else {
        // ------------------------------------------------ epilogue
        // warp w reads tensor-memory lanes 32 (w & 3) ..; warpgroup w >> 2
        // takes unit half g and column group cg (slots s = cg, cg + CG, ...)
        const int q4 = warp & 3, wg = warp >> 2, g = wg % NH, cg = wg / NH;
        const int j = 128 * g + 32 * q4 + lane;  // hidden unit
        const uint32_t lane_off = (uint32_t)(q4 * 32) << 16;
        const uint32_t tz = tmem + lane_off + 128u * g;          // z, then y
        const uint32_t tcc = tmem + lane_off + 128u * (NH + g);  // c
        const uint32_t tlg = tmem + lane_off;                     // logits (lanes 32 q4 + 0..15)
        // unit j's element of row k (mod 8) of a K-major tile, 128-byte swizzle
        // (16-byte group c of row k at c ^ (k & 7)); rows n .. n + 7 of a tile, n a
        // multiple of 8, are at tile + 128 n + koff[0 .. 7]
        uint32_t koff[8];
#pragma unroll
        for (int k = 0; k < 8; ++k)
            koff[k] = (uint32_t)(j >> 6) * 16384u + 128u * k + ((uint32_t)(((j & 63) >> 3) ^ k) << 4) + (uint32_t)(j & 7) * 2u;
        const uint32_t hta = smem_u32(ht), xta = smem_u32(xt);
        auto st16 = [&](uint32_t a, uint16_t v) { asm volatile("st.shared.b16 [%0], %1;" ::"r"(a), "h"(v)); };
        float *res = A.res + (size_t)blockIdx.x * 2 * kCols * H;
        uint32_t pm = 0;  // m2e phase of this thread's unit half
        bool ok = !M.abort_flag;
        // this unit half's barriers, named barrier (2 + g) and leader thread
        const uint32_t e2m = smem_u32(&M.e2m[g]), m2e = smem_u32(&M.m2e[g]);
        const uint32_t hbar = 2u + (uint32_t)g, hcount = (uint32_t)(kEpi / NH);
        const bool leader = tid == 128 * g;

        // One thread polls the MMA thread's barrier and a named barrier
        // releases the others (hundreds of pollers would contend for the
        // shared memory the tensor core reads its operands from); the
        // epilogue's signal is one arrival after a named barrier.
        auto wait_m2e = [&]() {
            bool w = true;
            if (leader) w = ok && wait_ab(m2e, pm, ab);
            const bool bad = named_bar_or(hbar, hcount, !w || !ok);
            if (bad && ok && leader) {
                M.abort_flag = 1;
                set_status(A.status, PSR_ETIMEOUT);
            }
            ok = ok && !bad;
            pm ^= 1u;
            tc_after();
        };
        auto arrive_e2m = [&]() {
            fence_proxy_async();  // this thread's tile writes, before the MMAs read them
            tc_before();
            named_bar(hbar, hcount);
            if (leader) mbar_arrive(e2m);
        };
        // Runs go(v, s, cc, n) for the 8-column chunks (columns n .. n + 7, chunk cc
        // in path order of slot s) of this thread's active slots, with the next
        // chunk's loads ld(v, n) in flight: a chunk's loads, gates and serial scan
        // are a chain of latencies that four warps per scheduler do not cover.
        // Columns past P_x are computed like the others: a column's values reach
        // no other column but through the scan, which starts after them.
        auto chunks = [&](auto &&ld, auto &&go) {
            auto next = [&](int &s, int &cc) {
                if (++cc == nch) {
                    cc = 0;
                    s += CG;
                    while (s < S && M.slot[s].job < 0) s += CG;
                }
                return s < S;
            };
            auto col = [&](int s, int cc) { return s * W + 8 * ((M.slot[s].row & 1) ? nch - 1 - cc : cc); };
            auto wait = [&](uint32_t(&v)[16]) { asm volatile("tcgen05.wait::ld.sync.aligned;" : PSR_P16(v, 0)::"memory"); };
            uint32_t va[16], vb[16];
            int s = cg - CG, cc = nch - 1;
            bool more = next(s, cc);
            if (more) ld(va, col(s, cc));
            while (more) {
                int s2 = s, c2 = cc;
                more = next(s2, c2);
                wait(va);
                if (more) ld(vb, col(s2, c2));
                go(va, s, cc, col(s, cc));
                if (!more) break;
                s = s2;
                cc = c2;
                more = next(s2, c2);
                wait(vb);
                if (more) ld(va, col(s2, c2));
                go(vb, s, cc, col(s, cc));
                s = s2;
                cc = c2;
            }
        };
        // Adds the pending row's readout sums to its job's total (fixed order), and
        // stores the job's result if that was its last row; then the current row is
        // the pending one (slot s, its warp).
        auto fold = [&](int s) {
            Slot2 &st = M.slot[s];
            if (lane == 0) {
                if (st.pend) {
                    float a = st.acc;
                    for (int c = 0; c < nch; ++c) a += st.part[c];
                    if (st.pend_last) A.out[st.pend_out] = 0.5f * a;
                    st.acc = st.pend_last ? 0.0f : a;
                }
                st.pend = st.job >= 0;
                st.pend_last = st.row + 1 >= Py;
                st.pend_out = st.out;
            }
            __syncwarp();
        };

        // slot update (warp s for slot s): finished or empty slots take the next
        // job, the others advance one patch row
        auto update = [&]() {
            for (int s = warp; s < S; s += NW) {
                Slot2 &st = M.slot[s];
                fold(s);
                const int job = st.job;
                if (job == -2) continue;
                const uint8_t *sp;
                int r;
                if (job == -1 || st.row + 1 >= Py) {
                    unsigned long long nj = 0;
                    if (lane == 0) nj = atomicAdd(A.job_counter, 1ull);
                    nj = __shfl_sync(0xffffffffu, nj, 0);
                    if ((long long)nj >= njobs) {
                        if (lane == 0) st.job = -2;
                        __syncwarp();
                        continue;
                    }
                    int sample = (int)nj, p = -1, qq = -1, r0 = 0;
                    int64_t place = (int64_t)nj;
                    if (A.mode == 1) {
                        const int64_t set = A.images > 1 ? (uint32_t)nj / (uint32_t)per_set : 0u;
                        place += set * (A.n_jobs - per_set);
                        const int32_t *e = A.entries + 3 * place;
                        sample = (int)(set * A.n_samples) + e[0];
                        p = e[1];
                        qq = e[2];
                        r0 = (p / Lx) >> 1;
                    }
                    sp = A.spins + (size_t)sample * N;
                    int up = 0;
                    for (int t = lane; t < 2 * r0 * Lx; t += 32) up += sp[t] & 1;
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) up += __shfl_xor_sync(0xffffffffu, up, o);
                    if (lane < Px) {
                        if (r0 > 0) st.vprev[lane] = (uint8_t)patch_value(sp, Lx, lane, r0 - 1, -1, -1);
                        st.v[lane] = (uint8_t)patch_value(sp, Lx, lane, r0, p, qq);
                    }
                    if (lane == 0) {
                        st.job = 0;
                        st.out = place;
                        st.sample = sample;
                        st.p = p;
                        st.q = qq;
                        st.row = r0;
                        st.r0 = r0;
                        st.n_up = up;
                    }
                    r = r0;
                } else {
                    r = st.row + 1;
                    sp = A.spins + (size_t)st.sample * N;
                    int pc = 0;
                    if (lane < Px) {
                        const int old = st.v[lane];
                        pc = __popc(old);
                        st.vprev[lane] = (uint8_t)old;
                        st.v[lane] = (uint8_t)patch_value(sp, Lx, lane, r, st.p, st.q);
                    }
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) pc += __shfl_xor_sync(0xffffffffu, pc, o);
                    if (lane == 0) {
                        st.n_up += pc;
                        st.row = r;
                    }
                }
                __syncwarp();
            }
        };
        // the slots of row step `row` are set: does a row step follow it?
        auto signal = [&](uint32_t row) {
            if (tid == 0) {
                bool more = false;
                for (int s = 0; s < S; ++s)
                    if (M.slot[s].job >= 0 && M.slot[s].row + 1 < Py) more = true;
                if (!more) more = (long long)atomicAdd(A.job_counter, 0ull) < njobs;
                M.go_flag[(row + 1) & 1] = more ? 1 : 0;
                mbar_arrive(smem_u32(&M.go[(row + 1) & 1]));
                mbar_arrive(smem_u32(&M.slots));
            }
        };
        // Readout: masked 16-way softmax of every patch of a row; warp w takes
        // columns 8 w .. 8 w + 7 (slot w / nch, chunk w % nch).  prepare() takes what
        // it needs of the row from the slot, softmax() runs once the next row's input
        // is written, while that row's first MMAs run (E_loc of the 16 x 16 model:
        // 7.82 ms with the readout and the slot update in line, 7.45 so).
        bool ro = false;                  // this warp has a row to read out
        uint32_t lr[8], allowed = 0, vals = 0;  // logits; bit e: this lane's value allowed in column e; 4-bit values
        int ncol = 0, dirn = 1;
        int64_t pos = 0;                  // place of column 0 in logp_out
        float ref = 0.0f;
        auto prepare = [&]() {
            const int s = warp / nch, i0 = 8 * (warp - s * nch);
            ro = warp < S * nch && M.slot[s].job >= 0;
            // (all set anew: none of them lives through the layers)
            allowed = vals = 0;
            ncol = 0;
            dirn = 1;
            pos = 0;
            ref = 0.0f;
            if (!ro) return;
            const Slot2 &st = M.slot[s];
            const int r = st.row;
            const bool odd = r & 1;
            const int pc_lane = __popc(lane & 15);
            ncol = min(8, Px - i0);
            dirn = odd ? -1 : 1;
            const int k0 = odd ? Px - 1 - i0 : i0;  // path position of column i0
            pos = (int64_t)st.sample * Np + r * Px + k0;
            ref = (A.mode == 1 && lane < ncol) ? A.logp_ref[pos + dirn * lane] : 0.0f;
            // up spins of the row's patches before path position `lane`
            const int c = odd ? Px - 1 - lane : lane;  // column at path position lane
            const int pc = lane < Px ? __popc(st.v[c]) : 0;
            int incl = pc;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int t = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += t;
            }
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const int k = k0 + dirn * e;
                const int up = st.n_up + __shfl_sync(0xffffffffu, incl - pc, k);
                const int down = 2 * r * Lx + 4 * k - up;
                if (!A.u1 || (up + pc_lane <= N / 2 && down + 4 - pc_lane <= N / 2)) allowed |= 1u << e;
                vals |= (uint32_t)(st.v[i0 + e] & 15) << (4 * e);
            }
        };
        auto softmax = [&]() {
            if (!ro) return;
            // the eight columns side by side (a column's two reductions are a
            // chain of eight shuffles); columns past P_x are not summed
            const float bo = A.theta[A.tl.bo + (lane & 15)];
            float lg[8], m[8], ex[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                lg[e] = __uint_as_float(lr[e]) + bo;
                m[e] = (allowed >> e) & 1u ? lg[e] : -INFINITY;
            }
#pragma unroll
            for (int o = 8; o > 0; o >>= 1)
#pragma unroll
                for (int e = 0; e < 8; ++e) m[e] = fmaxf(m[e], __shfl_xor_sync(0xffffffffu, m[e], o, 16));
#pragma unroll
            for (int e = 0; e < 8; ++e) ex[e] = (allowed >> e) & 1u ? __expf(lg[e] - m[e]) : 0.0f;
#pragma unroll
            for (int o = 8; o > 0; o >>= 1)
#pragma unroll
                for (int e = 0; e < 8; ++e) ex[e] += __shfl_xor_sync(0xffffffffu, ex[e], o, 16);
            float rsum = 0.0f;
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                float lp = (allowed >> e) & 1u ? lg[e] - m[e] - __logf(ex[e]) : -INFINITY;
                lp = __shfl_sync(0xffffffffu, lp, (vals >> (4 * e)) & 15u);
                const float rf = __shfl_sync(0xffffffffu, ref, e);
                if (e >= ncol) continue;
                if (A.mode != 1 && A.logp_out && lane == 0) A.logp_out[pos + dirn * e] = lp;
                rsum += A.mode == 1 ? lp - rf : lp;
            }
            if (lane == 0) M.slot[warp / nch].part[warp % nch] = rsum;
        };

        if (ok) update();
        if (epi_bar_or(!ok || *ab)) ok = false;
        if (ok) signal(0);
        for (uint32_t row_it = 0; ok; ++row_it) {
            // ---- layer-0 input: one-hot (v_H, v_V) of every column, K chunk 0
            {
                constexpr uint32_t kOne = F16 ? 0x3C00u : 0x3F80u;  // 1.0
                for (int id = tid; id < kCols * 8; id += kEpi) {
                    const int n = id >> 3, c = id & 7, s = n / W, i = n - s * W;
                    int vh = -1, vv = -1;
                    if (s < S && i < Px) {
                        const Slot2 &st = M.slot[s];
                        if (st.job >= 0) {
                            const bool odd = st.row & 1;
                            // the previous patch on the path: column i - 1 (even rows) or i + 1
                            if (odd ? (i + 1 < Px) : (i > 0)) vh = st.v[odd ? i + 1 : i - 1];
                            if (st.row > 0) vv = 16 + st.vprev[i];
                        }
                    }
                    uint32_t w4[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const int e0 = 8 * c + 2 * e, e1 = e0 + 1;
                        const uint32_t lo = (e0 == vh || e0 == vv) ? kOne : 0u;
                        const uint32_t hi = (e1 == vh || e1 == vv) ? kOne : 0u;
                        w4[e] = lo | (hi << 16);
                    }
                    *reinterpret_cast<uint4 *>(xt + n * 128 + ((c ^ (n & 7)) << 4)) =
                        make_uint4(w4[0], w4[1], w4[2], w4[3]);
                }
            }
            arrive_e2m();
            if (row_it > 0 && ok) softmax();  // of the row before

            for (int l = 0; l < nL; ++l) {
                // ---- gates and scan along each slot's row (path order)
                wait_m2e();
                {
                    const float hbz = 0.5f * A.theta[A.tl.bz[l] + j], bh = A.theta[A.tl.bh[l] + j];
                    const float2 hbz2 = make_float2(hbz, hbz), bh2 = make_float2(bh, bh);
                    const bool keep_res = (l >= 1) && (l + 1 < nL);
                    float *resw = res + (size_t)(l & 1) * kCols * H;
                    float h = 0.0f;
                    chunks(
                        [&](uint32_t(&v)[16], int n) {
                            tmem_ld8(tz + n, v[0], v[1], v[2], v[3], v[4], v[5], v[6], v[7]);
                            tmem_ld8(tcc + n, v[8], v[9], v[10], v[11], v[12], v[13], v[14], v[15]);
                        },
                        [&](uint32_t(&v)[16], int s, int cc, int n) {
                            float av[8], bv[8];
#pragma unroll
                            for (int k = 0; k < 8; k += 2) {
                                float2 a2, b2;
                                gates2(make_float2(__uint_as_float(v[k]), __uint_as_float(v[k + 1])),
                                       make_float2(__uint_as_float(v[8 + k]), __uint_as_float(v[9 + k])), hbz2, bh2, a2,
                                       b2);
                                av[k] = a2.x;
                                av[k + 1] = a2.y;
                                bv[k] = b2.x;
                                bv[k + 1] = b2.y;
                            }
                            if (cc == 0) h = 0.0f;  // the row starts from h_H = 0
                            const uint32_t a = hta + 128u * n;
                            if (M.slot[s].row & 1) {
                                const int k0 = Px - 1 - (n - s * W);  // the path's first column, if in this chunk
#pragma unroll
                                for (int k = 7; k >= 0; --k) {
                                    if (k == k0) h = 0.0f;
                                    h = fmaf(av[k], h, bv[k]);
                                    bv[k] = h;
                                    st16(a + koff[k], op_bits<F16>(h));
                                }
                            } else {
#pragma unroll
                                for (int k = 0; k < 8; ++k) {
                                    h = fmaf(av[k], h, bv[k]);
                                    bv[k] = h;
                                    st16(a + koff[k], op_bits<F16>(h));
                                }
                            }
                            if (keep_res) {
#pragma unroll
                                for (int k = 0; k < 8; ++k) resw[(size_t)(n + k) * H + j] = bv[k];
                            }
                        });
                }
                arrive_e2m();

                // ---- output map: x = GELU(y + residual)
                wait_m2e();
                {
                    const bool use_res = (l >= 2);
                    const float *resr = res + (size_t)((l - 1) & 1) * kCols * H;
                    chunks(
                        [&](uint32_t(&v)[16], int n) {
                            tmem_ld8(tz + n, v[0], v[1], v[2], v[3], v[4], v[5], v[6], v[7]);
#pragma unroll
                            for (int k = 0; k < 8; ++k)
                                v[8 + k] = use_res ? __float_as_uint(resr[(size_t)(n + k) * H + j]) : 0u;
                        },
                        [&](uint32_t(&v)[16], int, int, int n) {
                            const uint32_t a = xta + 128u * n;
#pragma unroll
                            for (int k = 0; k < 8; k += 2) {
                                const float2 x = gelu_bf16out2(
                                    __fadd2_rn(make_float2(__uint_as_float(v[k]), __uint_as_float(v[k + 1])),
                                               make_float2(__uint_as_float(v[8 + k]), __uint_as_float(v[9 + k]))));
                                st16(a + koff[k], op_bits<F16>(x.x));
                                st16(a + koff[k + 1], op_bits<F16>(x.y));
                            }
                        });
                }
                arrive_e2m();
            }

            // ---- end of the row: what its softmax needs, then the slots of the next
            // row (the MMA and image warps start on it), then the logits
            prepare();
            if (epi_bar_or(!ok || *ab)) {
                ok = false;
                break;
            }
            const bool last = !*(volatile int *)&M.go_flag[(row_it + 1) & 1];
            if (!last) update();
            else
                for (int s = warp; s < S; s += NW) fold(s);
            if (epi_bar_or(!ok)) {
                ok = false;
                break;
            }
            if (!last) signal(row_it + 1);
            wait_m2e();
#pragma unroll
            for (int e = 0; e < 8; ++e) lr[e] = 0;
            if (ro) {
                tmem_ld8(tlg + 8 * warp, lr[0], lr[1], lr[2], lr[3], lr[4], lr[5], lr[6], lr[7]);
                asm volatile("tcgen05.wait::ld.sync.aligned;"
                             : "+r"(lr[0]), "+r"(lr[1]), "+r"(lr[2]), "+r"(lr[3]), "+r"(lr[4]), "+r"(lr[5]),
                               "+r"(lr[6]), "+r"(lr[7])::"memory");
            }
            if (last) {
                if (ok) softmax();
                if (epi_bar_or(!ok)) {
                    ok = false;
                    break;
                }
                for (int s = warp; s < S; s += NW) fold(s);
                break;
            }
        }
        if (!ok) {
            M.abort_flag = 1;
            set_status(A.status, PSR_ETIMEOUT);
        }
    }
    tc_before();
    __syncthreads();
    if (warp == 0) {
        tc_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
    }
}

template <int H>
size_t fwd2d_tc_smem(int R) {
    return sizeof(Misc2) + 1024 + 2 * (size_t)(H / 64) * 16384 + (size_t)R * kSlice;
}

template <int H, bool F16>
cudaError_t launch_h(const Fwd2TcArgs &a, int grid, cudaStream_t stream) {
    const size_t smem = fwd2d_tc_smem<H>(a.R);
    cudaError_t e =
        cudaFuncSetAttribute(fwd2d_tc_kernel<H, F16>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    fwd2d_tc_kernel<H, F16><<<grid, kThreads2, smem, stream>>>(a);
    return cudaGetLastError();
}

// Weight slices in MMA order: 128 rows (units 128 g ..) x 64 inputs (64 kc ..)
// of one matrix, 128-byte swizzle (16-byte chunk c of row m at c ^ (m & 7)).
template <bool F16>
__global__ void pack2d_tc_kernel(const float *__restrict__ theta, T2Layout tl, Sched2 sc,
                                 uint8_t *__restrict__ wimg) {
    const int H = tl.H;
    const int64_t total = (int64_t)sc.n * 1024;
    for (int64_t id = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; id < total;
         id += (int64_t)gridDim.x * blockDim.x) {
        const int i = (int)(id >> 10), m = (int)((id >> 3) & 127), c = (int)(id & 7);
        const int ty = sc.type[i], l = sc.l[i], unit = 128 * sc.g[i] + m, k0 = 64 * sc.kc[i] + 8 * c;
        const int din = l == 0 ? 32 : H;
        uint32_t w[4];
#pragma unroll
        for (int e2 = 0; e2 < 4; ++e2) {
            float v2[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int k = k0 + 2 * e2 + h;
                float v = 0.0f;
                switch (ty) {
                    case kMtWz: if (k < din) v = theta[tl.Wz[l] + (int64_t)unit * din + k]; break;
                    case kMtWhx: if (k < din) v = theta[tl.Wh[l] + (int64_t)unit * (din + H) + k]; break;
                    case kMtWhv: v = theta[tl.Wh[l] + (int64_t)unit * (din + H) + din + k]; break;
                    case kMtC: v = theta[tl.C[l] + (int64_t)unit * H + k]; break;
                    case kMtD: if (k < din) v = theta[tl.D[l] + (int64_t)unit * din + k]; break;
                    default:  // W_o in rows 32 q + o of every lane quarter q
                        if ((unit & 31) < 16) v = theta[tl.Wo + (int64_t)(unit & 31) * H + k];
                        break;
                }
                v2[h] = v;
            }
            w[e2] = op_pack<F16>(v2[0], v2[1]);
        }
        *reinterpret_cast<uint4 *>(wimg + (size_t)i * kSlice + m * 128 + ((c ^ (m & 7)) << 4)) =
            make_uint4(w[0], w[1], w[2], w[3]);
    }
}

}  // namespace

// Slices of one row step, in the order the MMA thread consumes them.
Sched2 fwd2d_tc_schedule(int nL, int H) {
    Sched2 sc{};
    const int NH = H / 128, KC = H / 64;
    int n = 0;
    auto add = [&](int ty, int l, int g, int nk) {
        for (int kc = 0; kc < nk; ++kc, ++n) {
            sc.type[n] = (uint8_t)ty;
            sc.l[n] = (uint8_t)l;
            sc.g[n] = (uint8_t)g;
            sc.kc[n] = (uint8_t)kc;
        }
    };
    for (int l = 0; l < nL; ++l) {
        const int kin = l == 0 ? 1 : KC;
        for (int g = 0; g < NH; ++g) add(kMtWhv, l, g, KC);
        for (int g = 0; g < NH; ++g) {
            add(kMtWz, l, g, kin);
            add(kMtWhx, l, g, kin);
        }
        for (int g = 0; g < NH; ++g) add(kMtD, l, g, kin);
        for (int g = 0; g < NH; ++g) add(kMtC, l, g, KC);
    }
    add(kMtWo, 0, 0, KC);
    sc.n = n;
    return sc;
}

bool fwd2d_tc_supported(int nL, int H, int Lx) {
    return (H == 128 || H == 256) && nL >= 1 && nL <= kMaxLayers && Lx >= 2 && Lx <= 64 &&
           fwd2d_tc_schedule(nL, H).n <= kSchedMax;
}

void fwd2d_tc_geometry(int Lx, int *W, int *S) {
    const int Px = Lx / 2;
    *W = 8 * ((Px + 7) / 8);
    *S = kCols / *W;
    if (*S > kMaxSlots) *S = kMaxSlots;
}

size_t fwd2d_tc_image_bytes(int H, int Lx) {
    int W, S;
    fwd2d_tc_geometry(Lx, &W, &S);
    return (size_t)(H / 64) * W * 128;
}

size_t fwd2d_tc_weight_bytes(int nL, int H) { return (size_t)fwd2d_tc_schedule(nL, H).n * kSlice; }

size_t fwd2d_tc_ckpt_bytes(int nL, int H, int Lx, int Ly) {
    return (size_t)(Ly / 2) * nL * fwd2d_tc_image_bytes(H, Lx);
}

size_t fwd2d_tc_scratch_bytes(int nL, int H, int Lx, int grid) {
    int W, S;
    fwd2d_tc_geometry(Lx, &W, &S);
    return (size_t)grid * S * nL * fwd2d_tc_image_bytes(H, Lx);
}

size_t fwd2d_tc_res_floats(int H, int grid) { return (size_t)grid * 2 * kCols * H; }

cudaError_t launch_pack2d_tc(const float *theta, const T2Layout &tl, bool f16, uint8_t *wimg,
                             cudaStream_t stream) {
    const Sched2 sc = fwd2d_tc_schedule(tl.nL, tl.H);
    const int64_t total = (int64_t)sc.n * 1024;
    const int blocks = (int)((total + 255) / 256);
    if (f16) pack2d_tc_kernel<true><<<blocks, 256, 0, stream>>>(theta, tl, sc, wimg);
    else pack2d_tc_kernel<false><<<blocks, 256, 0, stream>>>(theta, tl, sc, wimg);
    return cudaGetLastError();
}

cudaError_t launch_fwd2d_tc(Fwd2TcArgs a, int grid, cudaStream_t stream) {
    int dev = 0, optin = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e != cudaSuccess) return e;
    const int H = a.tl.H;
    fwd2d_tc_geometry(a.Lx, &a.W, &a.S);
    a.n_slices = fwd2d_tc_schedule(a.tl.nL, H).n;
    const size_t base = (H == 256) ? fwd2d_tc_smem<256>(0) : fwd2d_tc_smem<128>(0);
    if ((size_t)optin < base + 2 * kSlice) return cudaErrorInvalidConfiguration;
    int R = (int)(((size_t)optin - base) / kSlice);
    a.R = R > kMaxRing ? kMaxRing : R;
    if (grid < 1) grid = 1;
    switch (H) {
        case 128: return a.f16 ? launch_h<128, true>(a, grid, stream) : launch_h<128, false>(a, grid, stream);
        case 256: return a.f16 ? launch_h<256, true>(a, grid, stream) : launch_h<256, false>(a, grid, stream);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace psr
