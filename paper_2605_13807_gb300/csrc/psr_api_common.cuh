// Internal helpers of the C ABI shared by the psr_api*.cu files: the
// context object, workspace carving, host/device staging, argument checks,
// per-stage events, the connected-configuration generator sequence and the
// autotuner's measurement loop.  Not part of the public ABI.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <cstdio>
#include <cstring>
#include <functional>
#include <new>
#include <vector>

#include "psr_internal.cuh"

namespace psr {
namespace apiutil {
// Bytes of layer arrays that a batch of a layered gradient may hold, unless
// psr_context_set_memory says otherwise.
constexpr size_t kGradBudget = size_t(2) << 30;
}  // namespace apiutil
}  // namespace psr

struct psr_context {
    cudaStream_t stream = nullptr;
    int device = 0;
    int num_sms = 1;
    void *ws = nullptr;
    size_t ws_size = 0;
    int *status = nullptr;  // device status word
    bool profiling = false;
    bool capturing = false;  // a CUDA graph is being captured on the stream
    cudaEvent_t ev_begin[PSR_STAGE_COUNT] = {};
    cudaEvent_t ev_end[PSR_STAGE_COUNT] = {};
    bool stage_ran[PSR_STAGE_COUNT] = {};
    uint64_t ws_generation = 0;  // bumped whenever the workspace moves
    size_t ws_limit = SIZE_MAX;  // largest workspace (psr_context_set_memory)
    // bytes of layer arrays a gradient's batch takes: the budget, or less once
    // the device had no room for it (grad_fitted)
    size_t grad_fit = psr::apiutil::kGradBudget;
    bool graphs = false;
    cudaGraphExec_t graph_exec = nullptr;
    std::vector<unsigned char> graph_key;  // arguments the cached graph was built for
    uint64_t graph_ws_generation = 0;
    // Autotuner: measured choices per (operation, shape), kept for the
    // context's lifetime.
    bool autotune = false;
    struct Tuned {
        int op;
        int64_t k0, k1, k2;
        int32_t v0, v1;
        float ms;
    };
    std::vector<Tuned> tuned;
    cudaEvent_t tune_ev[2] = {};
    // shape of the fused forward kernels fixed by psr_context_set_fwd_shape
    // ([0] FP32, [1] BF16; 0 = chosen per call: tuned, else the default)
    int fwd_shape_fixed[2] = {0, 0};
    // second workspace: arrays psr_vmc_step keeps across the calls it makes
    void *ws2 = nullptr;
    size_t ws2_size = 0;
};

namespace psr {
namespace apiutil {

// Bump allocator over the workspace.  Each entry point runs its carving
// sequence twice: once with a null base to size it, once for real.
struct Carver {
    char *base = nullptr;
    size_t off = 0;
    template <class T>
    T *get(size_t count) {
        off = (off + 255) & ~size_t(255);
        T *p = base ? reinterpret_cast<T *>(base + off) : nullptr;
        off += count * sizeof(T);
        return p;
    }
};

inline int from_cuda(cudaError_t e) {
    if (e == cudaSuccess) return PSR_OK;
    if (e == cudaErrorMemoryAllocation) return PSR_ENOMEM;
    return PSR_ECUDA;
}

#define PSR_TRY(expr)                          \
    do {                                       \
        int _rc = from_cuda(expr);             \
        if (_rc != PSR_OK) return _rc;         \
    } while (0)

inline bool is_device_ptr(const void *p) {
    if (!p) return false;
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

inline int ensure_ws(psr_context *ctx, size_t bytes) {
    if (bytes <= ctx->ws_size) return PSR_OK;
    if (bytes > ctx->ws_limit) return PSR_ENOMEM;
    PSR_TRY(cudaStreamSynchronize(ctx->stream));
    if (ctx->ws) cudaFree(ctx->ws);
    ctx->ws = nullptr;
    ctx->ws_size = 0;
    size_t want = bytes + bytes / 8 + (1u << 20);
    if (want > ctx->ws_limit) want = ctx->ws_limit;
    cudaError_t e = cudaMalloc(&ctx->ws, want);
    if (e != cudaSuccess) {
        cudaGetLastError();
        ctx->ws = nullptr;
        return PSR_ENOMEM;
    }
    ctx->ws_size = want;
    ctx->ws_generation++;
    return PSR_OK;
}

// Reads and clears the device status word (synchronises the stream).
inline int take_status(psr_context *ctx) {
    PSR_TRY(cudaStreamSynchronize(ctx->stream));
    int st = 0;
    PSR_TRY(cudaMemcpy(&st, ctx->status, sizeof(int), cudaMemcpyDeviceToHost));
    if (st != 0) PSR_TRY(cudaMemset(ctx->status, 0, sizeof(int)));
    return st;
}

inline int check_params(const psr_params *p, int64_t n, int32_t L) {
    if (!p || !p->ctx || !p->theta) return PSR_EINVAL;
    if (p->n_layers < 1 || p->n_layers > kMaxLayers) return PSR_EINVAL;
    if (p->hidden != 32 && p->hidden != 64 && p->hidden != 128) return PSR_EINVAL;
    if (p->u1_mask != 0 && p->u1_mask != 1) return PSR_EINVAL;
    if (p->precision == PSR_FP16) return PSR_EUNSUPPORTED;  // the 2D model's forward only
    if (p->precision != PSR_FP32 && p->precision != PSR_BF16) return PSR_EINVAL;
    if (n < 1 || L < 1) return PSR_EINVAL;
    if (n > (int64_t)1 << 31) return PSR_EINVAL;
    if (p->u1_mask && (L % 2)) return PSR_EINVAL;
    if (p->precision == PSR_BF16 &&
        (p->hidden != 128 || p->n_layers != 3 || bf16_packed_bytes() == 0))
        return PSR_EUNSUPPORTED;
    return PSR_OK;
}

inline int check_ham(const psr_hamiltonian *h) {
    if (!h) return PSR_EINVAL;
    if (h->kind != PSR_HEISENBERG && h->kind != PSR_TFIM) return PSR_EINVAL;
    if (h->Lx < 1 || h->Ly < 1 || (int64_t)h->Lx * h->Ly > (1 << 24)) return PSR_EINVAL;
    if (h->pbc != 0 && h->pbc != 1) return PSR_EINVAL;
    if (h->marshall != 0 && h->marshall != 1) return PSR_EINVAL;
    if (h->kind == PSR_HEISENBERG && h->marshall) {
        // bipartite unless a wrapped dimension has odd length
        const bool wx = h->pbc && h->Lx >= 3, wy = h->pbc && h->Ly >= 3;
        if ((wx && (h->Lx & 1)) || (wy && (h->Ly & 1))) return PSR_EINVAL;
    }
    return PSR_OK;
}

inline int64_t words_per_row(int N) { return (N + 63) / 64 + 1; }

// Stages an input array: returns the device pointer to use (the caller's own
// if it is device memory, else a workspace copy filled by an async H2D).
template <class T>
inline int stage_in(const T *src, T *dst_ws, size_t count, bool dev, cudaStream_t st, const T **use) {
    if (dev) {
        *use = src;
        return PSR_OK;
    }
    PSR_TRY(cudaMemcpyAsync(dst_ws, src, count * sizeof(T), cudaMemcpyHostToDevice, st));
    *use = dst_ws;
    return PSR_OK;
}

// Records the begin/end event of a stage when profiling is on.
struct StageScope {
    psr_context *ctx;
    int stage;
    StageScope(psr_context *c, int s) : ctx(c), stage(s) {
        if (ctx->profiling && !ctx->capturing) {
            cudaEventRecord(ctx->ev_begin[stage], ctx->stream);
            ctx->stage_ran[stage] = true;
        }
    }
    ~StageScope() {
        if (ctx->profiling && !ctx->capturing) cudaEventRecord(ctx->ev_end[stage], ctx->stream);
    }
};

inline void reset_stages(psr_context *ctx) {
    for (int i = 0; i < PSR_STAGE_COUNT; ++i) ctx->stage_ran[i] = false;
}

// Shared body of psr_connected and the first half of every local-energy call.
struct ConnBufs {
    int32_t *bonds;
    int64_t *counts;
    int64_t *offsets;
    float *diag;
    int32_t *entries;
};

inline int enqueue_connected(psr_context *ctx, const psr_hamiltonian *ham, const uint8_t *sp, int64_t n,
                      const ConnBufs &b, HamDev &hd) {
    cudaStream_t st = ctx->stream;
    const int N = ham->Lx * ham->Ly;
    hd.kind = ham->kind;
    hd.N = N;
    hd.nb = bond_count(ham->Lx, ham->Ly, ham->pbc);
    hd.bonds = b.bonds;
    hd.J = (float)ham->J;
    hd.h = (float)ham->h;
    hd.coeff = ham->kind == PSR_HEISENBERG ? (float)((ham->marshall ? -0.5 : 0.5) * ham->J)
                                           : (float)(-ham->h);
    if (hd.nb > 0) PSR_TRY(launch_bonds(ham->Lx, ham->Ly, ham->pbc, b.bonds, st));
    PSR_TRY(launch_count_connected(hd, sp, n, b.counts, b.diag, st));
    PSR_TRY(launch_exclusive_scan(b.counts, n, b.offsets, st));
    PSR_TRY(launch_fill_connected(hd, sp, n, b.offsets, b.entries, st));
    return PSR_OK;
}

inline int64_t max_entries_per_sample(const psr_hamiltonian *ham) {
    const int N = ham->Lx * ham->Ly;
    return ham->kind == PSR_HEISENBERG ? bond_count(ham->Lx, ham->Ly, ham->pbc) : N;
}

// ---------------------------------------------------------------- autotuner

enum { kTuneScan = 1, kTuneSample = 2, kTuneSample2d = 3, kTuneSampleLru = 4, kTuneFwd = 5 };

// Times run(i) for every candidate i on the context's stream with CUDA
// events (two runs each when a run is short, the second counted) and
// returns the index of the fastest.  Synchronises the stream.
template <class Run>
int measure_candidates(psr_context *ctx, int count, Run run, int *best, float *best_ms) {
    if (!ctx->tune_ev[0]) {
        PSR_TRY(cudaEventCreate(&ctx->tune_ev[0]));
        PSR_TRY(cudaEventCreate(&ctx->tune_ev[1]));
    }
    cudaStream_t st = ctx->stream;
    *best = 0;
    *best_ms = -1.0f;
    for (int i = 0; i < count; ++i) {
        float ms = 0.0f;
        for (int rep = 0; rep < 2; ++rep) {
            PSR_TRY(cudaEventRecord(ctx->tune_ev[0], st));
            int rc = run(i);
            if (rc != PSR_OK) return rc;
            PSR_TRY(cudaEventRecord(ctx->tune_ev[1], st));
            PSR_TRY(cudaEventSynchronize(ctx->tune_ev[1]));
            PSR_TRY(cudaEventElapsedTime(&ms, ctx->tune_ev[0], ctx->tune_ev[1]));
            if (ms > 50.0f) break;  // long runs: the first is representative
        }
        if (*best_ms < 0.0f || ms < *best_ms) {
            *best_ms = ms;
            *best = i;
        }
    }
    return PSR_OK;
}

inline const psr_context::Tuned *find_tuned(const psr_context *ctx, int op, int64_t k0, int64_t k1,
                                     int64_t k2) {
    for (const auto &t : ctx->tuned)
        if (t.op == op && t.k0 == k0 && t.k1 == k1 && t.k2 == k2) return &t;
    return nullptr;
}

// ------------------------------------------- shapes of the fused forwards
// BF16 (tcgen05) forward: sequences per MMA stream, 1 (four streams, N = 32)
// or 2 (two streams, N = 64).  FP32 forward: window, 32 or 16 sites.
// Every shape computes the same function; the FP32 window changes only the
// summation order of a configuration's log P (both resume every 16 sites), the
// BF16 shapes give identical results.
constexpr int kFwdShapeDefault[2] = {kChunkF32, 1};
constexpr int kFwdShapes[2][2] = {{kChunkF32, kChunkGrad}, {1, 2}};

inline bool fwd_shape_valid(bool bf16, int shape) {
    return shape == kFwdShapes[bf16][0] || shape == kFwdShapes[bf16][1];
}

// Key of the forward launches of one call: precision, kind of call (0: log
// psi of the samples, 1: samples + connected configurations) and the
// (sites, samples) of every sample set.
struct FwdKey {
    int64_t k0, k1, k2;
};
inline FwdKey fwd_key(bool bf16, int what, int groups, const int *N, const int64_t *n) {
    uint64_t h = 1469598103934665603ull;  // FNV-1a over the sizes
    for (int g = 0; g < groups; ++g) {
        h = (h ^ (uint64_t)N[g]) * 1099511628211ull;
        h = (h ^ (uint64_t)n[g]) * 1099511628211ull;
    }
    return FwdKey{bf16 ? 1 : 0, what, (int64_t)(h >> 1)};
}

// The shape a call uses: the fixed one, else the tuned one, else the default.
inline int fwd_shape(const psr_context *ctx, bool bf16, const FwdKey &k, bool *tuned) {
    *tuned = false;
    if (ctx->fwd_shape_fixed[bf16]) return ctx->fwd_shape_fixed[bf16];
    if (const psr_context::Tuned *t = find_tuned(ctx, kTuneFwd, k.k0, k.k1, k.k2)) {
        *tuned = true;
        return t->v0;
    }
    return kFwdShapeDefault[bf16];
}

// With the autotuner on and the shape neither fixed nor tuned (and no graph
// being captured), times run(shape) for both shapes and records the faster;
// *shape receives the shape to use.  run must enqueue the call's complete
// forward launches (idempotent).  Synchronises the stream when it tunes.
template <class Run>
inline int tune_fwd_shape(psr_context *ctx, bool bf16, const FwdKey &k, Run run, int *shape) {
    bool tuned = false;
    *shape = fwd_shape(ctx, bf16, k, &tuned);
    if (!ctx->autotune || tuned || ctx->capturing || ctx->fwd_shape_fixed[bf16]) return PSR_OK;
    int best = 0;
    float ms = 0.0f;
    int rc = measure_candidates(ctx, 2, [&](int i) { return run(kFwdShapes[bf16][i]); }, &best, &ms);
    if (rc != PSR_OK) return rc;
    psr_context::Tuned t{kTuneFwd, k.k0, k.k1, k.k2, kFwdShapes[bf16][best], 0, ms};
    ctx->tuned.push_back(t);
    *shape = t.v0;
    return PSR_OK;
}

// ------------------------------------------------ gradients by layers
// The layer-by-layer gradients hold every layer's arrays of a batch of
// samples; batches are sized to the context's budget of them.  A sample that
// needs more by itself goes to the chunk-recompute kernel of its model, which
// keeps only chunk carries.

// Samples per batch for `per` floats of arrays a sample; 0: too long.
inline int64_t grad_batch(const psr_context *ctx, size_t per, int64_t sites, int64_t n) {
    const size_t bytes = per * sizeof(float);
    if (bytes > ctx->grad_fit || sites >= (int64_t)1 << 30) return 0;
    int64_t B = (int64_t)(ctx->grad_fit / bytes);
    const int64_t most = ((int64_t)1 << 30) / sites;
    if (B > most) B = most;
    return B < n ? B : n;
}

// A batch of `asked` samples found no room, one of `got` did (0: the
// chunk-recompute kernel).  Later calls start from there: each failed attempt
// waits for the stream, gives the workspace back and allocates it anew, which
// also makes psr_step_batch record its graph again.
inline void grad_fitted(psr_context *ctx, size_t per, int64_t asked, int64_t got) {
    const size_t fit = got > 0 ? (size_t)got * per * sizeof(float) : per * sizeof(float) - 1;
    if (got < asked && fit < ctx->grad_fit) ctx->grad_fit = fit;
}

// How the products of a gradient run.  FP32 sums over samples: three-part split
// operands on the tensor cores from width 64 on (error against FP64 no larger
// than with FP32 multiply-adds; the chain at hidden 64, 256 sites, 400 samples:
// 0.9e-6 against 1.5e-6).  FP32 O_k rows: CUDA cores, because a single row
// shows the tensor cores' rounding toward zero (4.4e-7 against 2.5e-7), which
// cancels in a sum.  BF16 O_k rows: two-part split.
inline gemm::Engine grad_engine(const psr_context *ctx, int H, bool sum, bool bf16_rows = false) {
    return gemm::Engine{bf16_rows ? 2 : sum && H >= 64 ? 3 : 0, ctx->num_sms, ctx->status};
}

inline bool grad_bf16_rows(const psr_params *p, const float *dout) {
    return p->precision == PSR_BF16 && p->hidden == 128 && dout == nullptr;
}

inline bool aligned16p(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

inline size_t grad_f32_floats(int nL, int H, int L) { return grad_f32_floats_per_site(nL, H) * (size_t)L; }

inline int64_t grad_f32_batch(const psr_context *ctx, int nL, int H, int L, int64_t n) {
    return grad_batch(ctx, grad_f32_floats(nL, H, L), L, n);
}

// Carves the batch arrays of launch_grad_f32 into A (sum: a weighted sum over
// the samples, else O_k rows).
inline void grad_f32_carve(Carver &c, int nL, int H, int L, int64_t B, bool sum, bool copy_theta, GradF32Args &A) {
    const size_t M = (size_t)B * L, arr = M * H;
    const int64_t P = theta_layout(nL, H).total;
    A.theta = c.get<float>(copy_theta ? P : 0);
    for (int l = 0; l < nL; ++l) {
        A.a[l] = c.get<float>(l ? arr : 0);
        A.c[l] = c.get<float>(l ? arr : 0);
        A.h[l] = c.get<float>(arr);
        A.dy[l] = c.get<float>(arr);
        A.u[l] = c.get<float>(arr);
    }
    A.gy[0] = c.get<float>(arr);
    A.gy[1] = c.get<float>(arr);
    A.gh = c.get<float>(arr);
    A.dc = c.get<float>(arr);
    A.g = c.get<float>(M);
    A.range = grad_f32_range(H, M);
    A.rows = c.get<float>(sum ? (M + A.range - 1) / A.range * P : 0);
    A.small = c.get<float>(sum ? (size_t)B * grad_f32_small_floats(H) : 0);
}

// Enqueues the gradient of n samples of L sites (bit-packed, W words a row) in
// batches of B through the arrays in A: O_k rows (dout == NULL) or the
// dout-weighted sum into out.  bf16_rows: O_k rows of the BF16 path.
inline int enqueue_grad_f32(psr_context *ctx, int nL, int H, int u1, const float *theta, const float *pk,
                            const uint64_t *bits, int64_t n, int L, int W, const float *dout, float *out,
                            int64_t B, GradF32Args A, bool bf16_rows) {
    cudaStream_t st = ctx->stream;
    A.tl = theta_layout(nL, H);
    A.fl = f32_layout(nL, H);
    const int64_t P = A.tl.total;
    if (!aligned16p(theta)) {
        PSR_TRY(cudaMemcpyAsync(const_cast<float *>(A.theta), theta, P * sizeof(float), cudaMemcpyDeviceToDevice, st));
    } else {
        A.theta = theta;
    }
    A.N = L;
    A.W = W;
    A.u1 = u1;
    A.nL = nL;
    A.H = H;
    A.pk = pk;
    A.en = grad_engine(ctx, H, dout != nullptr, bf16_rows);
    if (dout) {
        A.sm = GradSmall{0, 2 * H, 3 * H, 5 * H, 6 * H, 8 * H, 10 * H};
        A.small_stride = grad_f32_small_floats(H);
        A.sum_out = out;
    } else {
        A.sm = GradSmall{A.tl.Wz[0], A.tl.bz[0], A.tl.Wh[0], A.tl.bh[0], A.tl.D[0], A.tl.Wo, A.tl.bo};
        A.small_stride = P;
        A.sum_out = nullptr;
    }
    for (int64_t s0 = 0; s0 < n; s0 += B) {
        A.n = (int)(n - s0 < B ? n - s0 : B);
        A.bits = bits + s0 * W;
        A.dout = dout ? dout + s0 : nullptr;
        if (!dout) A.rows = A.small = out + s0 * P;
        A.add = s0 > 0;
        PSR_TRY(launch_grad_f32(A, st));
    }
    return PSR_OK;
}

// psr2d_grad whose weights depend on log psi of the same samples: one forward
// for both (psr_api_models.cu).  lp [n] receives log psi, then weights(stream)
// enqueues what writes dout [n].  PSR_ENOMEM, with nothing enqueued, if the
// samples do not fit one batch.  Device arrays only.
int grad2d_after_logpsi(const psr_params *params, const uint8_t *spins, int64_t n, int32_t Lx, int32_t Ly, float *lp,
                        const std::function<cudaError_t(cudaStream_t)> &weights, const float *dout, float *dparams);

}  // namespace apiutil
}  // namespace psr
