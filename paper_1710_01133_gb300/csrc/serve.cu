// a7: continuous-batching server.  Requests (each an independent Caputo
// problem of Sec. 2 of arXiv:1710.01133 with its own right-hand side, dim,
// alpha, h and N) wait in a host queue and are admitted as "slots" while the
// device memory they need (weights, history, output, partials) fits in the
// server's HBM budget.  Each fabm_server_step advances every admitted slot by
// one block of 32 steps with one launch over a table of slots: a CTA per slot
// for the recurrence of block c (the right-hand side dispatched at run time),
// and beside them CTAs for the far history of block c+1, which derive their
// (slot, chunk, column) items from each slot's block index; the CTA that
// finishes a slot's last items adds its chunks in a fixed order.  Stream W
// computes weights and initial values of newly admitted slots beside the step's
// launch; new slots run their first block at the next step.  Finished slots are
// copied to host memory and their device memory is returned to the
// stream-ordered pool; the freed budget admits waiting requests at the next step.
//
// A step of a few hundred slots is bound by what surrounds the kernels, so the
// host uploads the slot table only when slots were admitted or retired, requests'
// inputs in it, the device counts the blocks, and a step is one launch and one
// wait (256 requests of 2^12 to 2^14 steps: 55 -> 52 us a step,
// one request 30..36 -> 20..27; the step that admits them 4.1 -> 2.1 ms, the steps
// that return their results 7.0 -> 4.8 ms in all).  A slot's chunking depends on its own block
// index only, so its result does not depend on the other requests in flight.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <deque>
#include <memory>
#include <mutex>
#include <unordered_map>
#include <vector>

#include "history_blocks.cuh"
#include "trace.h"
#include "recurrence.cuh"
#include "weights.cuh"

using namespace fabm;

namespace {

constexpr int kSL = kRecurL;        // block length of served solves (32)
constexpr int kMaxChunksSlot = 16;  // far-history chunks per slot and block
constexpr int kMinChunkPts = 1024;  // points per chunk at least

struct SlotDev {
    int rhs, dim, hk;
    int pad;
    int64_t N, w_ext;
    int64_t *Nb;  // device copy of N (read by the recurrence)
    double *F, *Y, *y0, *params, *WB, *WA, *WD, *G;
    double *y1;  // y'(0) (dim doubles) for 1 < alpha < 2, or NULL: Taylor part y0
    float *WBf, *WAf, *Ff;  // split slots: fp32 weights and f rounded to float
    void *part;  // double (FP64) or float2 (split) partials
    StepConsts kc;
    double alpha, inv_g1;
    unsigned long long *status;
    // the block of server step e is c0 + e from step `start` on; before it the
    // slot is skipped (its weights are being computed)
    int64_t c0, start;
    // the request's inputs, copied to the buffers above when the slot is set up
    double y0v[FABM_MAX_DIM], y1v[FABM_MAX_DIM], pv[kMaxParams];
    int resumed, pad2;  // history, solution and status come from a checkpoint
};

// Chunking of block c's far history for one slot: depends on c only, so a
// request's partial sums do not depend on the other requests in flight.
__host__ __device__ inline void slot_chunks(int64_t c, int64_t *kc, int *n)
{
    const int64_t k_end = (c - 1) * kSL;
    int64_t pts = (k_end + kMaxChunksSlot - 1) / kMaxChunksSlot;
    if (pts < kMinChunkPts) pts = kMinChunkPts;
    pts = (pts + 31) / 32 * 32;
    *kc = pts;
    *n = (int)((k_end + pts - 1) / pts);
}

__host__ __device__ inline int64_t slot_blocks(int64_t N) { return (N + kSL - 1) / kSL; }

// Block that the slot runs at server step e, or -1: not begun, or finished and waiting
// for host memory for its result.
__device__ inline int64_t slot_block(const SlotDev &s, int64_t e)
{
    const int64_t c = s.c0 + e;
    return e < s.start || c >= slot_blocks(s.N) ? -1 : c;
}

__device__ inline DevBatch slot_batch(const SlotDev &s)
{
    DevBatch bt{};
    bt.dim = s.dim;
    bt.B = 1;
    bt.cols = s.dim;
    bt.N = s.N;
    bt.N_each = s.Nb;
    bt.y0 = s.y0;
    bt.y1 = s.y1;
    bt.params = s.params;
    bt.F = s.F;
    bt.Ff = s.Ff;
    bt.ldF = s.dim;
    bt.Y = s.Y;
    bt.status = s.status;
    return bt;
}

// Runs fn.template operator()<Rhs, D>() for the slot's right-hand side.
template <class Fn>
__device__ inline void slot_dispatch(int rhs, int dim, Fn &&fn)
{
    switch (rhs) {
    case FABM_RHS_CONST:
        if (dim == 1) fn.template operator()<RhsConst, 1>();
        else if (dim == 2) fn.template operator()<RhsConst, 2>();
        else if (dim == 3) fn.template operator()<RhsConst, 3>();
        else fn.template operator()<RhsConst, 4>();
        break;
    case FABM_RHS_TIME:
        if (dim == 1) fn.template operator()<RhsTime, 1>();
        else if (dim == 2) fn.template operator()<RhsTime, 2>();
        else if (dim == 3) fn.template operator()<RhsTime, 3>();
        else fn.template operator()<RhsTime, 4>();
        break;
    case FABM_RHS_LINEAR:
        if (dim == 1) fn.template operator()<RhsLinear, 1>();
        else if (dim == 2) fn.template operator()<RhsLinear, 2>();
        else if (dim == 3) fn.template operator()<RhsLinear, 3>();
        else fn.template operator()<RhsLinear, 4>();
        break;
    case FABM_RHS_LORENZ: fn.template operator()<RhsLorenz, 3>(); break;
    case FABM_RHS_DUFFING: fn.template operator()<RhsDuffing, 2>(); break;
    case FABM_RHS_MANUFACTURED: fn.template operator()<RhsManufactured, 1>(); break;
    case FABM_RHS_LCR: fn.template operator()<RhsLcr, 2>(); break;
    default: break;
    }
}

// Weights (double, and fp32 copies for split slots) of new slots:
// blockIdx.y = new slot, stride over the distances.
__global__ void __launch_bounds__(kWeightThreads)
    weights_slots_kernel(const SlotDev *__restrict__ slots, const int *__restrict__ idx)
{
    const SlotDev &s = slots[idx[blockIdx.y]];
    const double inv_g2 = s.kc.inv_gamma2[0], alpha = s.alpha, inv_g1 = s.inv_g1;
    const int64_t w_ext = s.w_ext;
    double *WB = s.WB, *WA = s.WA, *WD = s.WD;
    float *WBf = s.WBf, *WAf = s.WAf;
    for (int64_t d0 = blockIdx.x * (int64_t)blockDim.x; d0 <= w_ext; d0 += (int64_t)gridDim.x * blockDim.x)
        weights_block(d0, w_ext, alpha, inv_g1, inv_g2, WB, WA, WD, [&](int64_t d) {
            if (WBf) {
                WBf[d] = (float)WB[d];
                WAf[d] = (float)WA[d];
            }
        });
}

// Inputs, and for slots that start from the beginning the initial values, of n
// new slots.
__global__ void init_slots_kernel(const SlotDev *__restrict__ slots, const int *__restrict__ idx,
                                  int n)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n) return;
    const SlotDev &s = slots[idx[j]];
    *s.Nb = s.N;
    for (int q = 0; q < FABM_MAX_DIM; ++q) {
        s.y0[q] = s.y0v[q];
        if (s.y1) s.y1[q] = s.y1v[q];
    }
    for (int q = 0; q < kMaxParams; ++q) s.params[q] = s.pv[q];
    if (s.resumed) return;
    *s.status = ~0ull;
    const DevBatch bt = slot_batch(s);
    slot_dispatch(s.rhs, s.dim, [&]<class R, int D>() { init_one<R, D>(bt, 0); });
}

// status[j] of n finished slots, for the host.
__global__ void collect_slots_kernel(const SlotDev *__restrict__ slots, const int *__restrict__ idx,
                                     int n, unsigned long long *__restrict__ status)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j < n) status[j] = *slots[idx[j]].status;
}

// Far history, one warp per (slot, chunk, column) item (FP64) or four: requests
// have one to three columns.  Each warp stages its own tiles of f and of the
// weights and runs the same per-column arithmetic as the batch kernels
// (hist_fp64_block / hist_fp32c_block), so a request's partial sums do not
// depend on which items share its CTA.
__device__ void hist_warp_f64(const SlotDev &s, int64_t c, int chunk, int64_t kc, int q,
                              double *sF, double *sB, double *sA)
{
    using hist::kL;
    constexpr int kT = hist::f64::kTile;
    const int a = threadIdx.x % kWarp, dim = s.dim;
    const int64_t k_end = (c - 1) * kSL;
    const int64_t k0 = (int64_t)chunk * kc;
    const int64_t k1 = k0 + kc < k_end ? k0 + kc : k_end;
    double sp = 0.0, sc = 0.0;
    for (int64_t t0 = k0; t0 < k1; t0 += kT) {
        const int64_t t1 = t0 + kT < k1 ? t0 + kT : k1;
        const int nk = (int)(t1 - t0);
        const int64_t d_min = c * kL + 2 - t1;
        for (int i = a; i < nk + kL - 1; i += kWarp) sB[i] = s.WB[d_min + i], sA[i] = s.WA[d_min + i];
        for (int i = a; i < nk; i += kWarp) sF[i] = s.F[(t0 + i) * dim + q];
        __syncwarp();
        const int base = a + nk - 1;
#pragma unroll 4
        for (int j = 0; j < nk; ++j) {
            const double f = sF[j];
            sp = fma(sB[base - j], f, sp);
            sc = fma(sA[base - j], f, sc);
        }
        __syncwarp();
    }
    double *out = static_cast<double *>(s.part) + ((int64_t)(chunk * 2) * kL + a) * dim + q;
    out[0] = sp;
    out[(int64_t)kL * dim] = sc;
}

__device__ void hist_warp_f32c(const SlotDev &s, int64_t c, int chunk, int64_t kc, int q,
                               float *sF, float *sB, float *sA)
{
    using hist::kL;
    constexpr int kT = hist::f32c::kTile, kG = hist::f32c::kGroup;
    constexpr int kRF = kT / kWarp, kRW = (kT + kL + kWarp - 1) / kWarp;
    const int a = threadIdx.x % kWarp, dim = s.dim;
    const int64_t k_end = (c - 1) * kSL;
    const int64_t k0 = (int64_t)chunk * kc;
    const int64_t k1 = k0 + kc < k_end ? k0 + kc : k_end;
    float sp = 0.f, cp = 0.f, sc = 0.f, cc = 0.f;
    // the next tile's f (the recurrence's float copy) and weights are loaded
    // into registers while the current tile is summed
    float rf[kRF], rb[kRW], ra[kRW];
    auto fetch = [&](int64_t t0) {
        const int64_t t1 = t0 + kT < k1 ? t0 + kT : k1;
        const int nk = (int)(t1 - t0);
        const int64_t d_min = c * kL + 2 - t1;
#pragma unroll
        for (int u = 0; u < kRW; ++u) {
            const int i = a + u * kWarp;
            rb[u] = i < nk + kL - 1 ? s.WBf[d_min + i] : 0.f;
            ra[u] = i < nk + kL - 1 ? s.WAf[d_min + i] : 0.f;
        }
#pragma unroll
        for (int u = 0; u < kRF; ++u) {
            const int i = a + u * kWarp;
            rf[u] = i < nk ? s.Ff[(t0 + i) * dim + q] : 0.f;
        }
    };
    if (k0 < k1) fetch(k0);
    for (int64_t t0 = k0; t0 < k1; t0 += kT) {
        const int64_t t1 = t0 + kT < k1 ? t0 + kT : k1;
        const int nk = (int)(t1 - t0);
#pragma unroll
        for (int u = 0; u < kRW; ++u) {
            const int i = a + u * kWarp;
            if (i < nk + kL - 1) sB[i] = rb[u], sA[i] = ra[u];
        }
#pragma unroll
        for (int u = 0; u < kRF; ++u) sF[a + u * kWarp] = rf[u];
        __syncwarp();
        if (t1 < k1) fetch(t1);
        const int base = a + nk - 1;
        int j = 0;
        for (; j + kG <= nk; j += kG) {
            float gp = 0.f, gc = 0.f;
#pragma unroll
            for (int u = 0; u < kG; ++u) {
                const float f = sF[j + u];
                gp = fmaf(sB[base - j - u], f, gp);
                gc = fmaf(sA[base - j - u], f, gc);
            }
            hist::f32c::kahan_add(sp, cp, gp);
            hist::f32c::kahan_add(sc, cc, gc);
        }
        float gp = 0.f, gc = 0.f;
        for (; j < nk; ++j) {
            const float f = sF[j];
            gp = fmaf(sB[base - j], f, gp);
            gc = fmaf(sA[base - j], f, gc);
        }
        hist::f32c::kahan_add(sp, cp, gp);
        hist::f32c::kahan_add(sc, cc, gc);
        __syncwarp();
    }
    float2 *out = static_cast<float2 *>(s.part) + ((int64_t)(chunk * 2) * kL + a) * dim + q;
    out[0] = make_float2(sp, -cp);
    out[(int64_t)kL * dim] = make_float2(sc, -cc);
}

// Four items of a slot by one warp in compensated fp32: eight lanes an item,
// four targets a lane.  As j advances a lane's window of weights moves by one, so
// a point costs it two weights and a quarter of a vector load of f for eight
// multiply-adds, where a lane per target took three loads for two (a step's
// shared-memory loads were what its history and the steps beside it waited for).
// Chosen from kQuadItems items a step on, where the loads count and not the
// latency of one item.  Steps with an item per warp / with four, us: 1024 slots of
// the Lorenz type, 39,000 items 439 / 290, 12,000 180 / 147, 6,000 128 / 125; 1024
// linear ones, 13,000 items 181 / 135, 4,000 86 / 94; 256 of the Lorenz type, 5,000
// items 87 / 92, 1,500 52 / 57; 64 slots, 400 items 29 / 33.
constexpr int kQuad = 4;
constexpr int64_t kQuadItems = 6144;
constexpr int kQT = 64;                      // points per tile
constexpr int kQF = kQT + 4, kQW = kQT + 33;  // strides of f and of the weights: banks apart
constexpr int kQuadFloats = 2 * kQuad * (kQF + 2 * kQW);

__device__ __forceinline__ void copy4(float *dst, const float *src, bool in)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(
                     (uint32_t)__cvta_generic_to_shared(dst)),
                 "l"(src), "r"(in ? 4 : 0)
                 : "memory");
}

__device__ void hist_quad_f32c(const SlotDev &s, int64_t c, int64_t kc, int n_chunks, int g0,
                               float *smem)
{
    using hist::kL;
    using hist::f32c::kahan_add;
    constexpr int kT = hist::f32c::kTile, kG = hist::f32c::kGroup;
    static_assert(kQT % kG == 0 && kT % kQT == 0);
    const int lane = threadIdx.x % kWarp, grp = lane / 8, l = lane % 8;
    const int dim = s.dim, g = g0 + grp;
    const bool valid = g < n_chunks * dim;
    const int chunk = valid ? g / dim : 0, q = valid ? g % dim : 0;
    const int64_t k_end = (c - 1) * kSL, k0 = (int64_t)chunk * kc;
    const int npts = valid ? (int)(k0 + kc < k_end ? kc : k_end - k0) : 0;
    const int most = (int)__reduce_max_sync(0xffffffffu, (unsigned)npts);
    float *sF = smem + grp * kQF, *sB = smem + kQuad * kQF + grp * kQW;
    float *sA = sB + kQuad * kQW;
    constexpr int kBuf = kQuadFloats / 2;
    // tile t: f of the points k0 + kQT t + j; window index i <-> distance
    // cL + 1 - (k0 + kQT t + kQT - 1) + i, of target a and point j: a + kQT - 1 - j
    auto fetch = [&](int t) {
        const int o = (t & 1) * kBuf;
        const int64_t t0 = k0 + (int64_t)t * kQT, d0 = c * kL + 2 - kQT - t0;
        const bool on = t * kQT < npts;
#pragma unroll
        for (int u = 0; u < kQT / 8; ++u) {
            const int i = l + 8 * u;
            const bool in = t * kQT + i < npts;
            copy4(sF + o + i, s.Ff + (in ? (t0 + i) * dim + q : 0), in);
        }
#pragma unroll
        for (int u = 0; u < (kQT + kL) / 8; ++u) {
            const int i = l + 8 * u;
            const bool in = on && d0 + i >= 0;
            copy4(sB + o + i, s.WBf + (in ? d0 + i : 0), in);
            copy4(sA + o + i, s.WAf + (in ? d0 + i : 0), in);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    float sp[4] = {}, cp[4] = {}, sc[4] = {}, cc[4] = {};
    fetch(0);
    for (int t = 0; t * kQT < most; ++t) {
        if ((t + 1) * kQT < most) {
            fetch(t + 1);
            asm volatile("cp.async.wait_group 1;" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
        }
        __syncwarp();
        const int o = (t & 1) * kBuf, nk = npts - t * kQT;
        if (nk > 0) {
            const float4 *fv = reinterpret_cast<const float4 *>(sF + o);
            const float *wb = sB + o + 4 * l + kQT - 1, *wa = sA + o + 4 * l + kQT - 1;
            float b[4], a[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) b[u] = wb[u], a[u] = wa[u];
#pragma unroll
            for (int j0 = 0; j0 < kQT; j0 += kG) {
                if (j0 < nk) {  // points past the chunk are zeros
                    float gp[4] = {}, gc[4] = {};
#pragma unroll
                    for (int u4 = 0; u4 < kG; u4 += 4) {
                        const float4 f4 = fv[(j0 + u4) / 4];
                        const float f[4] = {f4.x, f4.y, f4.z, f4.w};
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
#pragma unroll
                            for (int v = 0; v < 4; ++v) {
                                gp[v] = fmaf(b[v], f[u], gp[v]);
                                gc[v] = fmaf(a[v], f[u], gc[v]);
                            }
                            const int j = j0 + u4 + u + 1;  // the next point's weights
#pragma unroll
                            for (int v = 3; v > 0; --v) b[v] = b[v - 1], a[v] = a[v - 1];
                            if (j < kQT) b[0] = wb[-j], a[0] = wa[-j];
                        }
                    }
#pragma unroll
                    for (int v = 0; v < 4; ++v) kahan_add(sp[v], cp[v], gp[v]), kahan_add(sc[v], cc[v], gc[v]);
                }
            }
            // the fold after 512 points or the last one: of the rest that is not a
            // multiple of 16 (done above), or of nothing
            const bool end = nk <= kQT || (t + 1) % (kT / kQT) == 0;
            if (end && (nk >= kQT || nk % kG == 0)) {
#pragma unroll
                for (int v = 0; v < 4; ++v) kahan_add(sp[v], cp[v], 0.f), kahan_add(sc[v], cc[v], 0.f);
            }
        }
        __syncwarp();
    }
    if (valid) {
        float2 *out = static_cast<float2 *>(s.part) + ((int64_t)(chunk * 2) * kL + 4 * l) * dim + q;
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            out[(int64_t)v * dim] = make_float2(sp[v], -cp[v]);
            out[(int64_t)(kL + v) * dim] = make_float2(sc[v], -cc[v]);
        }
    }
}

constexpr int kHistBytesF64 = (hist::f64::kTile + 2 * (hist::f64::kTile + hist::kL)) * 8;
constexpr int kHistBytesF32 =
    std::max(kQuadFloats, hist::f32c::kTile + 2 * (hist::f32c::kTile + hist::kL)) * 4;
constexpr int kHistWarpBytes = kHistBytesF64 > kHistBytesF32 ? kHistBytesF64 : kHistBytesF32;
constexpr int kStepWarps = FABM_MAX_DIM + 1;  // the components and the forcing; history items
// In double four, one per SM sub-partition: a fifth warp of every CTA would load the
// FP64 unit of the same one (Lorenz type, 64 requests of 8000 steps 53.0 ms with five,
// 49.0 with four; 128 of 3000 steps 22.5, 20.2).
constexpr int kStepWarpsF64 = FABM_MAX_DIM;

// A slot's history items for its block cn.
__host__ __device__ inline int slot_items(int64_t cn, int dim)
{
    int64_t kc;
    int n;
    slot_chunks(cn, &kc, &n);
    return n * dim;
}

// The fixed-order sum of a slot's chunks: G[kind][t][col] over the chunks in
// ascending order (compensated double, or float-float rounded once to double).
__device__ void combine_slot(const SlotDev &s, int64_t cn, int n_chunks)
{
    const int n_out = 2 * kSL * s.dim;
    double *G = s.G + (int64_t)(cn % 2) * n_out;
    for (int o = threadIdx.x; o < n_out; o += blockDim.x) {
        if (s.hk == FABM_HIST_FP32C) {
            const float2 *p = static_cast<const float2 *>(s.part);
            float hi = 0.f, lo = 0.f;
            float2 v[kMaxChunksSlot];
#pragma unroll
            for (int ch = 0; ch < kMaxChunksSlot; ++ch)
                if (ch < n_chunks) v[ch] = __ldcg(p + (int64_t)ch * n_out + o);
#pragma unroll
            for (int ch = 0; ch < kMaxChunksSlot; ++ch)
                if (ch < n_chunks) ff_add_chunk(hi, lo, v[ch].x, v[ch].y);
            G[o] = (double)hi + (double)lo;
        } else {
            // Neumaier: the rounding error of every addition (TwoSum) is kept
            // in a second sum, added once at the end; chunk order fixed
            const double *p = static_cast<const double *>(s.part);
            double acc = 0.0, err = 0.0;
            for (int ch = 0; ch < n_chunks; ++ch) {
                const double v = __ldcg(p + (int64_t)ch * n_out + o);
                const double t = acc + v;
                const double bv = t - acc;
                err += (acc - (t - bv)) + (v - bv);
                acc = t;
            }
            G[o] = acc + err;
        }
    }
}

// One server step.  CTA x < ns: the step's block of slot x.  The other CTAs, hx
// per slot: the far history of the slot's next block, its (chunk, column) items
// in chunk-major order, `per` (1 or kQuad) to a warp, derived from the slot's block index, so the host
// uploads no work list; the CTA that finishes a slot's last items (a count per
// slot, left at zero) adds its chunks.  No CTA waits for another one.
__global__ void __launch_bounds__(kWarp *kStepWarps)
    step_slots_kernel(const SlotDev *__restrict__ slots, int64_t epoch, int ns, int hx, int per,
                      int *cnt)
{
    static_assert(recur_smem_doubles<FABM_MAX_DIM, 1>() * 8 <= kStepWarps * kHistWarpBytes &&
                  recur_split_smem_floats<FABM_MAX_DIM>() * 4 <= kStepWarps * kHistWarpBytes);
    __shared__ __align__(16) unsigned char smem[kStepWarps][kHistWarpBytes];
    __shared__ bool last;
    if ((int)blockIdx.x < ns) {
        const SlotDev &s = slots[blockIdx.x];
        const int64_t c = slot_block(s, epoch);  // -1: none (new slot)
        if (c < 0) return;
        const DevBatch bt = slot_batch(s);
        const DevWeights w{s.WB, s.WA, s.WD, s.w_ext};
        const double *G = c >= 2 ? s.G + (c % 2) * 2 * kSL * s.dim : nullptr;
        const bool split = s.hk == FABM_HIST_FP32C;
        slot_dispatch(s.rhs, s.dim, [&]<class R, int D>() {
            if (split)
                recur_block_split<R, D>(bt, 0, w, s.kc, c, G, reinterpret_cast<float *>(smem));
            else
                recur_block<R, D, 1>(bt, 0, w, s.kc, c, G, reinterpret_cast<double *>(smem));
        });
        return;
    }
    const int slot = ((int)blockIdx.x - ns) / hx, x = ((int)blockIdx.x - ns) % hx;
    const SlotDev s = slots[slot];
    const int64_t cn = slot_block(s, epoch) + 1;
    if (cn < 2 || cn >= slot_blocks(s.N)) return;
    int64_t kc;
    int n;
    slot_chunks(cn, &kc, &n);
    const int hw = blockDim.x / kWarp;
    const int items = n * s.dim, ctas = (items + hw * per - 1) / (hw * per);
    if (x >= ctas) return;
    const int w = threadIdx.x / kWarp, g = (x * hw + w) * per;
    if (g >= items) {
    } else if (per == kQuad) {
        hist_quad_f32c(s, cn, kc, n, g, reinterpret_cast<float *>(smem[w]));
    } else if (s.hk == FABM_HIST_FP32C) {
        float *sF = reinterpret_cast<float *>(smem[w]);
        float *sB = sF + hist::f32c::kTile;
        hist_warp_f32c(s, cn, g / s.dim, kc, g % s.dim, sF, sB, sB + hist::f32c::kTile + hist::kL);
    } else {
        double *sF = reinterpret_cast<double *>(smem[w]);
        double *sB = sF + hist::f64::kTile;
        hist_warp_f64(s, cn, g / s.dim, kc, g % s.dim, sF, sB, sB + hist::f64::kTile + hist::kL);
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        last = atomicAdd(cnt + slot, 1) == ctas - 1;
        if (last) cnt[slot] = 0;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    combine_slot(s, cn, n);
}

// ------------------------------------------------------------------- host ---

fabm_status srv_fail(fabm_status st, const char *fmt, ...)
{
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    set_last_error(buf);
    return st;
}

#define SRV_TRY(expr)                                                                        \
    do {                                                                                     \
        cudaError_t e_ = (expr);                                                             \
        if (e_ != cudaSuccess)                                                               \
            return srv_fail(e_ == cudaErrorMemoryAllocation ? FABM_ENOMEM : FABM_ECUDA,      \
                            "%s failed: %s", #expr, cudaGetErrorString(e_));                 \
    } while (0)

// State of a request taken at a block boundary (fabm_server_checkpoint): the
// next block to run, the history f and the solution rows known so far, both
// far-history buffers and the non-finite status word.
struct Ckpt {
    int64_t c = 0;
    unsigned long long status = ~0ull;
    std::vector<double> F, Y, G;  // rows x dim, rows x dim, 2 x 2 x kSL x dim
};

// Layout of a serialized checkpoint: this header, then F and Y (rows x dim
// each) and G (2 x 2 x kSL x dim), doubles in the host's byte order.
constexpr char kCkptMagic[8] = {'F', 'A', 'B', 'M', 'C', 'K', 'P', '2'};
struct CkptHead {
    char magic[8];
    int32_t precision, dim, rhs, n_params;
    double alpha, h;
    int64_t N, c, rows;
    unsigned long long status;
    double params[kMaxParams];
    double y0[FABM_MAX_DIM];
    int32_t has_y1, pad;
    double y1[FABM_MAX_DIM];  // y'(0) when has_y1 (1 < alpha < 2)
};

struct Req {
    int64_t ticket;
    int dim, rhs;
    double alpha, h;
    int64_t N;
    double params[kMaxParams];
    int n_params;
    double y0[FABM_MAX_DIM];
    double y1[FABM_MAX_DIM];  // y'(0), used when has_y1 (1 < alpha < 2)
    int has_y1;
    std::shared_ptr<const Ckpt> ckpt;  // set for a resumed request
};

struct Slot {
    Req req;
    int64_t c = 0, nblk = 0;
    size_t bytes = 0;
    void *mem = nullptr;
    SlotDev dev{};
    bool pending = false;  // admitted at this step: weights being computed, no block run yet
};

struct Result {
    int state;  // FABM_REQ_*
    fabm_status status;
    std::unique_ptr<double[]> y;  // n values once it has finished
    size_t n = 0;
};

size_t slot_bytes(const Req &r, int hk, int64_t *w_ext_out)
{
    const int64_t nblk = (r.N + kSL - 1) / kSL;
    const int64_t w_ext = nblk * kSL + 2 * kSL;
    *w_ext_out = w_ext;
    const int64_t n_chunks = kMaxChunksSlot;
    size_t b = 0;
    auto add = [&](size_t n) { b += (n + 255) / 256 * 256; };
    add(sizeof(int64_t));                                   // Nb
    add(sizeof(unsigned long long));                        // status
    add(sizeof(double) * FABM_MAX_DIM);                     // y0
    add(sizeof(double) * FABM_MAX_DIM);                     // y1
    add(sizeof(double) * kMaxParams);                       // params
    for (int i = 0; i < 3; ++i) add(sizeof(double) * (w_ext + 1));  // WB WA WD
    if (hk == FABM_HIST_FP32C) {
        for (int i = 0; i < 2; ++i) add(sizeof(float) * (w_ext + 1));
        add(sizeof(float) * (r.N + 1) * r.dim);             // Ff
    }
    add(sizeof(double) * (r.N + 1) * r.dim);                // F
    add(sizeof(double) * (r.N + 1) * r.dim);                // Y
    add(sizeof(double) * 2 * 2 * kSL * r.dim);              // G
    add((size_t)8 * n_chunks * 2 * kSL * r.dim);            // partials
    return b;
}

// Carves a slot's device block into its buffers.
void slot_layout(Slot &s, int hk, int64_t w_ext)
{
    uint8_t *p = static_cast<uint8_t *>(s.mem);
    auto take = [&](size_t n) {
        uint8_t *q = p;
        p += (n + 255) / 256 * 256;
        return q;
    };
    const Req &r = s.req;
    SlotDev &d = s.dev;
    d.rhs = r.rhs, d.dim = r.dim, d.hk = hk, d.N = r.N, d.w_ext = w_ext;
    d.Nb = reinterpret_cast<int64_t *>(take(sizeof(int64_t)));
    d.status = reinterpret_cast<unsigned long long *>(take(sizeof(unsigned long long)));
    d.y0 = reinterpret_cast<double *>(take(sizeof(double) * FABM_MAX_DIM));
    double *y1 = reinterpret_cast<double *>(take(sizeof(double) * FABM_MAX_DIM));
    d.y1 = r.has_y1 ? y1 : nullptr;
    d.params = reinterpret_cast<double *>(take(sizeof(double) * kMaxParams));
    d.WB = reinterpret_cast<double *>(take(sizeof(double) * (w_ext + 1)));
    d.WA = reinterpret_cast<double *>(take(sizeof(double) * (w_ext + 1)));
    d.WD = reinterpret_cast<double *>(take(sizeof(double) * (w_ext + 1)));
    d.WBf = d.WAf = d.Ff = nullptr;
    if (hk == FABM_HIST_FP32C) {
        d.WBf = reinterpret_cast<float *>(take(sizeof(float) * (w_ext + 1)));
        d.WAf = reinterpret_cast<float *>(take(sizeof(float) * (w_ext + 1)));
        d.Ff = reinterpret_cast<float *>(take(sizeof(float) * (r.N + 1) * r.dim));
    }
    d.F = reinterpret_cast<double *>(take(sizeof(double) * (r.N + 1) * r.dim));
    d.Y = reinterpret_cast<double *>(take(sizeof(double) * (r.N + 1) * r.dim));
    d.G = reinterpret_cast<double *>(take(sizeof(double) * 2 * 2 * kSL * r.dim));
    d.part = take((size_t)8 * kMaxChunksSlot * 2 * kSL * r.dim);
    d.kc.h = r.h;
    for (int q = 0; q < FABM_MAX_DIM; ++q) {
        d.kc.h_alpha[q] = std::pow(r.h, r.alpha);
        d.kc.inv_gamma2[q] = 1.0 / std::tgamma(r.alpha + 2.0);
    }
    for (int q = 0; q < FABM_MAX_DIM; ++q) d.y0v[q] = r.y0[q], d.y1v[q] = r.y1[q];
    for (int q = 0; q < kMaxParams; ++q) d.pv[q] = q < r.n_params ? r.params[q] : 0.0;
    d.resumed = r.ckpt ? 1 : 0;
    d.alpha = r.alpha;
    d.inv_g1 = 1.0 / std::tgamma(r.alpha + 1.0);
}


}  // namespace

struct fabm_server {
    int device = 0;
    int precision = FABM_FP64;
    size_t budget = 0, in_use = 0;
    int max_slots = 0;
    std::deque<Req> queue;
    std::vector<Slot> slots;
    std::unordered_map<int64_t, Result> results;
    std::unordered_map<int64_t, std::pair<int64_t, int>> shapes;  // ticket -> (N, dim)
    std::vector<int64_t> finished;  // finished since the last fabm_server_finished
    int64_t next_ticket = 1;
    cudaStream_t sR = nullptr, sW = nullptr;
    cudaEvent_t evIn = nullptr, evW = nullptr;
    int64_t epoch = 0;           // server steps with slots, the time base of their block indices
    SlotDev *d_slots = nullptr;  // device tables: the slots, uploaded when they change,
    int *d_idx = nullptr;        // and the indices of newly admitted or finished slots
    SlotDev *h_slots = nullptr;  // pinned staging
    int *h_idx = nullptr;
    int *d_cnt = nullptr;        // history CTAs done per slot, zero between steps
    unsigned long long *h_status = nullptr;  // pinned, written by the device
    bool table_dirty = true;     // the slot table changed since its last upload
    int64_t steps_done = 0, launches = 0;
    std::mutex mu;

    ~fabm_server()
    {
        for (auto &s : slots)
            if (s.mem) cudaFreeAsync(s.mem, sR);
        if (sR) cudaStreamSynchronize(sR);
        if (d_slots) cudaFree(d_slots);
        if (d_idx) cudaFree(d_idx);
        if (d_cnt) cudaFree(d_cnt);
        if (h_slots) cudaFreeHost(h_slots);
        if (h_status) cudaFreeHost(h_status);
        if (h_idx) cudaFreeHost(h_idx);
        if (sW) cudaStreamSynchronize(sW);
        if (evIn) cudaEventDestroy(evIn);
        if (evW) cudaEventDestroy(evW);
        if (sR) cudaStreamDestroy(sR);
        if (sW) cudaStreamDestroy(sW);
    }
};

namespace {

fabm_status server_step(fabm_server *S, int *n_active, int *n_waiting)
{
    const int hk = S->precision == FABM_SPLIT ? FABM_HIST_FP32C : FABM_HIST_FP64;
    // 1. admission: waiting requests in arrival order while the budget allows
    std::vector<int> fresh;
    while (!S->queue.empty() && (int)S->slots.size() < S->max_slots) {
        Req r = S->queue.front();
        int64_t w_ext;
        const size_t bytes = slot_bytes(r, hk, &w_ext);
        if (S->in_use + bytes > S->budget) {
            if (S->slots.empty()) {  // can never fit
                S->queue.pop_front();
                S->results[r.ticket] = {FABM_REQ_FAILED, FABM_ENOMEM, nullptr};
                S->finished.push_back(r.ticket);
                continue;
            }
            break;
        }
        Slot s;
        s.req = r;
        s.bytes = bytes;
        s.nblk = (r.N + kSL - 1) / kSL;
        cudaError_t e = take_injected_alloc_failure() ? cudaErrorMemoryAllocation
                                                      : cudaMallocAsync(&s.mem, bytes, S->sR);
        if (e != cudaSuccess) {
            if (S->slots.empty()) {
                S->queue.pop_front();
                S->results[r.ticket] = {FABM_REQ_FAILED, FABM_ENOMEM, nullptr};
                S->finished.push_back(r.ticket);
                continue;
            }
            break;  // retry when memory frees up
        }
        slot_layout(s, hk, w_ext);
        if (r.ckpt) s.c = r.ckpt->c;
        S->queue.pop_front();
        S->in_use += bytes;
        S->results[r.ticket] = {FABM_REQ_RUNNING, FABM_OK, nullptr};
        s.pending = true;
        fresh.push_back((int)S->slots.size());
        S->slots.push_back(s);
    }
    const int ns = (int)S->slots.size();
    *n_waiting = (int)S->queue.size();
    *n_active = ns;
    if (ns == 0) return FABM_OK;

    // 2. table: the slots, when they changed (a slot's block index follows from
    // the step number, its history, combine and recurrence items from the block
    // index, so a step without arrivals or departures uploads nothing), and the
    // indices of new slots
    const int64_t epoch = S->epoch;
    if (!fresh.empty()) S->table_dirty = true;
    if (S->table_dirty) {
        for (int i = 0; i < ns; ++i) {
            Slot &s = S->slots[i];
            if (s.pending) {  // first block at the next step
                s.dev.start = epoch + 1;
                s.dev.c0 = s.c - (epoch + 1);
            }
            S->h_slots[i] = s.dev;
        }
        SRV_TRY(cudaMemcpyAsync(S->d_slots, S->h_slots, sizeof(SlotDev) * ns, cudaMemcpyHostToDevice, S->sR));
        S->table_dirty = false;
    }
    int64_t items = 0;   // history items of the step,
    int most_items = 0;  // of the busiest slot
    for (int i = 0; i < ns; ++i) {
        const Slot &s = S->slots[i];
        const int64_t cn = s.c + 1;
        if (s.pending || cn < 2 || cn >= s.nblk) continue;
        const int n = slot_items(cn, s.req.dim);
        items += n;
        most_items = std::max(most_items, n);
    }
    const int per = hk == FABM_HIST_FP32C && items >= kQuadItems ? kQuad : 1;  // items per warp
    const int hw = hk == FABM_HIST_FP32C ? kStepWarps : kStepWarpsF64;  // warps per CTA
    const int hx = (most_items + hw * per - 1) / (hw * per);
    // 3. new slots: weights and initial values on stream W beside this step's
    // launches (they take ~0.1-0.2 ms of FP64 work, which had delayed the whole
    // step whenever requests arrived); the new slots run their first block at
    // the next step.  Their inputs travel in the table.
    if (!fresh.empty()) {
        for (size_t j = 0; j < fresh.size(); ++j) S->h_idx[j] = fresh[j];
        SRV_TRY(cudaMemcpyAsync(S->d_idx, S->h_idx, sizeof(int) * fresh.size(), cudaMemcpyHostToDevice, S->sR));
        for (int i : fresh) {
            Slot &s = S->slots[i];
            const Ckpt *k = s.req.ckpt.get();
            if (!k) continue;  // resumed: the saved state
            const size_t rows = k->F.size() / s.req.dim;
            SRV_TRY(cudaMemcpyAsync(s.dev.F, k->F.data(), sizeof(double) * rows * s.req.dim, cudaMemcpyHostToDevice, S->sR));
            if (s.dev.Ff)  // the float copy the fp32 history reads
                SRV_TRY(launch_to_float(s.dev.F, (int64_t)(rows * s.req.dim), s.dev.Ff, S->sR));
            SRV_TRY(cudaMemcpyAsync(s.dev.Y, k->Y.data(), sizeof(double) * rows * s.req.dim, cudaMemcpyHostToDevice, S->sR));
            SRV_TRY(cudaMemcpyAsync(s.dev.G, k->G.data(), sizeof(double) * k->G.size(), cudaMemcpyHostToDevice, S->sR));
            SRV_TRY(cudaMemcpyAsync(s.dev.status, &k->status, sizeof k->status, cudaMemcpyHostToDevice, S->sR));
        }
        SRV_TRY(cudaEventRecord(S->evIn, S->sR));
        SRV_TRY(cudaStreamWaitEvent(S->sW, S->evIn, 0));
        int64_t wmax = 0;
        for (int i : fresh) wmax = std::max(wmax, S->slots[i].dev.w_ext);
        const unsigned gx = (unsigned)std::min<int64_t>((wmax + kWeightThreads) / kWeightThreads, 64);
        weights_slots_kernel<<<dim3(gx, (unsigned)fresh.size()), kWeightThreads, 0, S->sW>>>(S->d_slots, S->d_idx);
        SRV_TRY(cudaGetLastError());
        init_slots_kernel<<<(unsigned)((fresh.size() + 127) / 128), 128, 0, S->sW>>>(
            S->d_slots, S->d_idx, (int)fresh.size());
        SRV_TRY(cudaGetLastError());
        SRV_TRY(cudaEventRecord(S->evW, S->sW));
        S->launches += 2;
    }
    // 4. one launch for all slots
    step_slots_kernel<<<(unsigned)(ns + ns * hx), kWarp * hw, 0, S->sR>>>(
        S->d_slots, epoch, ns, std::max(hx, 1), per, S->d_cnt);
    SRV_TRY(cudaGetLastError());
    ++S->launches;
    if (!fresh.empty()) SRV_TRY(cudaStreamWaitEvent(S->sR, S->evW, 0));
    SRV_TRY(cudaStreamSynchronize(S->sR));
    ++S->steps_done;
    ++S->epoch;

    // 5. advance; finished slots to host, memory back to the pool; the table
    // is compacted (and uploaded at the next step) only when a slot finished
    int n_done = 0;
    for (int i = 0; i < ns; ++i) {
        Slot &s = S->slots[i];
        s.req.ckpt.reset();  // restored on the device by now
        if (s.pending) {  // weights and initial values are in place: run from the next step
            s.pending = false;
            continue;
        }
        s.c = std::min(s.c + 1, s.nblk);  // at nblk already if a result had no room before
        if (s.c >= s.nblk) S->h_idx[n_done++] = i;
    }
    // room for every result before anything is copied; without it the finished slots
    // wait for the next step
    for (int j = 0; j < n_done; ++j) {
        const Slot &s = S->slots[S->h_idx[j]];
        Result &res = S->results[s.req.ticket];
        res.n = (size_t)(s.req.N + 1) * s.req.dim;
        if (!take_injected_alloc_failure())
            res.y.reset(new (std::nothrow) double[res.n]());  // touched here: the copy engine
                                                              // is slow on new pages
        if (!res.y) return srv_fail(FABM_ENOMEM, "host memory for a result");
    }
    if (n_done > 0) {
        SRV_TRY(cudaMemcpyAsync(S->d_idx, S->h_idx, sizeof(int) * n_done, cudaMemcpyHostToDevice, S->sR));
        collect_slots_kernel<<<(unsigned)((n_done + 127) / 128), 128, 0, S->sR>>>(
            S->d_slots, S->d_idx, n_done, S->h_status);
        SRV_TRY(cudaGetLastError());
        ++S->launches;
        for (int j = 0; j < n_done; ++j) {
            Slot &s = S->slots[S->h_idx[j]];
            Result &res = S->results[s.req.ticket];
            SRV_TRY(cudaMemcpyAsync(res.y.get(), s.dev.Y, sizeof(double) * res.n, cudaMemcpyDeviceToHost, S->sR));
        }
        SRV_TRY(cudaStreamSynchronize(S->sR));
        for (int j = 0; j < n_done; ++j) {
            Slot &s = S->slots[S->h_idx[j]];
            Result &res = S->results[s.req.ticket];
            const bool ok = S->h_status[j] == ~0ull;
            res.state = ok ? FABM_REQ_DONE : FABM_REQ_FAILED;
            res.status = ok ? FABM_OK : FABM_ENONFINITE;
            S->finished.push_back(s.req.ticket);
            SRV_TRY(cudaFreeAsync(s.mem, S->sR));
            S->in_use -= s.bytes;
        }
        S->slots.erase(std::remove_if(S->slots.begin(), S->slots.end(),
                                      [](const Slot &s) { return s.c >= s.nblk; }),
                       S->slots.end());
        S->table_dirty = true;
    }
    *n_active = (int)S->slots.size();
    return FABM_OK;
}

}  // namespace

extern "C" {

fabm_status fabm_server_create(size_t budget_bytes, int precision, int max_slots, fabm_server **out)
{
    set_last_error("");
    if (!out) return srv_fail(FABM_EINVAL, "out is NULL");
    *out = nullptr;
    if (precision != FABM_FP64 && precision != FABM_SPLIT)
        return srv_fail(FABM_EINVAL, "precision %d unknown", precision);
    if (max_slots < 1 || max_slots > (1 << 20)) return srv_fail(FABM_EINVAL, "max_slots %d", max_slots);
    if (budget_bytes == 0) return srv_fail(FABM_EINVAL, "budget is 0");
    fabm_server *S = new (std::nothrow) fabm_server();
    if (!S) return srv_fail(FABM_ENOMEM, "host allocation failed");
    S->budget = budget_bytes, S->precision = precision, S->max_slots = max_slots;
    cudaError_t e = cudaGetDevice(&S->device);
    if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&S->sR, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&S->sW, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&S->evIn, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaMalloc(&S->d_slots, sizeof(SlotDev) * max_slots);
    if (e == cudaSuccess) e = cudaMalloc(&S->d_idx, sizeof(int) * max_slots);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&S->evW, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaMalloc(&S->d_cnt, sizeof(int) * max_slots);
    if (e == cudaSuccess) e = cudaMemset(S->d_cnt, 0, sizeof(int) * max_slots);
    if (e == cudaSuccess) e = cudaMallocHost(&S->h_status, sizeof(unsigned long long) * max_slots);
    if (e == cudaSuccess) e = cudaMallocHost(&S->h_slots, sizeof(SlotDev) * max_slots);
    if (e == cudaSuccess) e = cudaMallocHost(&S->h_idx, sizeof(int) * max_slots);
    if (e != cudaSuccess) {
        delete S;
        return srv_fail(FABM_ECUDA, "fabm_server_create: %s", cudaGetErrorString(e));
    }
    *out = S;
    return FABM_OK;
}

static fabm_status server_submit(fabm_server *S, const fabm_request *q, const double *y1,
                                 int64_t *ticket)
{
    set_last_error("");
    if (!S || !q || !ticket) return srv_fail(FABM_EINVAL, "NULL argument");
    if (q->dim < 1 || q->dim > FABM_MAX_DIM) return srv_fail(FABM_EINVAL, "dim %d", q->dim);
    if (!(q->alpha > 0.0 && q->alpha < 2.0)) return srv_fail(FABM_EINVAL, "alpha %g", q->alpha);
    if (y1 && !(q->alpha > 1.0))
        return srv_fail(FABM_EINVAL, "y'(0) given for alpha %g <= 1", q->alpha);
    if (!(q->h > 0.0) || !std::isfinite(q->h)) return srv_fail(FABM_EINVAL, "h %g", q->h);
    if (q->N < 1 || q->N > (1LL << 31)) return srv_fail(FABM_EINVAL, "N %lld", (long long)q->N);
    const int np = rhs_n_params(q->rhs_id);
    if (np < 0 || !rhs_supports_dim(q->rhs_id, q->dim))
        return srv_fail(FABM_EINVAL, "rhs_id %d with dim %d unsupported", q->rhs_id, q->dim);
    if (q->n_params < np || q->n_params > kMaxParams || (q->n_params > 0 && !q->params))
        return srv_fail(FABM_EINVAL, "rhs_id %d needs %d params", q->rhs_id, np);
    if (!q->y0) return srv_fail(FABM_EINVAL, "y0 is NULL");
    Req r{};
    r.dim = q->dim, r.rhs = q->rhs_id, r.alpha = q->alpha, r.h = q->h, r.N = q->N;
    r.n_params = q->n_params;
    for (int i = 0; i < q->n_params; ++i) r.params[i] = q->params[i];
    for (int i = 0; i < q->dim; ++i) {
        if (!std::isfinite(q->y0[i])) return srv_fail(FABM_EINVAL, "y0 not finite");
        r.y0[i] = q->y0[i];
    }
    if (y1) {
        r.has_y1 = 1;
        for (int i = 0; i < q->dim; ++i) {
            if (!std::isfinite(y1[i])) return srv_fail(FABM_EINVAL, "y'(0) not finite");
            r.y1[i] = y1[i];
        }
    }
    std::lock_guard<std::mutex> lk(S->mu);
    r.ticket = S->next_ticket++;
    S->queue.push_back(r);
    S->results[r.ticket] = {FABM_REQ_WAITING, FABM_OK, nullptr};
    S->shapes[r.ticket] = {r.N, r.dim};
    *ticket = r.ticket;
    return FABM_OK;
}

fabm_status fabm_server_submit(fabm_server *S, const fabm_request *q, int64_t *ticket)
{
    return server_submit(S, q, nullptr, ticket);
}

fabm_status fabm_server_submit_ic(fabm_server *S, const fabm_request *q, const double *y1,
                                  int64_t *ticket)
{
    return server_submit(S, q, y1, ticket);
}

fabm_status fabm_server_step(fabm_server *S, int *n_active, int *n_waiting)
{
    set_last_error("");
    TraceRange tr("fabm_server_step");
    if (!S) return srv_fail(FABM_EINVAL, "server is NULL");
    int a = 0, w = 0;
    std::lock_guard<std::mutex> lk(S->mu);
    int prev = -1;
    if (cudaGetDevice(&prev) == cudaSuccess && prev != S->device) cudaSetDevice(S->device);
    fabm_status st = server_step(S, &a, &w);
    if (prev >= 0 && prev != S->device) cudaSetDevice(prev);
    if (n_active) *n_active = a;
    if (n_waiting) *n_waiting = w;
    return st;
}

fabm_status fabm_server_poll(fabm_server *S, int64_t ticket, int *state)
{
    set_last_error("");
    if (!S || !state) return srv_fail(FABM_EINVAL, "NULL argument");
    std::lock_guard<std::mutex> lk(S->mu);
    auto it = S->results.find(ticket);
    if (it == S->results.end()) return srv_fail(FABM_EINVAL, "unknown ticket %lld", (long long)ticket);
    *state = it->second.state;
    return FABM_OK;
}

fabm_status fabm_server_result(fabm_server *S, int64_t ticket, double *out)
{
    set_last_error("");
    if (!S || !out) return srv_fail(FABM_EINVAL, "NULL argument");
    std::lock_guard<std::mutex> lk(S->mu);
    auto it = S->results.find(ticket);
    if (it == S->results.end()) return srv_fail(FABM_EINVAL, "unknown ticket %lld", (long long)ticket);
    Result &r = it->second;
    if (r.state == FABM_REQ_WAITING || r.state == FABM_REQ_RUNNING)
        return srv_fail(FABM_EBUSY, "request %lld not finished", (long long)ticket);
    const fabm_status st = r.status;
    if (r.y) std::memcpy(out, r.y.get(), sizeof(double) * r.n);
    S->results.erase(it);
    S->shapes.erase(ticket);
    if (st != FABM_OK)
        return srv_fail(st, "request %lld failed (%s)", (long long)ticket,
                        st == FABM_ENONFINITE ? "non-finite value" : "does not fit the budget");
    return FABM_OK;
}

fabm_status fabm_server_wait(fabm_server *S, int64_t ticket, double *out)
{
    set_last_error("");
    if (!S || !out) return srv_fail(FABM_EINVAL, "NULL argument");
    for (;;) {
        int state = 0;
        const fabm_status st = fabm_server_poll(S, ticket, &state);
        if (st != FABM_OK) return st;
        if (state == FABM_REQ_DONE || state == FABM_REQ_FAILED) break;
        const fabm_status ss = fabm_server_step(S, nullptr, nullptr);
        if (ss != FABM_OK) return ss;
    }
    return fabm_server_result(S, ticket, out);
}

fabm_status fabm_server_checkpoint(fabm_server *S, int64_t ticket, void *buf, size_t cap,
                                   size_t *size)
{
    set_last_error("");
    if (!S || !size) return srv_fail(FABM_EINVAL, "NULL argument");
    std::lock_guard<std::mutex> lk(S->mu);
    const Req *r = nullptr;
    const Slot *slot = nullptr;
    for (const Slot &sl : S->slots)
        if (sl.req.ticket == ticket) slot = &sl, r = &sl.req;
    if (!r)
        for (const Req &q : S->queue)
            if (q.ticket == ticket) r = &q;
    if (!r) return srv_fail(FABM_EINVAL, "request %lld is not waiting or running", (long long)ticket);
    const int64_t c = slot ? slot->c : (r->ckpt ? r->ckpt->c : 0);
    const int64_t rows = c == 0 ? 0 : std::min<int64_t>(r->N, c * kSL) + 1;
    const size_t n_g = (size_t)4 * kSL * r->dim;
    const size_t need = sizeof(CkptHead) + sizeof(double) * ((size_t)2 * rows * r->dim + n_g);
    *size = need;
    if (!buf) return FABM_OK;
    if (cap < need) return srv_fail(FABM_EINVAL, "checkpoint needs %zu bytes, buffer has %zu", need, cap);
    CkptHead hd{};
    std::memcpy(hd.magic, kCkptMagic, 8);
    hd.precision = S->precision, hd.dim = r->dim, hd.rhs = r->rhs, hd.n_params = r->n_params;
    hd.alpha = r->alpha, hd.h = r->h, hd.N = r->N, hd.c = c, hd.rows = rows;
    hd.status = ~0ull;
    for (int i = 0; i < kMaxParams; ++i) hd.params[i] = r->params[i];
    for (int i = 0; i < FABM_MAX_DIM; ++i) hd.y0[i] = r->y0[i], hd.y1[i] = r->y1[i];
    hd.has_y1 = r->has_y1;
    uint8_t *p = static_cast<uint8_t *>(buf);
    double *F = reinterpret_cast<double *>(p + sizeof hd);
    double *Y = F + rows * r->dim;
    double *G = Y + rows * r->dim;
    if (slot) {  // between steps both streams are idle: plain copies
        const size_t n = sizeof(double) * rows * r->dim;
        SRV_TRY(cudaMemcpy(F, slot->dev.F, n, cudaMemcpyDeviceToHost));
        SRV_TRY(cudaMemcpy(Y, slot->dev.Y, n, cudaMemcpyDeviceToHost));
        SRV_TRY(cudaMemcpy(G, slot->dev.G, sizeof(double) * n_g, cudaMemcpyDeviceToHost));
        SRV_TRY(cudaMemcpy(&hd.status, slot->dev.status, sizeof hd.status, cudaMemcpyDeviceToHost));
    } else if (r->ckpt) {
        std::memcpy(F, r->ckpt->F.data(), sizeof(double) * r->ckpt->F.size());
        std::memcpy(Y, r->ckpt->Y.data(), sizeof(double) * r->ckpt->Y.size());
        std::memcpy(G, r->ckpt->G.data(), sizeof(double) * n_g);
        hd.status = r->ckpt->status;
    } else {
        std::memset(G, 0, sizeof(double) * n_g);
    }
    std::memcpy(p, &hd, sizeof hd);
    return FABM_OK;
}

fabm_status fabm_server_resume(fabm_server *S, const void *buf, size_t size, int64_t *ticket)
{
    set_last_error("");
    if (!S || !buf || !ticket) return srv_fail(FABM_EINVAL, "NULL argument");
    if (size < sizeof(CkptHead)) return srv_fail(FABM_EINVAL, "checkpoint of %zu bytes is truncated", size);
    CkptHead hd;
    std::memcpy(&hd, buf, sizeof hd);
    if (std::memcmp(hd.magic, kCkptMagic, 8) != 0) return srv_fail(FABM_EINVAL, "not a checkpoint");
    if (hd.precision != S->precision)
        return srv_fail(FABM_EINVAL, "checkpoint of precision %d on a server of precision %d",
                        hd.precision, S->precision);
    if (hd.dim < 1 || hd.dim > FABM_MAX_DIM || !rhs_supports_dim(hd.rhs, hd.dim) ||
        hd.n_params < rhs_n_params(hd.rhs) || hd.n_params > kMaxParams ||
        !(hd.alpha > 0.0 && hd.alpha < 2.0) || !(hd.h > 0.0) || hd.N < 1 || hd.N > (1LL << 31) ||
        (hd.has_y1 != 0 && hd.has_y1 != 1) || (hd.has_y1 && !(hd.alpha > 1.0)))
        return srv_fail(FABM_EINVAL, "checkpoint header is invalid");
    const int64_t nblk = (hd.N + kSL - 1) / kSL;
    const int64_t rows = hd.c == 0 ? 0 : std::min<int64_t>(hd.N, hd.c * kSL) + 1;
    const size_t n_g = (size_t)4 * kSL * hd.dim;
    if (hd.c < 0 || hd.c >= nblk || hd.rows != rows ||
        size != sizeof hd + sizeof(double) * ((size_t)2 * rows * hd.dim + n_g))
        return srv_fail(FABM_EINVAL, "checkpoint sizes are inconsistent");
    Req r{};
    r.dim = hd.dim, r.rhs = hd.rhs, r.alpha = hd.alpha, r.h = hd.h, r.N = hd.N;
    r.n_params = hd.n_params;
    for (int i = 0; i < kMaxParams; ++i) r.params[i] = hd.params[i];
    for (int i = 0; i < FABM_MAX_DIM; ++i) r.y0[i] = hd.y0[i], r.y1[i] = hd.y1[i];
    r.has_y1 = hd.has_y1;
    if (hd.c > 0) {
        auto k = std::make_shared<Ckpt>();
        const double *F = reinterpret_cast<const double *>(static_cast<const uint8_t *>(buf) + sizeof hd);
        k->c = hd.c;
        k->status = hd.status;
        k->F.assign(F, F + rows * hd.dim);
        k->Y.assign(F + rows * hd.dim, F + 2 * rows * hd.dim);
        k->G.assign(F + 2 * rows * hd.dim, F + 2 * rows * hd.dim + n_g);
        r.ckpt = std::move(k);
    }
    std::lock_guard<std::mutex> lk(S->mu);
    r.ticket = S->next_ticket++;
    S->queue.push_back(r);
    S->results[r.ticket] = {FABM_REQ_WAITING, FABM_OK, nullptr};
    S->shapes[r.ticket] = {r.N, r.dim};
    *ticket = r.ticket;
    return FABM_OK;
}

fabm_status fabm_server_shape(fabm_server *S, int64_t ticket, int64_t *N, int *dim)
{
    set_last_error("");
    if (!S || !N || !dim) return srv_fail(FABM_EINVAL, "NULL argument");
    std::lock_guard<std::mutex> lk(S->mu);
    auto it = S->shapes.find(ticket);
    if (it == S->shapes.end()) return srv_fail(FABM_EINVAL, "unknown ticket %lld", (long long)ticket);
    *N = it->second.first;
    *dim = it->second.second;
    return FABM_OK;
}

fabm_status fabm_server_cancel(fabm_server *S, int64_t ticket)
{
    set_last_error("");
    if (!S) return srv_fail(FABM_EINVAL, "server is NULL");
    std::lock_guard<std::mutex> lk(S->mu);
    auto it = S->results.find(ticket);
    if (it == S->results.end()) return srv_fail(FABM_EINVAL, "unknown ticket %lld", (long long)ticket);
    S->results.erase(it);
    S->shapes.erase(ticket);
    S->finished.erase(std::remove(S->finished.begin(), S->finished.end(), ticket), S->finished.end());
    for (auto q = S->queue.begin(); q != S->queue.end(); ++q)
        if (q->ticket == ticket) {
            S->queue.erase(q);
            return FABM_OK;
        }
    for (size_t i = 0; i < S->slots.size(); ++i)
        if (S->slots[i].req.ticket == ticket) {
            SRV_TRY(cudaFreeAsync(S->slots[i].mem, S->sR));
            S->in_use -= S->slots[i].bytes;
            S->slots.erase(S->slots.begin() + (std::ptrdiff_t)i);
            S->table_dirty = true;
            return FABM_OK;
        }
    return FABM_OK;  // finished: its result is dropped
}

fabm_status fabm_server_finished(fabm_server *S, int64_t *tickets, int max, int *n)
{
    set_last_error("");
    if (!S || !n || max < 0 || (max > 0 && !tickets)) return srv_fail(FABM_EINVAL, "bad argument");
    std::lock_guard<std::mutex> lk(S->mu);
    const int k = (int)std::min<size_t>((size_t)max, S->finished.size());
    for (int i = 0; i < k; ++i) tickets[i] = S->finished[i];
    S->finished.erase(S->finished.begin(), S->finished.begin() + k);
    *n = k;
    return FABM_OK;
}

fabm_status fabm_server_stats(const fabm_server *S, int64_t *steps, int64_t *launches,
                              size_t *bytes_in_use)
{
    set_last_error("");
    if (!S) return srv_fail(FABM_EINVAL, "server is NULL");
    if (steps) *steps = S->steps_done;
    if (launches) *launches = S->launches;
    if (bytes_in_use) *bytes_in_use = S->in_use;
    return FABM_OK;
}

fabm_status fabm_server_destroy(fabm_server *S)
{
    set_last_error("");
    if (!S) return FABM_OK;
    const int dev = S->device;
    int prev = -1;
    if (cudaGetDevice(&prev) == cudaSuccess && prev != dev) cudaSetDevice(dev);
    delete S;
    if (prev >= 0 && prev != dev) cudaSetDevice(prev);
    return FABM_OK;
}

}  // extern "C"
