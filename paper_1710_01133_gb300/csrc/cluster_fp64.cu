// a2 + a3 + a4 + a5 in double, one thread-block cluster per trajectory: a
// launch advances a superblock of n targets (m = nT+1 .. nT+n) of every
// trajectory, given the far history of its targets over the points k < n(T-1)
// (far_fft.cu).  Sec. 2 of arXiv:1710.01133 (Eq. abm, the corrector after it).
//
// What bounds it: GB300's FP64 unit takes a warp instruction in 64 cycles per
// SM sub-partition, dependent or not (measured: 64 cycles for chains of 1 and
// of 8 independent FMAs, one warp), so a step costs 64 cycles for each FP64
// instruction on its serial chain (accumulate, f, corrector, f) plus two
// exchanges between the components, and every other FP64 instruction that
// shares the chain's sub-partitions delays it.  One launch per block of 32
// steps spent two thirds of its time outside the chain: on launches, on
// loading the block's weights and on the lag blocks.
//
// Layout.  Targets are taken in blocks of 16; lane (kind, a) has target a's
// predictor (kind 0) or corrector (1) sum, so one FMA adds a point to both sums
// of a block.  Three parties share a block's sums, each with FP64 units to itself:
//   chain warps   (rank 0, one per component): the block's own points, the step;
//   prev warps    (rank 0, other sub-partitions): the 16 points of the block
//                 before it, each as soon as the chain has produced it;
//   helper warps  (ranks 1 .., four per CTA; in rank 0 for clusters of one): every
//                 earlier point k >= n(T-1), dealt out to the warps in turn; the
//                 warps of a CTA are added in shared memory, the CTAs by a
//                 finisher warp that owns a component's row and turns it into
//                 y0 + h^alpha (...).
// The chain stores f_k into the shared memory of every CTA of the cluster (one
// instruction: lane r writes to CTA r), and the finishers store their rows into
// the chain's CTA.  Both buffers are written once per launch and start out as
// a bit pattern that no result has, so a reader polls the value it needs and no
// flag or fence is on the way.  A helper sums the older points of block t + 1
// while the chain runs block t - 1; what is left when f of block t - 1 is
// complete is the addition of the rows, due 11 steps into block t.
//
// An FP64 result reaches the other units (shared memory, shuffles, integer
// code) about 50 cycles later than the FP64 unit itself, and a store to 16 CTAs
// holds up the stores behind it, so only the exchange stands between the
// instructions of a step, and the copies of f follow it.  Cycles per step: 355
// for the scalar system (four FP64 instructions and one hand-over), 720 for the Lorenz type (six
// and two exchanges).  Blocks of 32 with a warp instruction per kind took 457
// and 765; a chain of newest points only, the rest of the block summed by
// another warp a target ahead, 560 and 920 (the way there and back is longer
// than a step).
//
// Measured against one launch per kernel and block of 32 (whole solves):
// Lorenz-type 2^18 434 -> 91 ms, 16 x 2^15 102 -> 12.7, scalar 10^4 5.16 -> 1.79,
// LCR 256 x 2^13 of uneven length 67.2 -> 7.8.
//
// Every wait is bounded: a thread that gives up sets the error word and goes
// on without waiting, so that barriers are still met and the launch ends.
#include <algorithm>

#include "recurrence.cuh"
#include "sm100_ptx.cuh"

namespace fabm {
namespace {

using ptx::smem_u32;

constexpr int kB = 16;              // targets per block: a half-warp per kind
constexpr int kHelpWarps = 4;       // helper warps per CTA, one per SM sub-partition
constexpr int kBaseDue = 11;        // step of a block by which the next block's base row is needed
constexpr int kPw = 2 * (2 * kB + 2);  // h^a B(d), h^a A(d), d <= 2 kB + 1
constexpr unsigned long long kUnset = ~0ull;  // a NaN that no arithmetic instruction returns
constexpr long long kWaitDefault = 4000000000LL;

template <int D>
struct Roles {
    static constexpr int kPrev = D == 1 ? 1 : (D == 3 ? 1 : D);  // prev warps
    static constexpr int kPrevComps = D / kPrev;                  // components of each
    static constexpr int kPrev0 = D == 1 ? 1 : (D == 2 ? 2 : (D == 3 ? 3 : 4));
    static constexpr int kChainWarps = D == 4 ? 8 : 4;           // warps of rank 0's roles
};

// Shared memory of a CTA, in doubles from the start: f of both superblocks, then
// the chain's and prev warps' arrays (rank 0) and the helpers' (ranks 1 ..), in
// the same place where no CTA has both roles.
struct Layout {
    int sf, base, near, sy, pw, wb, wa, rows, red, total;
};
__host__ __device__ inline Layout layout(int D, int nW, int n, int CS)
{
    Layout l;
    const int H = CS > 1 ? CS - 1 : 1;
    const int ro = (D + H - 1) / H;  // rows a finisher owns at most
    int o = 0;
    l.sf = o, o += 2 * n * D;
    const int roles = o;
    l.base = o, o += n * 2 * D;
    l.near = o, o += 2 * D * kWarp;
    l.sy = o, o += 4 * D;
    l.pw = o, o += nW * kPw;
    const int chain_end = o;
    if (CS > 1) o = roles;
    l.wb = o, o += nW * (2 * n + 2);
    l.wa = o, o += nW * (2 * n + 2);
    l.rows = o, o += 2 * ro * H * kWarp;
    l.red = o, o += 2 * kHelpWarps * D * kWarp;
    l.total = o > chain_end ? o : chain_end;
    return l;
}

__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t cluster_size()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release;\nbarrier.cluster.wait.acquire;" ::: "memory");
}
__device__ __forceinline__ uint32_t mapa(uint32_t addr, uint32_t rank)
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
// A value to another CTA of the cluster; the pattern that marks an unset slot
// is replaced by another NaN.
__device__ __forceinline__ void put(uint32_t remote, double v)
{
    unsigned long long u = (unsigned long long)__double_as_longlong(v);
    if (u == kUnset) u ^= 1ull;
    asm volatile("st.relaxed.cluster.shared::cluster.b64 [%0], %1;" ::"r"(remote), "l"(u) : "memory");
}
__device__ __forceinline__ unsigned long long peek(const double *p)
{
    unsigned long long u;
    asm volatile("ld.relaxed.cluster.shared::cta.b64 %0, [%1];" : "=l"(u) : "r"(smem_u32(p)) : "memory");
    return u;
}
// The aligned form: the lanes of a warp have to arrive together.
__device__ __forceinline__ void named_sync(int id, int threads)
{
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

struct Waiter {
    long long limit;
    unsigned *err;
    bool ok = true;
    __device__ void give_up()
    {
        ok = false;
        atomicOr(err, 1u);
    }
    // the value at p once it is set
    __device__ __forceinline__ double get(const double *p)
    {
        unsigned long long u = peek(p);
        if (u == kUnset && ok) {
            const long long t0 = clock64();
            while ((u = peek(p)) == kUnset)
                if (clock64() - t0 > limit) {
                    give_up();
                    break;
                }
        }
        return __longlong_as_double((long long)u);
    }
    // phase `parity` of a barrier that other CTAs of the cluster arrive on
    __device__ void phase(uint64_t *bar, uint32_t parity)
    {
        if (!ok) return;
        const long long t0 = clock64();
        for (;;) {
            uint32_t done;
            asm volatile(
                "{\n .reg .pred p;\n"
                " mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
                " selp.u32 %0, 1, 0, p;\n}\n"
                : "=r"(done)
                : "r"(smem_u32(bar)), "r"(parity)
                : "memory");
            if (done) return;
            if (clock64() - t0 > limit) {
                give_up();
                return;
            }
        }
    }
};

struct Args {
    DevBatch bt;
    DevWeights w;
    StepConsts kc;
    int64_t T;        // superblock
    int n;            // targets per superblock, a multiple of 32
    const double *G;  // far history [2][n][cols] over k < n(T-1), or NULL (T < 2)
    const double *X;  // time-only part of f, [B][n] (aux_table_kernel), if Rhs::kForcing
    unsigned *err;
    long long wait;
};

struct Chain {
    const Args &a;
    int b;
    int64_t nT, Nb;
    int known, CS;
    double *sm;
    const Layout &l;
    int lane;
};

// The steps of component I; lane (kind, ta) has the sum of target ta of the
// block.  A step's serial path is newest point -> exchange -> f -> corrector ->
// exchange -> f; what else uses f_k is placed behind the addition that takes it
// inside the FP64 unit.
template <class Rhs, int D, int I>
__device__ __forceinline__ void chain_run(const Chain &c)
{
    const Args &a = c.a;
    const int lane = c.lane, ta = lane % kB;
    double *sm = c.sm;
    double p[kMaxParams];
#pragma unroll
    for (int q = 0; q < kMaxParams; ++q) p[q] = a.bt.params[(int64_t)c.b * kMaxParams + q];
    const double ha_ig2 = a.kc.h_alpha[I] * a.kc.inv_gamma2[I];
    const double aux0 = Rhs::kForcing ? 0.0 : Rhs::aux(0.0, p);
    const double *pw = sm + c.l.pw + (a.w.stride ? I * kPw : 0) + (lane / kB) * (kPw / 2);
    volatile double *sy = sm + c.l.sy;  // [2 parities][P, C][D]
    double *Yb = a.bt.Y + ((int64_t)c.b * (a.bt.N + 1) + c.nT + 1) * D + I;
    double *Fb = a.bt.F + (c.nT + 1) * a.bt.ldF + (int64_t)c.b * D + I;
    const double *near = sm + c.l.near + I * kWarp + lane;
    const uint32_t sf_to = lane < c.CS ? mapa(smem_u32(sm + c.l.sf + I), lane) : 0u;
    double fk = sm[c.l.sf + c.known * D + I], yc = 0.0, yo = 0.0, fo = 0.0;
    const double *X = Rhs::kForcing ? a.X + (int64_t)c.b * a.n : nullptr;
    double ax = aux0, ax_next = Rhs::kForcing ? X[lane] : 0.0;  // rows of 32 values, one ahead
    const int steps = (int)(c.Nb - c.nT < a.n ? c.Nb - c.nT : a.n);
    auto flush = [&](int j0, int cnt) {  // targets j0 .., a lane each
        if (lane < cnt) {
            Yb[(int64_t)(j0 + lane) * D] = yo;
            Fb[(int64_t)(j0 + lane) * a.bt.ldF] = fo;
            if (!(finite_bits(yo) && finite_bits(fo)))
                report_nonfinite(a.bt.status, c.nT + 1 + j0 + lane, c.b);
        }
    };
    for (int j0 = 0; j0 < steps; j0 += kB) {
        if (j0 % kWarp == 0) {
            if constexpr (Rhs::kForcing) {
                ax = ax_next;
                if (j0 + kWarp + lane < a.n) ax_next = X[j0 + kWarp + lane];
            }
        }
        double w = pw[ta + 1];
        const int cnt = steps - j0 < kB ? steps - j0 : kB;
        named_sync(2, (D + Roles<D>::kPrev) * kWarp);
        double acc = near[(j0 / kB & 1) * D * kWarp];
        for (int s = 0; s < cnt; ++s) {  // target nT+1+j0+s
            const int j = j0 + s;
            acc = fma(w, fk, acc);  // targets already done add distance 0 (weight 0)
            const double f_new = fk;
            w = pw[ta > s ? ta - s : 0];
            const double axs = Rhs::kForcing ? __shfl_sync(0xffffffffu, ax, j % kWarp) : ax;
            double y[D];
            const int par = (j & 1) * 2 * D;
            if constexpr (D > 1) {
                if (lane == s) sy[par + I] = acc;
            } else {
                y[0] = __shfl_sync(0xffffffffu, acc, s);
            }
            const double aC = __shfl_sync(0xffffffffu, acc, kB + s);
            if constexpr (D > 1) {
                named_sync(1, D * kWarp);
#pragma unroll
                for (int q = 0; q < D; ++q) y[q] = sy[par + q];
            }
            // behind the exchange, so that its store is not queued after these
            if (lane < c.CS) put(sf_to + (c.known + j) * D * 8, f_new);
            if (lane == ((j - 1) & (kWarp - 1))) yo = yc, fo = f_new;
            if (s == 0 && j % kWarp == 0 && j) flush(j - kWarp, kWarp);
            // every lane runs the step, so that f ends up in all of them
            const double fp = rhs_f64<Rhs, D>(I, y, p, axs);
            yc = fma(ha_ig2, fp, aC);
            if constexpr (D > 1) {
                sy[par + D + I] = yc;
                named_sync(1, D * kWarp);
#pragma unroll
                for (int q = 0; q < D; ++q) y[q] = sy[par + D + q];
            } else {
                y[0] = yc;
            }
            fk = rhs_f64<Rhs, D>(I, y, p, axs);
        }
    }
    const int last = (steps - 1) % kWarp;
    if (lane == last) yo = yc, fo = fk;
    flush(steps - 1 - last, last + 1);
}

// X[b][j] = aux(t_m, p_b) for m = nT+1+j, j < n.
template <class Rhs>
__global__ void aux_table_kernel(DevBatch bt, double h, int64_t T, int n, double *__restrict__ X)
{
    const int64_t total = (int64_t)bt.B * n;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t b = e / n, m = T * n + 1 + e % n;
        double p[kMaxParams];
#pragma unroll
        for (int q = 0; q < kMaxParams; ++q) p[q] = bt.params[b * kMaxParams + q];
        X[e] = m <= bt.N_each[b] ? Rhs::aux((double)m * h, p) : 0.0;
    }
}

// grid = B x (cluster size), cluster size CTAs per trajectory.
template <class Rhs, int D>
__global__ void __launch_bounds__((Roles<D>::kChainWarps + kHelpWarps + 1) * kWarp)
    cluster_kernel(const __grid_constant__ Args a)
{
    extern __shared__ __align__(16) double sm[];
    __shared__ uint64_t rows_full[2];
    using R = Roles<D>;
    const int warp = threadIdx.x / kWarp, lane = threadIdx.x % kWarp;
    const int CS = (int)cluster_size(), rank = (int)cluster_rank();
    const int H = CS > 1 ? CS - 1 : 1;      // CTAs with helper warps
    const int hr = CS > 1 ? rank - 1 : 0;   // this CTA among them (-1: none)
    const int hw0 = CS > 1 ? 0 : R::kChainWarps;
    const int b = (int)blockIdx.x / CS;
    const int n = a.n;
    const int64_t nT = a.T * n;
    const int64_t Nb = a.bt.N_each[b];
    if (nT >= Nb) return;  // trajectory finished (the whole cluster)
    const int nb = (int)((Nb - nT < n ? Nb - nT : n) + kB - 1) / kB;  // blocks of this launch
    const int64_t k0 = a.T > 0 ? nT - n : 0;                        // first point summed here
    const int known = (int)(nT - k0);                               // points before f_{nT}
    const int nW = a.w.stride ? D : 1;
    const Layout l = layout(D, nW, n, CS);
    const int ws = 2 * n + 2;
    double *sf = sm + l.sf, *base = sm + l.base;

    // known points, unset slots, weights
    for (int j = threadIdx.x; j < 2 * n * D; j += blockDim.x) {
        const int64_t k = k0 + j / D;
        sf[j] = k <= nT ? a.bt.F[k * a.bt.ldF + (int64_t)b * D + j % D]
                        : __longlong_as_double((long long)kUnset);
    }
    if (hr >= 0) {
        const int64_t dmax = known + nb * kB;  // largest distance (< w.N)
        for (int q = 0; q < nW; ++q)
            for (int j = threadIdx.x; j <= dmax; j += blockDim.x) {
                sm[l.wb + q * ws + j] = a.w.B[q * a.w.stride + j];
                sm[l.wa + q * ws + j] = a.w.A[q * a.w.stride + j];
            }
        if (threadIdx.x < 2) {
            int owned = 0;
            for (int q = hr; q < D; q += H) ++owned;
            ptx::mbar_init(&rows_full[threadIdx.x], owned ? owned * H : 1);
            ptx::fence_mbar_init();
        }
    }
    if (rank == 0) {
        for (int j = threadIdx.x; j < nb * 2 * D * kB; j += blockDim.x)
            base[j] = __longlong_as_double((long long)kUnset);
        for (int j = threadIdx.x; j < nW * kPw; j += blockDim.x) {
            const int q = j / kPw, d = j % (kPw / 2);
            const double *W = (j % kPw < kPw / 2 ? a.w.B : a.w.A) + q * a.w.stride;
            sm[l.pw + j] = pick<D>(a.kc.h_alpha, q) * W[d];
        }
    }
    Waiter wt{a.wait > 0 ? a.wait : kWaitDefault, a.err};
    cluster_sync();

    if (rank == 0 && warp < D) {
        const Chain ch{a, b, nT, Nb, known, CS, sm, l, lane};
        if constexpr (D == 1) {
            chain_run<Rhs, D, 0>(ch);
        } else {
            if (warp == 0) chain_run<Rhs, D, 0>(ch);
            else if (warp == 1) chain_run<Rhs, D, 1>(ch);
            else if (warp == 2) chain_run<Rhs, D, D >= 3 ? 2 : 0>(ch);
            else chain_run<Rhs, D, D >= 4 ? 3 : 0>(ch);
        }
    } else if (rank == 0 && warp >= R::kPrev0 && warp < R::kPrev0 + R::kPrev) {
        // ---- prev: the points of the block before each block, kPrevComps components ----
        constexpr int C = R::kPrevComps;
        const int c0 = (warp - R::kPrev0) * C;
        const double *pw = sm + l.pw + (lane / kB) * (kPw / 2) + kB + 1 + lane % kB;
        for (int t = 0; t < nb; ++t) {
            double nxt[C];
            if (t == 0) {
#pragma unroll
                for (int q = 0; q < C; ++q) nxt[q] = wt.get(base + (c0 + q) * kWarp + lane);
            } else {
#pragma unroll
                for (int q = 0; q < C; ++q) nxt[q] = 0.0;
                const double *f = sf + (known + (t - 1) * kB) * D + c0;
#pragma unroll 1
                for (int s = 0; s < kB; ++s) {
                    double w[C];
#pragma unroll
                    for (int q = 0; q < C; ++q) w[q] = pw[(nW > 1 ? (c0 + q) * kPw : 0) - s];
                    if (s == kBaseDue) {
#pragma unroll
                        for (int q = 0; q < C; ++q)
                            nxt[q] += wt.get(base + (t * D + c0 + q) * kWarp + lane);
                    }
#pragma unroll
                    for (int q = 0; q < C; ++q) nxt[q] = fma(w[q], wt.get(f + s * D + q), nxt[q]);
                }
            }
#pragma unroll
            for (int q = 0; q < C; ++q) sm[l.near + ((t & 1) * D + c0 + q) * kWarp + lane] = nxt[q];
            __syncwarp();  // lanes leave their waits one by one; the barrier takes whole warps
            named_sync(2, (D + R::kPrev) * kWarp);
        }
    } else if (hr >= 0 && warp >= hw0 && warp < hw0 + kHelpWarps) {
        // ---- helpers ----
        const int w = warp - hw0;
        const int g = hr * kHelpWarps + w, HW = H * kHelpWarps;
        const double *wk = sm + (lane < kB ? l.wb : l.wa) + lane % kB + 1;
        for (int t = 0; t < nb; ++t) {
            const int lim = known + (t > 1 ? t - 1 : 0) * kB;  // points k0 .. k0+lim-1
            const double *wt0 = wk + known + t * kB;           // weight of point index j: wt0[-j]
            double acc[D];
#pragma unroll
            for (int q = 0; q < D; ++q) acc[q] = 0.0;
            auto add = [&](int j, const double (&f)[D]) {
                if (nW > 1) {
#pragma unroll
                    for (int q = 0; q < D; ++q) acc[q] = fma(wt0[q * ws - j], f[q], acc[q]);
                } else {
                    const double v = wt0[-j];
#pragma unroll
                    for (int q = 0; q < D; ++q) acc[q] = fma(v, f[q], acc[q]);
                }
            };
            int j = g;
            const int old = lim < known ? lim : known;
#pragma unroll 4
            for (; j < old; j += HW) {
                double f[D];
#pragma unroll
                for (int q = 0; q < D; ++q) f[q] = sf[j * D + q];
                add(j, f);
            }
#pragma unroll 2
            for (; j < lim; j += HW) {
                double f[D];
#pragma unroll
                for (int q = 0; q < D; ++q) f[q] = wt.get(sf + j * D + q);
                add(j, f);
            }
            // the CTA's four warps, then the row's owner
            double(*red)[D][kWarp] =
                reinterpret_cast<double(*)[D][kWarp]>(sm + l.red) + (t & 1) * kHelpWarps;
#pragma unroll
            for (int q = 0; q < D; ++q) red[w][q][lane] = acc[q];
            __syncwarp();  // as above
            named_sync(3, kHelpWarps * kWarp);
            if (w < D) {
                // the slot's last rows, of block t-2, are used up once the chain has
                // stepped on from that block's first target
                if (t >= 2) wt.get(sf + (known + (t - 2) * kB + 1) * D);
                const int q = w, ro = (D + H - 1) / H;
                const double v = (red[0][q][lane] + red[1][q][lane]) + (red[2][q][lane] + red[3][q][lane]);
                const uint32_t owner = CS > 1 ? 1 + q % H : 0;
                put(mapa(smem_u32(sm + l.rows + (((t & 1) * ro + q / H) * H + hr) * kWarp + lane), owner), v);
                __syncwarp();
                if (lane == 0) {
                    const uint32_t bar = mapa(smem_u32(&rows_full[t & 1]), owner);
                    asm volatile("fence.acq_rel.cluster;\n"
                                 "mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar)
                                 : "memory");
                }
            }
        }
    } else if (hr >= 0 && hr < D && warp == hw0 + kHelpWarps) {
        // ---- finisher: the rows of the components hr, hr + H, ... ----
        const int ro = (D + H - 1) / H, kind = lane / kB, ta = lane % kB;
        for (int t = 0; t < nb; ++t) {
            const int64_t m = nT + t * kB + 1 + ta;
            for (int i = hr; i < D; i += H) {
                const int64_t col = (int64_t)b * D + i;
                double far = a.G ? a.G[((int64_t)kind * n + t * kB + ta) * a.bt.cols + col] : 0.0;
                if (kind) far = fma(a.w.D[i * a.w.stride + m], a.bt.F[col], far);
                const double y0 = a.bt.y0[col];
                const double Tm = a.bt.y1 ? fma((double)m * a.kc.h, a.bt.y1[col], y0) : y0;
                if (i == hr) wt.phase(&rows_full[t & 1], (t >> 1) & 1);
                const double *r = sm + l.rows + (((t & 1) * ro + i / H) * H) * kWarp + lane;
                double v = 0.0;
                for (int h = 0; h < H; ++h) v += r[h * kWarp];
                put(mapa(smem_u32(base + (t * D + i) * kWarp + lane), 0),
                    fma(pick<D>(a.kc.h_alpha, i), far + v, Tm));
            }
        }
    }
    cluster_sync();  // no CTA leaves while another may still write to its shared memory
}

template <class Rhs, int D>
cudaError_t cluster_config(int B, int CS, int n, int nW, bool alone, cudaLaunchConfig_t *cfg,
                           cudaLaunchAttribute *attr)
{
    constexpr int kc = Roles<D>::kChainWarps;
    const int warps = CS > 1 ? (kc > kHelpWarps + 1 ? kc : kHelpWarps + 1) : kc + kHelpWarps + 1;
    size_t smem = sizeof(double) * (size_t)layout(D, nW, n, CS).total;
    if (alone && smem < 120 * 1024) smem = 120 * 1024;  // one CTA per SM
    constexpr size_t kMaxSmem = 226 * 1024;
    if (smem > kMaxSmem) return cudaErrorInvalidConfiguration;
    *cfg = cudaLaunchConfig_t{};
    cfg->gridDim = dim3((unsigned)(B * CS));
    cfg->blockDim = dim3((unsigned)(warps * kWarp));
    cfg->dynamicSmemBytes = smem;
    attr->id = cudaLaunchAttributeClusterDimension;
    attr->val.clusterDim.x = (unsigned)CS, attr->val.clusterDim.y = 1, attr->val.clusterDim.z = 1;
    cfg->attrs = attr;
    cfg->numAttrs = 1;
    auto k = cluster_kernel<Rhs, D>;
    // the same limit in every call: a solver on another thread may be about to launch
    // this kernel with another size
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxSmem);
    if (e == cudaSuccess && CS > 8)
        e = cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    return e;
}

}  // namespace

int cluster_max_active(int rhs, int dim, bool multi, int CS, int n)
{
    int num = 0;
    dispatch_rhs(rhs, dim, [&]<class R, int D>() {
        cudaLaunchConfig_t cfg;
        cudaLaunchAttribute attr;
        if (cluster_config<R, D>(1, CS, n, multi ? D : 1, CS > 1, &cfg, &attr) != cudaSuccess ||
            cudaOccupancyMaxActiveClusters(&num, cluster_kernel<R, D>, &cfg) != cudaSuccess)
            num = 0;
        cudaGetLastError();
    });
    return num;
}

cudaError_t launch_cluster_fp64(int rhs, const DevBatch &bt, const DevWeights &w,
                                const StepConsts &k, int64_t T, int n, int CS, bool alone,
                                const double *G,
                                const double *X, unsigned *err, long long wait_cycles, cudaStream_t st)
{
    cudaError_t e = cudaErrorInvalidValue;
    dispatch_rhs(rhs, bt.dim, [&]<class R, int D>() {
        cudaLaunchConfig_t cfg;
        cudaLaunchAttribute attr;
        e = cluster_config<R, D>(bt.B, CS, n, w.stride ? D : 1, alone, &cfg, &attr);
        if (e != cudaSuccess) return;
        cfg.stream = st;
        const Args a{bt, w, k, T, n, G, X, err, wait_cycles};
        e = cudaLaunchKernelEx(&cfg, cluster_kernel<R, D>, a);
    });
    return e;
}

cudaError_t launch_aux_rows(int rhs, const DevBatch &bt, double h, int64_t T, int n, double *X,
                            cudaStream_t st)
{
    const int64_t blocks = std::min<int64_t>(((int64_t)bt.B * n + 127) / 128, 152 * 16);
    const bool ok = dispatch_rhs(rhs, bt.dim, [&]<class R, int D>() {
        aux_table_kernel<R><<<(unsigned)blocks, 128, 0, st>>>(bt, h, T, n, X);
    });
    return ok ? cudaGetLastError() : cudaErrorInvalidValue;
}

}  // namespace fabm
