// a4 + a5 on the tensor-history path: the predictor -> f -> corrector -> f
// chain of Sec. 2 of arXiv:1710.01133 with one lane per column (trajectory b,
// component i), 32/D trajectories to a team of five warps.
//
// The history launches (far segments and the newest segments, history_far.cu,
// history_split.cu) deliver every point k < cL of block c, so a step only adds
// the points of its own block.  Targets m = cL+1+a, a < 64, points f_{cL+j},
// j = 0..64, in sub-blocks of 8 targets:
//   helpers (4 warps, each 4 of a sub-block's 16 sums): the base T + h^a G_P(m)
//           or h^a (G_C(m) + D(m) f_0) from the history and the points before the
//           sub-block.  All but the last 8 of them are summed while the chain
//           runs the sub-block before; the last 8 once it is done;
//   chain   (1 warp): the sub-block's own points and the step: y^P, exchange of
//           y^P between the lanes of the trajectory (shuffles), f(t, y^P),
//           y = T + h^a (... + f^P / Gamma(a+2)), exchange, f(t, y);
//   output  by the helpers, a sub-block behind: the float-float increment
//           h^a (...) in the double-sized slot of y (finish_y_kernel adds the
//           Taylor part in double after the last block), f as a float-float
//           pair, and after the last step the bf16 slices of the segment that
//           the next blocks' history reads.
// All in float-float; GB300 runs FP64 at 1/64 of the fp32 rate with a long
// latency, so no FP64 operation is left: the time-only part of f comes from a
// table (aux_kernel, on another stream), parameters and y_0 from float-float
// copies, and y becomes a double once at the end.
//
// The float-float operations of a column, and their order, do not depend on the
// number of warps: the sums run over the points in ascending order whoever adds
// them.  (They decide the last bits of f, and those now and then a slice.)
//
// What bounds it: alone, the latency of a step's float-float operations (a
// product takes 25 cycles, a sum 32, a multiply-add 36, a shuffle 26; ~450 cycles
// a step for the Lorenz type); beside the tensor kernels, which leave wide
// batches few SMs, its issue slots.  Hence the helpers, their weights held in
// registers (11 loads for 32 products), operand selection instead of branches
// on the component, and the slices written here instead of by a launch of their
// own.  A block of 64 steps alone, one or two warps per 32 columns before / now:
// LCR 1024 58 (a lane per target) / 37.5 us, Lorenz type 256 37 (likewise) / 34,
// oscillator 4096 97 / 49.  Whole solves: LCR 1024 x 2^14 24.1 / 20.2 ms, Lorenz
// type 256 x 2^16 87.8 / 52.4, 256 x 2^18 495 / 425, oscillator 4096 x 2^13 20.4 /
// 16.9, 4096 x 2^16 317 / 308.  Measured and dropped: a second chain warp for
// the sub-block's sums, handed over target by target (40 instead of 37 us, LCR),
// helpers that take each point as it appears (40), sub-blocks of 4 (20.7 instead
// of 19.8 ms, both on one box).
#include <algorithm>
#include <type_traits>

#include "recurrence.cuh"
#include "split_slices.cuh"

namespace fabm {
namespace {

constexpr int kColL = kSplitSeg;   // targets per block
constexpr int kSub = 8;            // targets per sub-block
constexpr int kHelpers = 4;
constexpr int kSums = 2 * kSub / kHelpers;  // sums per helper
constexpr int kRows = kSub / kHelpers;      // output rows per helper
constexpr int kTeam = 1 + kHelpers;  // warps per team
constexpr int kMaxTeams = 3;         // teams per CTA at most (registers: <= 136 per thread)

// Shared memory of a team.
struct TeamMem {
    FF f[kColL + 1][kWarp];        // f_{cL+j} of the team's columns
    FF inc[kColL][kWarp];          // increments of y
    FF sum[2 * kSub][kWarp];       // handed to the chain: sums over the points before the
    FF base[2 * kSub][kWarp];      // sub-block (running sum, errors) and bases, P then C
    FF T[kSub][kWarp];             // Taylor part, if y'(0) is given
    FF aux[kSub][kWarp];           // forcing of the sub-block
};
// Of a CTA: h^a B(d), h^a A(d), d = 0..64, then the teams.
constexpr size_t team_smem_bytes(int teams)
{
    return sizeof(FF) * 2 * (kColL + 2) + teams * sizeof(TeamMem);
}

__device__ __forceinline__ bool finite_f(float x)
{
    return (__float_as_uint(x) & 0x7f800000u) != 0x7f800000u;
}

__device__ __forceinline__ FF ld_ff(const float2 *p)
{
    const float2 v = *p;
    return FF(v.x, v.y);
}

// History of every point before block c for target a of column col, kind k
// (0 predictor, 1 corrector): the far value plus the near partials (at most
// kMaxNear), all loads issued before the additions.
constexpr int kMaxNear = 3;
__device__ __forceinline__ void hist_load(const HistIn &h, int k, int a, int64_t col, int cols,
                                          float2 (&v)[kMaxNear + 1])
{
    v[0] = h.G ? h.G[((int64_t)k * h.g_rows + h.g_off + a) * cols + col] : make_float2(0.f, 0.f);
#pragma unroll
    for (int ch = 0; ch < kMaxNear; ++ch)
        v[ch + 1] = ch < h.n_near ? h.near[(((int64_t)ch * 2 + k) * kColL + a) * cols + col]
                                  : make_float2(0.f, 0.f);
}
__device__ __forceinline__ FF hist_sum(const HistIn &h, const float2 (&v)[kMaxNear + 1])
{
    if (h.near_as_chunk) {  // the chunk after the last of G (combine_split_kernel)
        float hi = v[0].x, lo = v[0].y;
        ff_add_chunk(hi, lo, v[1].x, v[1].y);
        return FF(hi, lo);
    }
    FF s(v[0].x, v[0].y);
#pragma unroll
    for (int ch = 1; ch <= kMaxNear; ++ch) s = s + FF(v[ch].x, v[ch].y);
    return s;
}
__device__ __forceinline__ FF hist_in(const HistIn &h, int k, int a, int64_t col, int cols)
{
    float2 v[kMaxNear + 1];
    hist_load(h, k, a, col, cols, v);
    return hist_sum(h, v);
}
// Time-only part of f for the 64 targets of block c: X[a][b] = aux(t_m, p_b),
// m = 64c+1+a, as float-float pairs.
template <class Rhs>
__global__ void aux_kernel(DevBatch bt, double h, int64_t c, float2 *__restrict__ X)
{
    const int64_t n = (int64_t)kColL * bt.B;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int a = (int)(e / bt.B);
        const int64_t b = e % bt.B;
        double p[kMaxParams];
#pragma unroll
        for (int q = 0; q < kMaxParams; ++q) p[q] = bt.params[b * kMaxParams + q];
        const FF v = ff_from_double(Rhs::aux((double)(c * kColL + 1 + a) * h, p));
        X[e] = make_float2(v.hi, v.lo);
    }
}

// y_m = T(t_m) + (hi + lo) in double for m = m_lo .. min(m_hi, N_each[b])
// (m_lo >= 1), where the recurrence left the float-float increment (hi, lo) in
// y's slot; T = y0, or y0 + t y'(0) for 1 < alpha < 2.
__global__ void finish_y_kernel(DevBatch bt, double h, int64_t m_lo, int64_t m_hi)
{
    const int64_t per_traj = (m_hi - m_lo + 1) * bt.dim;
    const int64_t n = (int64_t)bt.B * per_traj;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t b = e / per_traj, r = e % per_traj;
        const int64_t m = m_lo + r / bt.dim;
        const int i = (int)(r % bt.dim);
        if (m > bt.N_each[b]) continue;
        double *slot = bt.Y + (b * (bt.N + 1) + m) * bt.dim + i;
        const float2 v = *reinterpret_cast<const float2 *>(slot);
        const double y0 = bt.y0[b * bt.dim + i];
        const double T = bt.y1 ? fma((double)m * h, bt.y1[b * bt.dim + i], y0) : y0;
        *slot = T + ((double)v.x + (double)v.y);
    }
}

__device__ __forceinline__ void team_sync(int id)
{
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(kTeam * kWarp) : "memory");
}

struct TeamArgs {
    DevBatch bt;
    const float2 *WB, *WA, *WD;
    const float2 *par, *y0;  // float-float copies: [B][kMaxParams], [cols]
    float2 ha, ha_ig2;       // h^a, h^a / Gamma(a+2)
    double h;
    int64_t c;
    HistIn hin;
    const float2 *X;         // forcing table of block c ([64][B] pairs), if Rhs::kForcing
    __nv_bfloat16 *Fs;       // slices and exponents of segment c, or NULL (last block)
    int *Ef;
    int n_ct;
};

// Team q of CTA x advances the trajectories 32/D * (x * teams + q) ...
// Y1: bt.y1 is set (1 < alpha < 2, Taylor part y0 + t y'(0)).
template <class Rhs, int D, bool Y1>
__global__ void __launch_bounds__(kMaxTeams *kTeam *kWarp)
    recur_team_kernel(const __grid_constant__ TeamArgs a)
{
    constexpr int TPW = kWarp / D;  // trajectories per team
    extern __shared__ __align__(16) FF smem_ff[];
    FF *sB = smem_ff, *sA = smem_ff + (kColL + 2);
    const int warp = threadIdx.x / kWarp, lane = threadIdx.x % kWarp;
    // warps 0 and 4 share an SM sub-partition, so the chain (role 0) is warp 1
    const int team = warp / kTeam, role = (warp % kTeam + kTeam - 1) % kTeam;
    TeamMem &tm = reinterpret_cast<TeamMem *>(smem_ff + 2 * (kColL + 2))[team];
    const int bar1 = 1 + 2 * team, bar2 = 2 + 2 * team;

    for (int d = threadIdx.x; d <= kColL; d += blockDim.x) sB[d] = ld_ff(a.WB + d), sA[d] = ld_ff(a.WA + d);
    const DevBatch &bt = a.bt;
    const int g = lane / D, i = lane % D;
    const int64_t b = ((int64_t)blockIdx.x * (blockDim.x / (kTeam * kWarp)) + team) * TPW + g;
    const bool act = g < TPW && b < bt.B;
    const int64_t bb = act ? b : 0;  // in-range index for the loads of idle lanes
    const int64_t col = bb * D + i;
    const int64_t m0 = a.c * kColL;
    const int64_t Nb = act ? bt.N_each[bb] : 0;
    const int steps = (int)(Nb - m0 < 0 ? 0 : (Nb - m0 < kColL ? Nb - m0 : kColL));
    const int wsteps = (int)__reduce_max_sync(0xffffffffu, (unsigned)steps);
    const float2 *F2 = reinterpret_cast<const float2 *>(bt.F);
    if (role == 0) tm.f[0][lane] = ld_ff(F2 + m0 * bt.ldF + col);
    __syncthreads();         // the only CTA-wide barrier
    if (wsteps == 0) return;  // every trajectory of the team has finished (uniform over the team)
    const FF T0 = ld_ff(a.y0 + col);

    if (role == 0) {
        // ---- chain ----
        FF pf[kMaxParams];
#pragma unroll
        for (int q = 0; q < kMaxParams; ++q) pf[q] = ld_ff(a.par + bb * kMaxParams + q);
        // the time-independent aux is a constant right-hand side's p0 or nothing
        const FF aux0 = std::is_same_v<Rhs, RhsConst> ? pf[0] : FF(0);
        const FF ha_ig2(a.ha_ig2.x, a.ha_ig2.y);
        FF fn = tm.f[0][lane];
        for (int a0 = 0; a0 < wsteps; a0 += kSub) {
            team_sync(bar1);  // f up to f_{cL+a0} is in tm.f
            team_sync(bar2);  // the helpers' sums are in tm.sum
            FF accP[kSub], accC[kSub];
#pragma unroll
            for (int r = 0; r < kSub; ++r) accP[r] = tm.sum[r][lane], accC[r] = tm.sum[kSub + r][lane];
            // no test of wsteps in here (targets past the last are computed and
            // dropped): the steps of a sub-block are one stretch of code, so that
            // the work off the serial path fills its latencies
#pragma unroll
            for (int r = 0; r < kSub; ++r) {
                const FF T = Y1 ? tm.T[r][lane] : T0;
                const FF yp = T + (tm.base[r][lane] + ff_norm(accP[r]));
                const FF ax = Rhs::kForcing ? tm.aux[r][lane] : aux0;
                FF y[D];
#pragma unroll
                for (int q = 0; q < D; ++q) y[q] = D == 1 ? yp : shfl_ff(yp, g * D + q);
                const FF fp = Rhs::template lanes<D>(i, y, yp, pf, ax);
                // h^a (history + f^P / Gamma(a+2))
                const FF rc = tm.base[kSub + r][lane] + ff_fma(ha_ig2, fp, ff_norm(accC[r]));
                const FF yc = T + rc;
#pragma unroll
                for (int q = 0; q < D; ++q) y[q] = D == 1 ? yc : shfl_ff(yc, g * D + q);
                tm.inc[a0 + r][lane] = rc;
                fn = Rhs::template lanes<D>(i, y, yc, pf, ax);
                tm.f[a0 + r + 1][lane] = fn;
#pragma unroll
                for (int r2 = r + 1; r2 < kSub; ++r2) {
                    dot2_acc(accP[r2], sB[r2 - r], fn);
                    dot2_acc(accC[r2], sA[r2 - r], fn);
                }
            }
        }
        team_sync(bar1);  // the last sub-block is done
        if (!a.Fs) return;
    } else {
        // ---- helpers: kSums sums of kind `kind`, targets r0 .. of each sub-block ----
        const int hq = role - 1, kind = hq & 1, r0 = kSums * (hq >> 1);
        const FF *w = kind ? sA : sB;
        const FF ha(a.ha.x, a.ha.y);
        const FF f0 = ld_ff(F2 + col);
        float2 *Fw = reinterpret_cast<float2 *>(bt.F);
        float2 *Yb = reinterpret_cast<float2 *>(bt.Y + bb * (bt.N + 1) * D);
        FF sum[kSums];  // running sums and errors (dot2_acc)
        float2 hv[kSums][kMaxNear + 1], wd[kSums];
        FF xa[kRows];
        // history and forcing of the sub-block at a0, loaded ahead of their use
        auto fetch = [&](int a0) {
#pragma unroll
            for (int q = 0; q < kSums; ++q) {
                const int t = a0 + r0 + q;
                hist_load(a.hin, kind, t, col, bt.cols, hv[q]);
                if (kind) wd[q] = a.WD[m0 + 1 + t];
            }
            if (Rhs::kForcing) {
#pragma unroll
                for (int q = 0; q < kRows; ++q)
                    xa[q] = ld_ff(a.X + (int64_t)(a0 + kRows * hq + q) * bt.B + bb);
            }
        };
        // the points j0 .. j0+kSub-1 to the targets s0+r0 ..
        auto add = [&](int j0, int s0) {
            const int d0 = s0 + r0 + 1 - j0 - (kSub - 1);
            FF wv[kSums + kSub - 1];
#pragma unroll
            for (int u = 0; u < kSums + kSub - 1; ++u) wv[u] = w[d0 + u];
#pragma unroll
            for (int u = 0; u < kSub; ++u) {
                const FF f = tm.f[j0 + u][lane];
#pragma unroll
                for (int q = 0; q < kSums; ++q) dot2_acc(sum[q], wv[q + kSub - 1 - u], f);
            }
        };
        auto write_out = [&](int a0) {  // its share of the targets from a0 on
#pragma unroll
            for (int q = 0; q < kRows; ++q) {
                const int t = a0 + kRows * hq + q;
                if (act && t < steps) {
                    const int64_t m = m0 + 1 + t;
                    const FF r = tm.inc[t][lane], fn = tm.f[t + 1][lane];
                    Yb[m * D + i] = make_float2(r.hi, r.lo);
                    Fw[m * bt.ldF + col] = make_float2(fn.hi, fn.lo);
                    if (!(finite_f(r.hi) && finite_f(fn.hi))) report_nonfinite(bt.status, m, (int)bb);
                }
            }
        };
        // h^a times the history of the sub-block at a0
        FF base[kSums], T[kSums];
        auto set_bases = [&](int a0) {
#pragma unroll
            for (int q = 0; q < kSums; ++q) {
                FF v = ha * hist_sum(a.hin, hv[q]);
                if (kind) v = ff_fma(FF(wd[q].x, wd[q].y), f0, v);
                base[q] = v;
                if constexpr (Y1)
                    if (!kind)
                        T[q] = ff_from_double(
                            fma((double)(m0 + 1 + a0 + r0 + q) * a.h, bt.y1[col], bt.y0[col]));
            }
        };
        // the sums' first point, j = 0
        auto start = [&](int a0) {
            const FF f = tm.f[0][lane];
#pragma unroll
            for (int q = 0; q < kSums; ++q) {
                sum[q] = FF(0);
                dot2_acc(sum[q], w[a0 + r0 + q + 1], f);
            }
        };
        fetch(0);
        set_bases(0);
        for (int a0 = 0; a0 < wsteps; a0 += kSub) {
            team_sync(bar1);
            // the newest points (j = a0-7 .. a0, or j = 0) complete the sub-block's sums
            if (a0 == 0) start(0);
            else add(a0 - kSub + 1, a0);
#pragma unroll
            for (int q = 0; q < kSums; ++q) {
                tm.sum[kSub * kind + r0 + q][lane] = sum[q];
                tm.base[kSub * kind + r0 + q][lane] = base[q];
                if (Y1 && !kind) tm.T[r0 + q][lane] = T[q];
            }
            if (Rhs::kForcing) {
#pragma unroll
                for (int q = 0; q < kRows; ++q) tm.aux[kRows * hq + q][lane] = xa[q];
            }
            team_sync(bar2);
            // beside the chain's sub-block: outputs of the one before, and the
            // next one's sums over the points known now
            if (a0 > 0) write_out(a0 - kSub);
            const int an = a0 + kSub;
            if (an < wsteps) {
                fetch(an);
                start(an);
                for (int j = 1; j <= a0; j += kSub) add(j, an);
                set_bases(an);
            }
        }
        team_sync(bar1);
        write_out((wsteps - 1) / kSub * kSub);
        if (!a.Fs) return;
    }

    // the segment's slices: column = lane, points j' = 8 k1 .. (j' = 63 - j)
    if (!act) return;
    float m = 0.f;
#pragma unroll 8
    for (int j = 0; j < kColL; ++j)
        if (j <= steps) m = fmaxf(m, fabsf(tm.f[j][lane].hi));
    const int E = slice_exponent(m);
    const int ct = (int)(col / 128), cloc = (int)(col % 128);
    __nv_bfloat16 *base = slice_base(a.Fs, a.c, a.n_ct, ct, cloc);
    for (int k1 = role; k1 < 8; k1 += kTeam) {
        float hi[8], lo[8];
#pragma unroll
        for (int k0 = 0; k0 < 8; ++k0) {
            const int j = 63 - (8 * k1 + k0);
            const FF f = j <= steps ? tm.f[j][lane] : FF(0);
            hi[k0] = f.hi, lo[k0] = f.lo;
        }
        uint32_t w[3][4];
        slice8(hi, lo, E, w);
#pragma unroll
        for (int q = 0; q < 3; ++q)
            *reinterpret_cast<uint4 *>(base + q * (128 * kSplitSeg) + k1 * (128 * 8)) =
                make_uint4(w[q][0], w[q][1], w[q][2], w[q][3]);
    }
    if (role == 0) a.Ef[(a.c * a.n_ct + ct) * 128 + cloc] = E;
}

// The same block with one lane per target (targets a and a+32 on lane a), one
// CTA of D warps per trajectory: for narrow batches, where one lane per column
// leaves the GPU mostly idle.  Every pending target adds the newest point as
// it appears; the owner of the next target runs the step, the components
// exchange y through shared memory.  Same inputs and outputs as
// recur_team_kernel, but the segment's slices are left to slice_f_kernel.
template <class Rhs, int D>
__global__ void __launch_bounds__(D *kWarp)
    recur_targets_kernel(DevBatch bt, const float2 *__restrict__ WB, const float2 *__restrict__ WA,
                         const float2 *__restrict__ WD, StepConsts kc, int64_t c,
                         const HistIn hin, const float2 *__restrict__ X)
{
    constexpr int TPL = kColL / kWarp;
    __shared__ FF sB[kColL + 1], sA[kColL + 1];
    __shared__ FF sy[2][D];
    const int b = blockIdx.x;
    const int i = threadIdx.x / kWarp, lane = threadIdx.x % kWarp;
    const int64_t Nb = bt.N_each[b];
    const int64_t m0 = c * kColL;
    if (m0 >= Nb) return;  // trajectory finished (uniform over the CTA)
    for (int d = threadIdx.x; d <= kColL; d += blockDim.x) sB[d] = ld_ff(WB + d), sA[d] = ld_ff(WA + d);

    double p[kMaxParams];
    FF pf[kMaxParams];
#pragma unroll
    for (int q = 0; q < kMaxParams; ++q) {
        p[q] = bt.params[(int64_t)b * kMaxParams + q];
        pf[q] = ff_from_double(p[q]);
    }
    const int64_t col = (int64_t)b * D + i;
    const float2 *F2 = reinterpret_cast<const float2 *>(bt.F);
    const double y0 = bt.y0[col];
    const double y1 = bt.y1 ? bt.y1[col] : 0.0;
    const FF ha = ff_from_double(kc.h_alpha[0]);
    const FF ha_ig2 = ff_from_double(kc.h_alpha[0] * kc.inv_gamma2[0]);
    const FF f0 = ld_ff(F2 + col);
    const FF aux0 = Rhs::kForcing ? FF(0) : ff_from_double(Rhs::aux(0.0, p));

    FF T[TPL], bP[TPL], bC[TPL], ax[TPL], nP[TPL], nC[TPL], rc[TPL], fo[TPL];
#pragma unroll
    for (int t = 0; t < TPL; ++t) {
        const int a = lane + kWarp * t;
        const int64_t m = m0 + 1 + a;
        T[t] = bt.y1 ? ff_from_double(fma((double)m * kc.h, y1, y0)) : ff_from_double(y0);
        const FF gP = hist_in(hin, 0, a, col, bt.cols);
        const FF gC = hist_in(hin, 1, a, col, bt.cols);
        bP[t] = ha * gP;
        bC[t] = ff_fma(ld_ff(WD + m), f0, ha * gC);
        ax[t] = Rhs::kForcing ? ld_ff(X + (int64_t)a * bt.B + b) : aux0;
        nP[t] = nC[t] = rc[t] = fo[t] = FF(0);
    }
    FF fk = ld_ff(F2 + m0 * bt.ldF + col);  // the newest known point, f_{cL}
    __syncthreads();

    const int steps = (int)(Nb - m0 < kColL ? Nb - m0 : kColL);
    for (int s = 0; s < steps; ++s) {
        // every pending target adds the point cL+s; targets already done add
        // the weight of distance 0, which is 0
#pragma unroll
        for (int t = 0; t < TPL; ++t) {
            const int d = lane + kWarp * t - s + 1;
            const int dd = d > 0 ? d : 0;
            dot2_acc(nP[t], sB[dd], fk);
            dot2_acc(nC[t], sA[dd], fk);
        }
        const int owner = s % kWarp, slot = s / kWarp;  // uniform over the CTA
        FF yp(0), ncor(0), tt(0), bc(0), axs(0);
#pragma unroll
        for (int t = 0; t < TPL; ++t)
            if (t == slot) yp = T[t] + (bP[t] + ff_norm(nP[t])), ncor = ff_norm(nC[t]), tt = T[t],
                           bc = bC[t], axs = ax[t];
        FF fn(0), r(0);
        if constexpr (D == 1) {
            if (lane == owner) {
                const FF fp = Rhs::template one<D>(0, &yp, pf, axs);
                r = bc + ff_fma(ha_ig2, fp, ncor);
                const FF yc = tt + r;
                fn = Rhs::template one<D>(0, &yc, pf, axs);
            }
        } else {
            if (lane == owner) sy[0][i] = yp;
            __syncthreads();
            if (lane == owner) {
                FF y[D];
#pragma unroll
                for (int q = 0; q < D; ++q) y[q] = sy[0][q];
                const FF fp = Rhs::template one<D>(i, y, pf, axs);
                r = bc + ff_fma(ha_ig2, fp, ncor);
                sy[1][i] = tt + r;
            }
            __syncthreads();
            if (lane == owner) {
                FF y[D];
#pragma unroll
                for (int q = 0; q < D; ++q) y[q] = sy[1][q];
                fn = Rhs::template one<D>(i, y, pf, axs);
            }
        }
#pragma unroll
        for (int t = 0; t < TPL; ++t)
            if (t == slot && lane == owner) rc[t] = r, fo[t] = fn;
        fk = shfl_ff(fn, owner);
    }

    // the block's increments of y and f, one target per lane
    float2 *Yb = reinterpret_cast<float2 *>(bt.Y + (int64_t)b * (bt.N + 1) * D);
    float2 *Fw = reinterpret_cast<float2 *>(bt.F);
#pragma unroll
    for (int t = 0; t < TPL; ++t) {
        const int a = lane + kWarp * t;
        if (a < steps) {
            const int64_t m = m0 + 1 + a;
            Yb[m * D + i] = make_float2(rc[t].hi, rc[t].lo);
            Fw[m * bt.ldF + col] = make_float2(fo[t].hi, fo[t].lo);
            if (!(finite_f(rc[t].hi) && finite_f(fo[t].hi))) report_nonfinite(bt.status, m, b);
        }
    }
}

}  // namespace

cudaError_t prepare_recur_cols(int rhs, int dim)
{
    cudaError_t e = cudaSuccess;
    const bool ok = dispatch_rhs(rhs, dim, [&]<class R, int D>() {
        auto prep = [&](auto kernel) {
            cudaFuncAttributes fa;
            if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, kernel);
            if (e == cudaSuccess && fa.numRegs * kMaxTeams * kTeam * kWarp > 65536)
                e = cudaErrorInvalidConfiguration;
            if (e == cudaSuccess)
                e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)team_smem_bytes(kMaxTeams));
        };
        prep(recur_team_kernel<R, D, false>);
        prep(recur_team_kernel<R, D, true>);
    });
    return ok ? e : cudaErrorInvalidValue;
}

int recur_cols_warps(int dim, int64_t B) { return (int)((B + kWarp / dim - 1) / (kWarp / dim)); }

cudaError_t launch_recur_cols(int rhs, const DevBatch &bt, const float2 *WB, const float2 *WA,
                              const float2 *WD, const StepConsts &k, int64_t c, const HistIn &hin,
                              const ColsIn &in, int warps_per_cta, cudaStream_t st)
{
    if (warps_per_cta < 0) return cudaErrorInvalidValue;
    if (hin.n_near < 0 || hin.n_near > kMaxNear) return cudaErrorInvalidValue;
    bool need_x = false;
    const bool ok = dispatch_rhs(rhs, bt.dim, [&]<class R, int D>() {
        need_x = R::kForcing;
        if (need_x && !in.X) return;
        if (warps_per_cta == 0) {  // one lane per target
            recur_targets_kernel<R, D><<<(unsigned)bt.B, D * kWarp, 0, st>>>(bt, WB, WA, WD, k, c,
                                                                             hin, in.X);
            return;
        }
        const int teams = recur_cols_warps(D, bt.B), per = std::min(warps_per_cta, kMaxTeams);
        const unsigned blocks = (unsigned)((teams + per - 1) / per);
        auto pair = [](double v) {
            const float hi = (float)v;
            return make_float2(hi, (float)(v - (double)hi));
        };
        const TeamArgs a{bt, WB, WA, WD, in.par, in.y0, pair(k.h_alpha[0]),
                         pair(k.h_alpha[0] * k.inv_gamma2[0]), k.h, c, hin, in.X, in.Fs, in.Ef, in.n_ct};
        if (bt.y1)
            recur_team_kernel<R, D, true><<<blocks, per * kTeam * kWarp, team_smem_bytes(per), st>>>(a);
        else
            recur_team_kernel<R, D, false><<<blocks, per * kTeam * kWarp, team_smem_bytes(per), st>>>(a);
    });
    return ok && !(need_x && !in.X) ? cudaGetLastError() : cudaErrorInvalidValue;
}

bool rhs_has_forcing(int rhs, int dim)
{
    bool f = false;
    dispatch_rhs(rhs, dim, [&]<class R, int D>() { f = R::kForcing; });
    return f;
}

cudaError_t launch_aux_table(int rhs, const DevBatch &bt, double h, int64_t c, float2 *X,
                             cudaStream_t st)
{
    const int64_t n = (int64_t)kColL * bt.B;
    int64_t blocks = (n + 127) / 128;
    if (blocks > 152 * 8) blocks = 152 * 8;
    const bool ok = dispatch_rhs(rhs, bt.dim, [&]<class R, int D>() {
        aux_kernel<R><<<(unsigned)blocks, 128, 0, st>>>(bt, h, c, X);
    });
    return ok ? cudaGetLastError() : cudaErrorInvalidValue;
}

cudaError_t launch_finish_y(const DevBatch &bt, double h, int64_t m_lo, int64_t m_hi,
                            cudaStream_t st)
{
    if (m_lo < 1 || m_hi > bt.N) return cudaErrorInvalidValue;
    if (m_hi < m_lo) return cudaSuccess;
    const int64_t n = (int64_t)bt.B * (m_hi - m_lo + 1) * bt.dim;
    int64_t blocks = (n + 255) / 256;
    if (blocks > 152 * 16) blocks = 152 * 16;
    finish_y_kernel<<<(unsigned)blocks, 256, 0, st>>>(bt, h, m_lo, m_hi);
    return cudaGetLastError();
}

}  // namespace fabm
