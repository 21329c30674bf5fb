// a4 + a5 in double: the sequential predictor -> f -> corrector -> f chain of
// Sec. 2 of arXiv:1710.01133 (Eq. abm, the corrector after it) inside one
// block of L = 32*TPL targets.  One CTA per trajectory, one warp per
// component.
//
// Warp i keeps, in lane a + 32t, the running predictor and corrector sums of
// component i for target m = cL+1+a+32t:
//   start   far part from the history kernels (points k < (c-1)L) and the
//           k = 0 correction D(m) f_0;
//   lag 1   the L points of block c-1, all known when the block starts;
//   steps   for s = 0..L-1 the point k = cL+s becomes known; every pending
//           target adds its term, and the owner of target k+1 then has the
//           whole sum and runs the step: y^P_i, exchange of y^P across the
//           component warps, f_i(t, y^P), y_i, exchange of y, f_i(t, y).
// The accumulators hold y0 + h^alpha * (partial sum) and the weights are
// pre-multiplied by h^alpha, so the owner's accumulate of the newest point is
// already y^P (and y0 + h^alpha S^C): six dependent FP64 operations per step
// for a Lorenz-type component (accumulate, f, corrector, f).
// On GB300 a warp FP64 instruction takes the FP64 pipe for many cycles
// whatever the number of active lanes, so adding f_k to all pending targets
// of a warp costs one instruction per sum, and the components run on separate
// warps so that their chains overlap.  The time-only part of f (forcing) is
// evaluated for every target at block start, off the chain.
#pragma once

#include "rhs.cuh"

namespace fabm {


// v[q] for a runtime q < D without indexing the array dynamically (which
// would copy the kernel's parameter block to local memory).
template <int D>
__device__ inline double pick(const double (&v)[FABM_MAX_DIM], int q)
{
    double r = v[0];
#pragma unroll
    for (int k = 1; k < D; ++k)
        if (q == k) r = v[k];
    return r;
}

__device__ inline void report_nonfinite(unsigned long long *status, int64_t step, int traj)
{
    atomicMin(status, ((unsigned long long)step << 24) | (unsigned long long)traj);
}

// Finite test on the exponent bits (no floating-point compare).
__device__ inline bool finite_bits(double x)
{
    return ((unsigned)__double2hiint(x) & 0x7ff00000u) != 0x7ff00000u;
}

// y_0 and f_0 = f(0, y_0) of trajectory b; f_pairs: F holds float-float pairs.
template <class Rhs, int D>
__device__ inline void init_one(const DevBatch &bt, int b, bool f_pairs = false, const FFInputs &ff = {})
{
    double y[D], p[kMaxParams];
#pragma unroll
    for (int i = 0; i < kMaxParams; ++i) p[i] = bt.params[(int64_t)b * kMaxParams + i];
#pragma unroll
    for (int i = 0; i < D; ++i) y[i] = bt.y0[(int64_t)b * D + i];
    const double aux = Rhs::aux(0.0, p);
    bool ok = true;
    if (ff.par) {
#pragma unroll
        for (int i = 0; i < kMaxParams; ++i) {
            const FF v = ff_from_double(p[i]);
            ff.par[(int64_t)b * kMaxParams + i] = make_float2(v.hi, v.lo);
        }
#pragma unroll
        for (int i = 0; i < D; ++i) {
            const FF v = ff_from_double(y[i]);
            ff.y0[(int64_t)b * D + i] = make_float2(v.hi, v.lo);
        }
    }
#pragma unroll
    for (int i = 0; i < D; ++i) {
        const double f = Rhs::template one<D>(i, y, p, aux);
        bt.Y[(int64_t)b * (bt.N + 1) * D + i] = y[i];
        if (f_pairs) {
            const float hi = __double2float_rn(f);
            reinterpret_cast<float2 *>(bt.F)[(int64_t)b * D + i] =
                make_float2(hi, __double2float_rn(f - (double)hi));
        } else {
            bt.F[(int64_t)b * D + i] = f;
        }
        if (bt.Ff) bt.Ff[(int64_t)b * D + i] = (float)f;
        ok = ok && finite_bits(y[i]) && finite_bits(f);
    }
    if (!ok) report_nonfinite(bt.status, 0, b);
}

// Shared-memory doubles recur_block<*, D, TPL, LAG> needs.
template <int D, int TPL, int LAG = 1>
__host__ __device__ constexpr int recur_smem_doubles()
{
    return 2 * ((LAG + 1) * kWarp * TPL + 1) * D + 2 * D + (LAG * kWarp * TPL + 1) * D;
}

// One block of steps for trajectory b of the batch, run by a CTA of at least D
// warps; smem holds recur_smem_doubles<D, TPL, LAG>() doubles.  The far part G
// covers the points k < (c - LAG) L; the LAG blocks before block c are summed
// here.
template <class Rhs, int D, int TPL, int LAG = 1>
__device__ void recur_block(const DevBatch &bt, int b, const DevWeights &w, const StepConsts &kc,
                            int64_t c, const double *G, double *smem)
{
    constexpr int L = kWarp * TPL;
    // weights pre-multiplied by h^alpha: in the steps the accumulators hold y0 +
    // h^alpha * sum, so adding the newest point to the owner's accumulator yields y^P
    // directly
    constexpr int W = (LAG + 1) * L + 1;  // distances 0 .. (LAG+1) L
    double *sB = smem;                   // [D][W], per component (its own order)
    double *sA = sB + D * W;             // [D][W]
    double(*sy)[D] = reinterpret_cast<double(*)[D]>(sA + D * W);  // [2][D]
    double(*sF)[D] = sy + 2;             // [LAG L + 1][D]: f of the lag blocks and f_{m0}
    // component of this warp; warps beyond D (a CTA sized for a larger
    // dimension) mirror component 0 and write nothing
    const bool act = threadIdx.x / kWarp < D;
    const int i = act ? threadIdx.x / kWarp : 0;
    const int lane = threadIdx.x % kWarp;
    const int64_t Nb = bt.N_each[b];
    const int64_t m0 = c * L;  // f_{m0} is the newest known point
    if (m0 >= Nb) return;      // trajectory finished (uniform over the CTA)
    const int nW = w.stride ? D : 1;  // one weight set per order
    for (int j = threadIdx.x; j < nW * W; j += blockDim.x) {
        const int q = j / W, jj = j % W;
        const double hq = pick<D>(kc.h_alpha, q);
        sB[j] = hq * w.B[q * w.stride + jj];
        sA[j] = hq * w.A[q * w.stride + jj];
    }
    // rows m0-LAG*L .. m0 of this trajectory's history, all loads in flight at once
    for (int j = threadIdx.x; j < (LAG * L + 1) * D; j += blockDim.x) {
        const int64_t row = m0 - LAG * L + j / D;
        sF[j / D][j % D] = row >= 0 ? bt.F[row * bt.ldF + (int64_t)b * D + j % D] : 0.0;
    }
    __syncthreads();

    double p[kMaxParams];
#pragma unroll
    for (int q = 0; q < kMaxParams; ++q) p[q] = bt.params[(int64_t)b * kMaxParams + q];
    const double y0 = bt.y0[(int64_t)b * D + i];
    const int64_t col = (int64_t)b * D + i;
    const double ha = pick<D>(kc.h_alpha, i);
    const double ha_ig2 = ha * pick<D>(kc.inv_gamma2, i);
    const double *wD = w.D + i * w.stride;
    if (w.stride) sB += i * W, sA += i * W;  // this warp's component's order

    double accP[TPL], accC[TPL], baseP[TPL], baseC[TPL], aux[TPL];
    const double f0 = bt.F[col];
    const double y1 = bt.y1 ? bt.y1[col] : 0.0;
#pragma unroll
    for (int t = 0; t < TPL; ++t) {
        const int a = lane + kWarp * t;
        const int64_t m = m0 + 1 + a;
        aux[t] = Rhs::aux((double)m * kc.h, p);
        // Taylor part of the initial data at t_m: y0, or y0 + t_m y'(0) for 1 < alpha < 2
        const double Tm = bt.y1 ? fma((double)m * kc.h, y1, y0) : y0;
        const double gP = G ? G[(int64_t)a * bt.cols + col] : 0.0;
        const double gC = fma(wD[m], f0, G ? G[(int64_t)(L + a) * bt.cols + col] : 0.0);
        baseP[t] = fma(ha, gP, Tm);
        baseC[t] = fma(ha, gC, Tm);
        accP[t] = accC[t] = 0.0;
    }
    if (c >= 1) {  // lag blocks: k = m0-LAG*L+j, d = m-k = LAG*L+1+a-j in [2, (LAG+1)L]
        for (int j = 0; j < LAG * L; ++j) {
            const double fk = sF[j][i];
#pragma unroll
            for (int t = 0; t < TPL; ++t) {
                const int d = LAG * L + 1 + lane + kWarp * t - j;
                accP[t] = fma(sB[d], fk, accP[t]);
                accC[t] = fma(sA[d], fk, accC[t]);
            }
        }
    }
    // the lag blocks' sum is added to the base as a whole: one by one, each of its
    // points would be rounded to a unit of the base's last place (2-norm error against
    // binary128: scalar, 60 steps 2.9e-16 .. 3.5e-16, now 2.1e-16 .. 2.5e-16; 2000 steps
    // 4.3e-16 .. 4.8e-16, now 3.2e-16 .. 3.8e-16)
#pragma unroll
    for (int t = 0; t < TPL; ++t) accP[t] += baseP[t], accC[t] += baseC[t];

    double fk = sF[LAG * L][i];
    const int steps = (int)(Nb - m0 < L ? Nb - m0 : L);
    double *Yb = bt.Y + (int64_t)b * (bt.N + 1) * D;
    for (int s = 0; s < steps; ++s) {
        // add the newest point k = m0+s; for the owner of target k+1 this
        // completes y^P (accP) and y0 + h^a S^C (accC)
#pragma unroll
        for (int t = 0; t < TPL; ++t) {
            const int d = lane + kWarp * t - s + 1;
            const int dd = d > 0 ? d : 0;  // done targets add B(0) = A(0) = 0
            accP[t] = fma(sB[dd], fk, accP[t]);
            accC[t] = fma(sA[dd], fk, accC[t]);
        }
        const int owner = s % kWarp, slot = s / kWarp;  // uniform over the CTA
        double yp = 0.0, aC = 0.0, ax = 0.0;
#pragma unroll
        for (int t = 0; t < TPL; ++t)
            if (t == slot) yp = accP[t], aC = accC[t], ax = aux[t];
        double fn = 0.0, yc = 0.0;
        if constexpr (D == 1) {
            if (lane == owner) {
                const double fp = rhs_f64<Rhs, D>(0, &yp, p, ax);
                yc = fma(ha_ig2, fp, aC);
                fn = rhs_f64<Rhs, D>(0, &yc, p, ax);
            }
        } else {
            if (act && lane == owner) sy[0][i] = yp;
            __syncthreads();
            if (lane == owner) {
                double y[D];
#pragma unroll
                for (int q = 0; q < D; ++q) y[q] = sy[0][q];
                const double fp = rhs_f64<Rhs, D>(i, y, p, ax);
                yc = fma(ha_ig2, fp, aC);  // corrector
                if (act) sy[1][i] = yc;
            }
            __syncthreads();
            if (lane == owner) {
                double y[D];
#pragma unroll
                for (int q = 0; q < D; ++q) y[q] = sy[1][q];
                fn = rhs_f64<Rhs, D>(i, y, p, ax);
            }
        }
        if (act && lane == owner) {
            const int64_t mm = m0 + 1 + s;
            Yb[mm * D + i] = yc;
            bt.F[mm * bt.ldF + col] = fn;
            if (!(finite_bits(yc) && finite_bits(fn))) report_nonfinite(bt.status, mm, b);
        }
        fk = __shfl_sync(0xffffffffu, fn, owner);
    }
}

// ---- split precision ----
//
// The same block of steps for the split path with no FP64 operation on the
// serial chain of a step.  Per target (lane a):
//   base    y0 + h^alpha (far part + D(m) f_0), FP64, at block start;
//   near    the lag blocks and the in-block points, h^alpha w(d) f_k summed in
//           float-float (ff.cuh, ~48 bits) as the points become known;
//   step    y^P = base_P + near_P,  inc = near_C + h^alpha/Gamma(alpha+2) f(t, y^P),
//           then f(t, base_C + inc), all in float-float; the owner of the target
//           keeps inc and f;
//   end     y = base_C + inc (the FP64 corrector update) and f_k are written
//           as doubles, one target per lane, for the whole block at once.
// Float-float carries ~48 bits, so the recurrence adds rounding far below
// that of the split history; GB300 issues its fp32 at 64 times the FP64 rate
// and a float-float operation completes in fewer cycles than one FP64
// operation, so the chain is shorter and wide batches no longer saturate the
// FP64 pipe.
//
// What bounds it: the latency of a step's operations (~450 cycles for the
// Lorenz type).  Every lane runs the step on values that the owner puts into
// shared memory, so f ends up in all of them without another shuffle and no lane
// diverges; a component's code is compiled for it, so a warp converts and
// branches on nothing it does not use; the forcing is evaluated by a warp of its
// own beside the lag blocks; all global loads of a block are issued together.
// Whole solves: Lorenz type 2^16 35.7 -> 25.8 ms (of that 5 ms from SMs of its own,
// history_fp32c.cu), scalar 10^4 3.43 -> 2.92, oscillator 20 x 2^13 5.8 -> 4.0.
template <int D, int LAG = 1>
__host__ __device__ constexpr int recur_split_smem_floats()
{
    return 4 * ((LAG + 1) * kWarp + 1) * D + 8 * D + 2 * (LAG * kWarp + 1) * D + 2 * kWarp;
}
// Warps of a CTA for recur_block_split: one per component, and one for the forcing.
template <class Rhs, int D>
constexpr int recur_split_warps()
{
    return D + (Rhs::kForcing ? 1 : 0);
}

template <int D, int LAG>
struct SplitMem {
    static constexpr int L = kWarp, W = (LAG + 1) * L + 1;  // distances 0 .. (LAG+1) L
    FF *sB, *sA;      // [D or 1][W]  h^alpha_i B_i(d), A_i(d)
    FF (*sy)[2 * D];  // [2 parities][predictor, corrector][D]
    FF (*sF)[D];      // [LAG L + 1][D]: f of the lag blocks and f_{m0}
    FF *aux;          // [L] forcing
    __device__ explicit SplitMem(float *smem)
    {
        sB = reinterpret_cast<FF *>(smem);
        sA = sB + D * W;
        sy = reinterpret_cast<FF(*)[2 * D]>(sA + D * W);
        sF = reinterpret_cast<FF(*)[D]>(sy + 2);
        aux = reinterpret_cast<FF *>(sF + LAG * L + 1);
    }
};

// What a component's warp reads from global memory, loaded before anything waits.
struct SplitIn {
    double p[kMaxParams], y0, y1, f0, wD, gP, gC;
};

// Component I's part, by one warp; barrier 1 joins the D component warps.
template <class Rhs, int D, int LAG, int I>
__device__ __forceinline__ void split_steps(const DevBatch &bt, int b, const DevWeights &w,
                                            const StepConsts &kc, int64_t c, int64_t Nb,
                                            const SplitIn &in0, const SplitMem<D, LAG> &m)
{
    constexpr int L = kWarp;
    const int lane = threadIdx.x % kWarp;
    const int64_t m0 = c * L, mt = m0 + 1 + lane;
    const FF *sB = m.sB + (w.stride ? I * m.W : 0), *sA = m.sA + (w.stride ? I * m.W : 0);
    FF pf[kMaxParams];
#pragma unroll
    for (int q = 0; q < kMaxParams; ++q) pf[q] = ff_from_double(in0.p[q]);
    const int64_t col = (int64_t)b * D + I;
    const double ha = kc.h_alpha[I];
    const FF ha_ig2 = ff_from_double(ha * kc.inv_gamma2[I]);
    const double Tm = bt.y1 ? fma((double)mt * kc.h, in0.y1, in0.y0) : in0.y0;  // Taylor part at t_m
    const double gP = in0.gP, gC = fma(in0.wD, in0.f0, in0.gC);
    const double baseC = fma(ha, gC, Tm);
    const FF bP = ff_from_double(fma(ha, gP, Tm)), bC = ff_from_double(baseC);
    FF nP(0), nC(0), inc(0), fo(0);
    if (c >= 1) {  // lag blocks: k = m0-LAG*L+j, d = LAG*L+1+a-j in [2, (LAG+1)L]
#pragma unroll 8
        for (int j = 0; j < LAG * L; ++j) {
            const FF fk = m.sF[j][I];
            const int d = LAG * L + 1 + lane - j;
            nP = ff_fma(sB[d], fk, nP);
            nC = ff_fma(sA[d], fk, nC);
        }
    }
    FF ax(0);
    if constexpr (Rhs::kForcing) {
        asm volatile("bar.sync 2, %0;" ::"r"((D + 1) * kWarp) : "memory");
        ax = m.aux[lane];
    } else {
        ax = ff_from_double(Rhs::aux((double)mt * kc.h, in0.p));
    }

    FF fk = m.sF[LAG * L][I];
    const int steps = (int)(Nb - m0 < L ? Nb - m0 : L);
    FF wB = sB[lane + 1], wA = sA[lane + 1];
    for (int s = 0; s < steps; ++s) {
        // the newest point k = m0+s; done targets add B(0) = A(0) = 0
        nP = ff_fma(wB, fk, nP);
        nC = ff_fma(wA, fk, nC);
        const int d = lane - s > 0 ? lane - s : 0;
        wB = sB[d], wA = sA[d];
        const FF yp = bP + nP;
        FF y[D];
        volatile float *sy = reinterpret_cast<volatile float *>(m.sy[s & 1]);
        if constexpr (D > 1) {
            if (lane == s) sy[2 * I] = yp.hi, sy[2 * I + 1] = yp.lo;
            asm volatile("bar.sync 1, %0;" ::"r"(D * kWarp) : "memory");
#pragma unroll
            for (int q = 0; q < D; ++q) y[q] = FF(sy[2 * q], sy[2 * q + 1]);
        } else {
            y[0] = shfl_ff(yp, s);
        }
        const FF nc = shfl_ff(nC, s), bc = shfl_ff(bC, s);
        const FF axs = Rhs::kForcing ? shfl_ff(ax, s) : ax;
        const FF fp = Rhs::template one<D>(I, y, pf, axs);
        const FF in = ha_ig2 * fp + nc;  // corrector increment
        const FF yc = bc + in;
        if constexpr (D > 1) {
            if (lane == 0) sy[2 * D + 2 * I] = yc.hi, sy[2 * D + 2 * I + 1] = yc.lo;
            asm volatile("bar.sync 1, %0;" ::"r"(D * kWarp) : "memory");
#pragma unroll
            for (int q = 0; q < D; ++q) y[q] = FF(sy[2 * D + 2 * q], sy[2 * D + 2 * q + 1]);
        } else {
            y[0] = yc;
        }
        fk = Rhs::template one<D>(I, y, pf, axs);
        if (lane == s) inc = in, fo = fk;
    }

    // FP64 corrector update and f of the block's targets, one per lane
    if (lane < steps) {
        const double yc = baseC + ff_to_double(inc);
        const double fd = ff_to_double(fo);
        bt.Y[((int64_t)b * (bt.N + 1) + mt) * D + I] = yc;
        bt.F[mt * bt.ldF + col] = fd;
        if (bt.Ff) bt.Ff[mt * bt.ldF + col] = (float)fd;  // the fp32 history's input
        if (!(finite_bits(yc) && finite_bits(fd))) report_nonfinite(bt.status, mt, b);
    }
}

// smem: recur_split_smem_floats<D, LAG>() floats, 16-byte aligned; LAG as for
// recur_block; a CTA of at least recur_split_warps<Rhs, D>() warps.
template <class Rhs, int D, int LAG = 1>
__device__ void recur_block_split(const DevBatch &bt, int b, const DevWeights &w,
                                  const StepConsts &kc, int64_t c, const double *G, float *smem)
{
    constexpr int L = kWarp;
    const SplitMem<D, LAG> m(smem);
    const int warp = threadIdx.x / kWarp, lane = threadIdx.x % kWarp;
    const int64_t m0 = c * L;
    // every load that does not depend on another one, in flight together
    const int64_t Nb = bt.N_each[b];
    const int nW = w.stride ? D : 1;  // one weight set per order
    const int tid = threadIdx.x, nthr = blockDim.x, nF = (LAG * L + 1) * D;
    auto weight_index = [&](int j) { return (int64_t)(j / m.W) * w.stride + j % m.W; };
    auto f_at = [&](int j) {
        const int64_t row = m0 - LAG * L + j / D;
        return row >= 0 ? bt.F[row * bt.ldF + (int64_t)b * D + j % D] : 0.0;
    };
    double wb[2] = {}, wa[2] = {}, f[2] = {};
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        const int j = tid + u * nthr;
        if (j < nW * m.W) wb[u] = w.B[weight_index(j)], wa[u] = w.A[weight_index(j)];
        if (j < nF) f[u] = f_at(j);
    }
    SplitIn in{};
    if (warp < D) {
        const int64_t col = (int64_t)b * D + warp;
#pragma unroll
        for (int q = 0; q < kMaxParams; ++q) in.p[q] = bt.params[(int64_t)b * kMaxParams + q];
        in.y0 = bt.y0[col];
        if (bt.y1) in.y1 = bt.y1[col];
        in.f0 = bt.F[col];
        in.wD = w.D[warp * w.stride + m0 + 1 + lane];
        if (G) in.gP = G[(int64_t)lane * bt.cols + col], in.gC = G[(int64_t)(L + lane) * bt.cols + col];
    }
    if (m0 >= Nb) return;
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        const int j = tid + u * nthr;
        if (j < nW * m.W) {
            const double hq = pick<D>(kc.h_alpha, j / m.W);
            m.sB[j] = ff_from_double(hq * wb[u]);
            m.sA[j] = ff_from_double(hq * wa[u]);
        }
        if (j < nF) m.sF[j / D][j % D] = ff_from_double(f[u]);
    }
    for (int j = tid + 2 * nthr; j < nW * m.W; j += nthr) {  // several orders
        const double hq = pick<D>(kc.h_alpha, j / m.W);
        m.sB[j] = ff_from_double(hq * w.B[weight_index(j)]);
        m.sA[j] = ff_from_double(hq * w.A[weight_index(j)]);
    }
    for (int j = tid + 2 * nthr; j < nF; j += nthr) m.sF[j / D][j % D] = ff_from_double(f_at(j));
    __syncthreads();
    if (warp < D) {
        if (D == 1 || warp == 0) split_steps<Rhs, D, LAG, 0>(bt, b, w, kc, c, Nb, in, m);
        else if (D == 2 || warp == 1) split_steps<Rhs, D, LAG, D >= 2 ? 1 : 0>(bt, b, w, kc, c, Nb, in, m);
        else if (D == 3 || warp == 2) split_steps<Rhs, D, LAG, D >= 3 ? 2 : 0>(bt, b, w, kc, c, Nb, in, m);
        else split_steps<Rhs, D, LAG, D >= 4 ? 3 : 0>(bt, b, w, kc, c, Nb, in, m);
    } else if (Rhs::kForcing && warp == D) {
        double p[kMaxParams];
#pragma unroll
        for (int q = 0; q < kMaxParams; ++q) p[q] = bt.params[(int64_t)b * kMaxParams + q];
        m.aux[lane] = ff_from_double(Rhs::aux((double)(m0 + 1 + lane) * kc.h, p));
        asm volatile("bar.sync 2, %0;" ::"r"((D + 1) * kWarp) : "memory");
    }
}

}  // namespace fabm
