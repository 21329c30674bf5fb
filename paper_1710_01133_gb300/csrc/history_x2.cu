// a2 + a3 in double-double (FP64X2 precision): the far part of the hereditary
// sums of Sec. 2 of arXiv:1710.01133, as hist_fp64_kernel computes it, with
// the weights as double-double pairs (wh + wl) and every product and sum kept
// to about twice double precision.  This is the mode the paper keeps for precise
// runs (long double), not the fast one.
//
// What bounds it: the FP64 unit, which takes a warp instruction in 64 cycles per
// SM sub-partition whatever it is, so the number of FP64 instructions per weight
// and point is the time.  A running sum that starts at a power of two M, at least
// four times the sum of all |w f| that it takes, stays within a quarter of M, so
// every partial sum is a multiple of the same unit u = M 2^-53 and differences of
// them are exact (the pre-rounding of Ogita, Rump and Oishi's AccSum):
//   q' = fma(wh, f, q)        q' - q is w f rounded to a multiple of u
//   t  = q' - q               exact
//   lo += fma(wh, f, -t)      what the rounding left, itself below u
//   lo  = fma(wl, f, lo)      the weight's low part
// Five instructions instead of the eleven of a product with its error and Dot2
// (two for the product, six for the sum's rounding error, three for the low
// parts).  M comes from the exponents of the largest f and the largest weight of
// the points (integer instructions while they are staged), so it exceeds the sum
// of |w f| by 4 to 32 times the ratio of the largest |w f| to the mean one; what is
// lost is a few 2^-106 M, far below the rounding to double at the end.  Whole
// solves against the scheme in binary128 (nine systems and orders): largest error
// 4.4e-16 .. 9.0e-16 of the scale, 7.8e-16 .. 1.4e-15 with Dot2 and the steps that
// went with it.
// Chunk partials are pairs (hi, lo), combined in a fixed order and rounded once.
//
// A CTA takes up to four columns and a chunk of points, a quarter for each of its
// four warps (one per sub-partition), so that a weight read from shared memory
// serves all columns and no warp idles for want of a column.  Lorenz type, history
// of one block at k = 16000, cold caches: 81 -> 36 us (30 FP64 instructions per point
// and 32 targets: 26 us); sum of the chunks 39 -> 6.6 us.  Whole solve of 2^14 steps
// 40.4 -> 12.3 ms, 256 x 2^12 254 -> 121.
#include "fabm_internal.cuh"

namespace fabm {
namespace {

constexpr int kCols = 4;    // columns per CTA
constexpr int kWarps = 4;   // parts of a chunk, one per warp
constexpr int kL = kRecurL;
constexpr int kTile = 256;  // points staged in shared memory at a time
constexpr int kWin = kTile + kL;

// exponent field of a double from its high word
__device__ __forceinline__ int exp_field(unsigned hi) { return (int)(hi >> 20); }
__device__ __forceinline__ unsigned abs_hi(double x) { return (unsigned)__double2hiint(x) & 0x7fffffffu; }

// The power of two with exponent field e, kept finite and away from subnormals.
// Where the rule asks for a field beyond kTopField, terms scaled down by kScaleBits
// are added instead, so that sums up to the end of the range stay finite and exact.
constexpr int kTopField = 2046;
constexpr int kScaleBits = 64;
constexpr double kScaleDown = 0x1p-64, kScaleUp = 0x1p64;
__device__ __forceinline__ double pow2_field(int e)
{
    e = e < 64 ? 64 : (e > 2046 ? 2046 : e);
    return __hiloint2double(e << 20, 0);
}

// (hi, lo) += x with the rounding error of hi + x (TwoSum)
__device__ __forceinline__ void two_sum(double &hi, double &lo, double x)
{
    const double s = hi + x;
    const double z = s - hi;
    lo += (hi - (s - z)) + (x - z);
    hi = s;
}

// A warp's points j0 .. j1-1 of the staged tile for NC columns: wnd0 is lane a's
// weight of point 0, point j's is wnd0[-j].  sum[q][kind] starts at M[q].
template <int NC, bool MULTI>
__device__ __forceinline__ void add_points(const double *sF, const double *wBh, const double *wBl,
                                           const double *wAh, const double *wAl, int j0, int j1,
                                           double (&sum)[kCols][2], double (&lo)[kCols][2])
{
#pragma unroll 2
    for (int j = j0; j < j1; ++j) {
        double bh = wBh[-j], bl = wBl[-j], ah = wAh[-j], al = wAl[-j];
#pragma unroll
        for (int q = 0; q < NC; ++q) {
            if (MULTI && q) {
                bh = wBh[q * kWin - j], bl = wBl[q * kWin - j];
                ah = wAh[q * kWin - j], al = wAl[q * kWin - j];
            }
            const double f = sF[j * kCols + q];
            const double nb = fma(bh, f, sum[q][0]), na = fma(ah, f, sum[q][1]);
            const double tb = nb - sum[q][0], ta = na - sum[q][1];
            sum[q][0] = nb, sum[q][1] = na;
            lo[q][0] += fma(bh, f, -tb);
            lo[q][1] += fma(ah, f, -ta);
            lo[q][0] = fma(bl, f, lo[q][0]);
            lo[q][1] = fma(al, f, lo[q][1]);
        }
    }
}

struct Tiles {
    double f[kTile * kCols];
    double bh[kCols][kWin], bl[kCols][kWin], ah[kCols][kWin], al[kCols][kWin];
};
struct Sums {
    double2 part[kWarps][kCols][2][kWarp];
};
union Smem {
    Tiles t;
    Sums s;
};

// The sums of hist_x2_kernel's chunk k0 .. k1-1 where values are so large (|f| from
// about 2^1005 on) that M would pass the end of the range: one thread per sum, terms
// scaled down, products with their errors and TwoSum.  Out of line, as the test costs
// a solve of ordinary values under 1 % this way and 2 to 5 % with the scaling inside the
// kernel's loop.
template <bool MULTI>
__device__ __noinline__ void top_chunk(const double *F, int64_t ldF, int cols, const double *WBh,
                                       const double *WBl, const double *WAh, const double *WAl,
                                       int64_t c, int64_t k0, int64_t k1, double2 *part,
                                       int64_t wstride, int dim, double *G)
{
    const int col0 = blockIdx.y * kCols, ncol = min(kCols, cols - col0);
    for (int o = threadIdx.x; o < ncol * 2 * kWarp; o += kWarp * kWarps) {
        const int q = o / (2 * kWarp), kind = o / kWarp % 2, t = o % kWarp;
        const int64_t col = col0 + q, wo = (MULTI ? col % dim * wstride : 0) + c * kL + 1 + t;
        const double *wh = (kind ? WAh : WBh) + wo, *wl = (kind ? WAl : WBl) + wo;
        unsigned mx = 0;
        for (int64_t k = k0; k < k1; ++k) mx = max(mx, abs_hi(F[k * ldF + col]));
        const bool down = exp_field(mx) > 1023;
        double hi = 0.0, lo = 0.0;
        for (int64_t k = k0; k < k1; ++k) {
            const double f = F[k * ldF + col] * (down ? kScaleDown : 1.0), p = wh[-k] * f;
            const double e = fma(wh[-k], f, -p);
            two_sum(hi, lo, p);
            lo += e;
            lo = fma(wl[-k], f, lo);
        }
        if (down) hi *= kScaleUp, lo *= kScaleUp;
        const int64_t out = (kind * kL + t) * (int64_t)cols + col;
        if (G)
            G[out] = hi + lo;
        else
            part[(int64_t)blockIdx.x * 2 * kL * cols + out] = make_double2(hi, lo);
    }
}

// grid = (n_chunks, ceil(cols / 4)); block = 128.  Chunk `chunk` covers the
// points [chunk*kc, min((chunk+1)*kc, k_end)) of target block c (targets
// m = cL+1+a, lane a); part[chunk][kind][a][col] = (hi, lo), or with one chunk, if
// G is given, G[kind][a][col] = hi + lo (wide batches; the sum of the chunks as a
// launch of its own took a third as long again: scalar, 16,384 x 100 steps,
// 2.28 -> 2.14 ms).  MULTI: one order
// per component (column col's weights at offset (col % dim) * wstride).
template <bool MULTI>
__global__ void __launch_bounds__(kWarp *kWarps)
    hist_x2_kernel(const double *__restrict__ F, int64_t ldF, int cols, const double *__restrict__ WBh,
                   const double *__restrict__ WBl, const double *__restrict__ WAh,
                   const double *__restrict__ WAl, int64_t c, int64_t kc, int64_t k_end,
                   double2 *__restrict__ part, int64_t wstride, int dim, double *__restrict__ G)
{
    __shared__ Smem sm;
    __shared__ unsigned max_f[2][kCols], max_w[2][kCols];  // high words, by parity of the tile
    const int64_t chunk = blockIdx.x;
    const int col0 = blockIdx.y * kCols;
    const int64_t k0 = chunk * kc;
    const int64_t k1 = k0 + kc < k_end ? k0 + kc : k_end;
    const int ncol = min(kCols, cols - col0);
    const int w = threadIdx.x / kWarp;
    const int a = threadIdx.x % kWarp;
    const bool one_tile = k1 - k0 <= kTile;
    double hi[kCols][2], lo[kCols][2];
#pragma unroll
    for (int q = 0; q < kCols; ++q) hi[q][0] = hi[q][1] = lo[q][0] = lo[q][1] = 0.0;
    if (threadIdx.x < 2 * kCols) {
        max_f[threadIdx.x / kCols][threadIdx.x % kCols] = 0u;
        max_w[threadIdx.x / kCols][threadIdx.x % kCols] = 0u;
    }
    __syncthreads();

    int par = 0;
    for (int64_t t0 = k0; t0 < k1; t0 += kTile, par ^= 1) {
        const int64_t t1 = t0 + kTile < k1 ? t0 + kTile : k1;
        const int nk = (int)(t1 - t0);
        // window index i <-> d = cL+2-t1 + i, i < nk+L-1 (as hist_fp64_block)
        const int64_t d_min = c * kL + 2 - t1;
        const int nwin = nk + kL - 1;
        for (int v = 0; v < (MULTI ? ncol : 1); ++v) {
            const int64_t o = (MULTI ? (int64_t)((col0 + v) % dim) * wstride : 0) + d_min;
            unsigned mw = 0;
            for (int i = threadIdx.x; i < nwin; i += kWarp * kWarps) {
                const double bh = WBh[o + i], ah = WAh[o + i];
                sm.t.bh[v][i] = bh;
                sm.t.ah[v][i] = ah;
                sm.t.bl[v][i] = WBl[o + i];
                sm.t.al[v][i] = WAl[o + i];
                mw = max(mw, max(abs_hi(bh), abs_hi(ah)));
            }
            mw = __reduce_max_sync(0xffffffffu, mw);
            if (a == 0) atomicMax(&max_w[par][v], mw);
        }
        unsigned mf = 0;  // this thread's column is threadIdx.x % kCols throughout
        for (int i = threadIdx.x; i < nk * kCols; i += kWarp * kWarps) {
            const int k = i / kCols, j = i % kCols;
            const double f = j < ncol ? F[(t0 + k) * ldF + col0 + j] : 0.0;
            sm.t.f[i] = f;
            mf = max(mf, abs_hi(f));
        }
#pragma unroll
        for (int off = kCols; off < kWarp; off <<= 1) mf = max(mf, __shfl_xor_sync(0xffffffffu, mf, off));
        if (a < kCols) atomicMax(&max_f[par][a], mf);
        __syncthreads();
        if (threadIdx.x < kCols) max_f[par ^ 1][threadIdx.x] = max_w[par ^ 1][threadIdx.x] = 0u;
        // |w f| < 2^(ef + ew - 2044) for exponent fields ef, ew; nk terms; times four
        const int lg = 32 - __clz(nk);
        double M[kCols], sum[kCols][2];
        bool top = false;
#pragma unroll
        for (int q = 0; q < kCols; ++q) {
            const int ef = exp_field(max_f[par][q]);
            const int e = ef + exp_field(max_w[par][MULTI ? q : 0]) - 1019 + lg;
            top = top || (e > kTopField && ef < 2047);  // infinities and NaNs stay what they are
            M[q] = pow2_field(e);
            sum[q][0] = sum[q][1] = M[q];
        }
        if (top) {  // in every thread, or in none
            top_chunk<MULTI>(F, ldF, cols, WBh, WBl, WAh, WAl, c, k0, k1, part, wstride, dim, G);
            return;
        }
        const int j0 = w * nk / kWarps, j1 = (w + 1) * nk / kWarps;
        const int base = a + nk - 1;  // d - d_min for point t0+j: a + nk-1-j
        const double *pbh = sm.t.bh[0] + base, *pbl = sm.t.bl[0] + base;
        const double *pah = sm.t.ah[0] + base, *pal = sm.t.al[0] + base;
        switch (ncol) {
        case 1: add_points<1, MULTI>(sm.t.f, pbh, pbl, pah, pal, j0, j1, sum, lo); break;
        case 2: add_points<2, MULTI>(sm.t.f, pbh, pbl, pah, pal, j0, j1, sum, lo); break;
        case 3: add_points<3, MULTI>(sm.t.f, pbh, pbl, pah, pal, j0, j1, sum, lo); break;
        default: add_points<4, MULTI>(sm.t.f, pbh, pbl, pah, pal, j0, j1, sum, lo); break;
        }
#pragma unroll
        for (int q = 0; q < kCols; ++q)
#pragma unroll
            for (int kind = 0; kind < 2; ++kind) {
                if (q >= ncol) continue;
                const double x = sum[q][kind] - M[q];  // exact
                if (one_tile)
                    hi[q][kind] = x;
                else
                    two_sum(hi[q][kind], lo[q][kind], x);
            }
        __syncthreads();
    }

#pragma unroll
    for (int q = 0; q < kCols; ++q)
#pragma unroll
        for (int kind = 0; kind < 2; ++kind)
            if (q < ncol) sm.s.part[w][q][kind][a] = make_double2(hi[q][kind], lo[q][kind]);
    __syncthreads();
    // the four warps' sums; of one tile they are multiples of the same unit with a
    // sum below M, so adding them is exact
    for (int o = threadIdx.x; o < ncol * 2 * kWarp; o += kWarp * kWarps) {
        const int q = o / (2 * kWarp), kind = o / kWarp % 2, t = o % kWarp;
        double2 s = sm.s.part[0][q][kind][t];
#pragma unroll
        for (int v = 1; v < kWarps; ++v) {
            const double2 x = sm.s.part[v][q][kind][t];
            if (one_tile)
                s.x += x.x;
            else
                two_sum(s.x, s.y, x.x);
            s.y += x.y;
        }
        if (G)  // the only chunk
            G[(kind * kL + t) * (int64_t)cols + col0 + q] = s.x + s.y;
        else
            part[((chunk * 2 + kind) * kL + t) * (int64_t)cols + col0 + q] = s;
    }
}

// a3: G[kind][a][col] = sum over chunks of (hi + lo), R lanes per output with the
// chunks r, r+R, ..., up to kBatch of a lane's added at a time by the same rule as
// above (M from the largest hi of the group's lanes), then the lanes; rounded once
// to double.  Every thread runs the same number of rounds, so the shuffles always
// see full warps.  Bound by latency (loads, then ~40 FP64 instructions).
constexpr int kBatch = 5;
template <int R>
__global__ void reduce_x2_kernel(const double2 *__restrict__ part, int n_chunks, int64_t n_out,
                                 double *__restrict__ G)
{
    const int64_t gtid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int r = (int)(gtid % R);
    const int64_t groups = (int64_t)gridDim.x * blockDim.x / R;
    const bool one = n_chunks <= R * kBatch;
    constexpr int lg = R == 32 ? 8 : (R == 8 ? 6 : 3);  // R * kBatch <= 2^lg
    for (int64_t base = 0; base < n_out; base += groups) {
        const int64_t o = base + gtid / R;
        double hi = 0, lo = 0;
        for (int c0 = 0; c0 < n_chunks; c0 += R * kBatch) {
            double2 v[kBatch];
            unsigned mx = 0;
#pragma unroll
            for (int u = 0; u < kBatch; ++u) {
                const int ch = c0 + u * R + r;
                v[u] = o < n_out && ch < n_chunks ? part[(int64_t)ch * n_out + o] : make_double2(0.0, 0.0);
                mx = max(mx, abs_hi(v[u].x));
            }
#pragma unroll
            for (int off = R / 2; off > 0; off >>= 1)
                mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, off));
            int e = exp_field(mx) + 3 + lg;
            const bool big = e > kTopField;  // the same in the output's lanes
            if (big) {
                e -= kScaleBits, lo *= kScaleDown;
#pragma unroll
                for (int u = 0; u < kBatch; ++u) v[u].x *= kScaleDown, v[u].y *= kScaleDown;
            }
            const double M = pow2_field(e);
            double s = M;
#pragma unroll
            for (int u = 0; u < kBatch; ++u) {
                const double n = s + v[u].x;
                lo += v[u].x - (n - s);
                lo += v[u].y;
                s = n;
            }
            double x = s - M;
            if (big) x *= kScaleUp, lo *= kScaleUp;
            if (one)
                hi = x;
            else
                two_sum(hi, lo, x);
        }
#pragma unroll
        for (int off = R / 2; off > 0; off >>= 1) {
            const double ohi = __shfl_xor_sync(0xffffffffu, hi, off);
            const double olo = __shfl_xor_sync(0xffffffffu, lo, off);
            if (one)
                hi += ohi;  // exact
            else
                two_sum(hi, lo, ohi);
            lo += olo;
        }
        if (r == 0 && o < n_out) G[o] = hi + lo;
    }
}

}  // namespace

cudaError_t launch_hist_x2(const DevBatch &bt, const DevWeights &w, const DevWeightsLo &wl,
                           int64_t c, int lag, int n_chunks, int64_t kc, bool alone, double2 *part,
                           double *G, cudaStream_t st)
{
    const int64_t k_end = (c - lag) * kL;
    if (lag < 1) return cudaErrorInvalidValue;
    if (k_end <= 0) return cudaSuccess;
    dim3 grid((unsigned)n_chunks, (unsigned)((bt.cols + kCols - 1) / kCols));
    auto run = [&](auto kernel, int64_t stride, int dim) -> cudaError_t {
        const size_t smem = alone ? kAloneSmem : 0;  // beside the static arrays
        if (alone) {
            const cudaError_t e =
                cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            if (e != cudaSuccess) return e;
        }
        kernel<<<grid, kWarp * kWarps, smem, st>>>(bt.F, bt.ldF, bt.cols, w.B, wl.B, w.A, wl.A, c, kc,
                                                   k_end, part, stride, dim, n_chunks == 1 ? G : nullptr);
        return cudaGetLastError();
    };
    return w.stride ? run(hist_x2_kernel<true>, w.stride, bt.dim) : run(hist_x2_kernel<false>, 0, 1);
}

cudaError_t launch_reduce_x2(const double2 *part, int n_chunks, int cols, double *G, cudaStream_t st)
{
    const int64_t n_out = 2LL * kL * cols;
    auto run = [&](auto kernel, int R) {
        // one warp per CTA while that leaves SMs idle: the sums are FP64 chains
        const int threads = n_out * R <= 152 * 4 * kWarp ? kWarp : 256;
        const int64_t b = (n_out * R + threads - 1) / threads;
        kernel<<<(unsigned)(b > 152 * 16 ? 152 * 16 : b), threads, 0, st>>>(part, n_chunks, n_out, G);
    };
    if (n_chunks >= 64)
        run(reduce_x2_kernel<32>, 32);
    else if (n_chunks >= 16)
        run(reduce_x2_kernel<8>, 8);
    else
        run(reduce_x2_kernel<1>, 1);
    return cudaGetLastError();
}

}  // namespace fabm
