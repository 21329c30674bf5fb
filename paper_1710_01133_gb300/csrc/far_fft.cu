// a2 in double for the far points: the hereditary sums of Sec. 2 of
// arXiv:1710.01133 over whole segments of n points, as circular convolutions
// of length M = 2n (the overlap method: for target superblock T and segment S
// with lag g = T - S >= 2, the sums over the points of S for all n targets of T
// are n entries of one circular convolution of f, padded with n zeros, with
// the 2n - 1 weights of the distances n(g-1)+2 .. n(g+1)).
//
// The transform of a segment is taken once and kept, so a superblock costs one
// forward transform of the segment that has just become far, T - 1 products
// of spectra, and one inverse transform, against 4 n^2 multiply-adds per segment
// for the direct sums: n / 2 times fewer FP64 instructions (GB300 retires two
// FP64 FMAs per clock and SM, so they are what the direct sums cost).
//
// The two weight kinds are one complex weight B + iA: f is real, so the real
// part of the convolution is the predictor's sum and the imaginary part the
// corrector's.  Columns are never packed together: the rounding error of a
// column's sums is relative to its own f, and a column that becomes non-finite
// leaves the others alone.
//
// A transform's rounding error is relative to the largest of its sums, so what
// is constant goes around it: w(ng+1), the middle weight of a lag's window, is
// taken off the window's weights, and the inverse kernel adds it times the sum
// of the segment's f (both with compensated additions).  The weights of a far
// window differ little (1 - alpha times 2/g relative), so what is left to the
// transforms, and their error, is a small part of the sums.  Error of whole
// solves against binary128 (2-norm, direct sums / these): scalar 0.8, 20,000
// steps 5.8e-16 / 5.3e-16 (8.4e-16 without the middle weights), scalar 1.5
// 4.8e-16 / 3.4e-16 (1.1e-15), Lorenz type 0.98, 11,000 steps 5.5e-16 / 3.8e-16
// (9.2e-16), LCR 4.0e-16 / 2.5e-16 (4.4e-16).
//
// In-place radix-4 transforms in shared memory, decimation in frequency
// forward and in time backward, so the spectra stay in digit-reversed order
// and nothing is reordered.  The weights carry the factor 1/M.
#include "recurrence.cuh"

namespace fabm {
namespace {

constexpr int kThreads = 256;

__device__ __forceinline__ double2 cmul(double2 a, double2 w)
{
    return make_double2(fma(a.x, w.x, -(a.y * w.y)), fma(a.x, w.y, a.y * w.x));
}
__device__ __forceinline__ double2 cmul_conj(double2 a, double2 w)  // a conj(w)
{
    return make_double2(fma(a.x, w.x, a.y * w.y), fma(a.y, w.x, -(a.x * w.y)));
}
__device__ __forceinline__ double2 operator+(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 operator-(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }

// tw[j] = exp(-2 pi i j / M)
__device__ void fft_forward(double2 *s, int M, const double2 *__restrict__ tw)
{
    int len = M;
    for (; len >= 4; len /= 4) {
        const int q = len / 4, stride = M / len;
        for (int t = threadIdx.x; t < M / 4; t += blockDim.x) {
            const int j = t % q;
            double2 *x = s + (t / q) * len + j;
            const double2 a0 = x[0], a1 = x[q], a2 = x[2 * q], a3 = x[3 * q];
            const double2 s02 = a0 + a2, d02 = a0 - a2, s13 = a1 + a3, d13 = a1 - a3;
            x[0] = s02 + s13;
            const double2 y1 = make_double2(d02.x + d13.y, d02.y - d13.x);  // d02 - i d13
            const double2 y2 = s02 - s13;
            const double2 y3 = make_double2(d02.x - d13.y, d02.y + d13.x);
            if (j == 0) {
                x[q] = y1, x[2 * q] = y2, x[3 * q] = y3;
            } else {
                x[q] = cmul(y1, tw[j * stride]);
                x[2 * q] = cmul(y2, tw[2 * j * stride]);
                x[3 * q] = cmul(y3, tw[3 * j * stride]);
            }
        }
        __syncthreads();
    }
    if (len == 2) {
        for (int t = threadIdx.x; t < M / 2; t += blockDim.x) {
            const double2 a0 = s[2 * t], a1 = s[2 * t + 1];
            s[2 * t] = a0 + a1, s[2 * t + 1] = a0 - a1;
        }
        __syncthreads();
    }
}

// The reverse of fft_forward with conjugate factors: M times its inverse.
__device__ void fft_backward(double2 *s, int M, const double2 *__restrict__ tw)
{
    int len = 4;
    if (__popc(M - 1) % 2) {  // log2 M odd: the radix-2 stage first
        for (int t = threadIdx.x; t < M / 2; t += blockDim.x) {
            const double2 a0 = s[2 * t], a1 = s[2 * t + 1];
            s[2 * t] = a0 + a1, s[2 * t + 1] = a0 - a1;
        }
        __syncthreads();
        len = 8;
    }
    for (; len <= M; len *= 4) {
        const int q = len / 4, stride = M / len;
        for (int t = threadIdx.x; t < M / 4; t += blockDim.x) {
            const int j = t % q;
            double2 *x = s + (t / q) * len + j;
            double2 b0 = x[0], b1 = x[q], b2 = x[2 * q], b3 = x[3 * q];
            if (j) {
                b1 = cmul_conj(b1, tw[j * stride]);
                b2 = cmul_conj(b2, tw[2 * j * stride]);
                b3 = cmul_conj(b3, tw[3 * j * stride]);
            }
            const double2 s02 = b0 + b2, d02 = b0 - b2, s13 = b1 + b3, d13 = b1 - b3;
            x[0] = s02 + s13;
            x[q] = make_double2(d02.x - d13.y, d02.y + d13.x);  // d02 + i d13
            x[2 * q] = s02 - s13;
            x[3 * q] = make_double2(d02.x + d13.y, d02.y - d13.x);
        }
        __syncthreads();
    }
}

__global__ void twiddle_kernel(int M, double2 *tw)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= M) return;
    double s, c;
    sincospi(2.0 * (double)j / (double)M, &s, &c);
    tw[j] = make_double2(c, -s);
}

// What[set][g] for the lags g = 2 + blockIdx.x: v[u] = w(ng+1+u) - w(ng+1), u < n,
// and v[M-u] = w(ng+1-u) - w(ng+1), 0 < u < n, w = (B + iA) / M.  blockIdx.y:
// weight set.
__global__ void __launch_bounds__(kThreads)
    weight_spectra_kernel(const double *__restrict__ WB, const double *__restrict__ WA,
                          int64_t wstride, int n, int g_max, const double2 *__restrict__ tw,
                          double2 *__restrict__ What)
{
    extern __shared__ double2 s[];
    const int M = 2 * n;
    const int64_t g = 2 + blockIdx.x;
    const double *B = WB + blockIdx.y * wstride, *A = WA + blockIdx.y * wstride;
    const double inv = 1.0 / (double)M, Bg = B[n * g + 1], Ag = A[n * g + 1];
    for (int u = threadIdx.x; u < M; u += blockDim.x) {
        const int64_t d = n * g + 1 + (u < n ? u : u - M);
        s[u] = u == n ? make_double2(0.0, 0.0) : make_double2((B[d] - Bg) * inv, (A[d] - Ag) * inv);
    }
    __syncthreads();
    fft_forward(s, M, tw);
    double2 *out = What + ((int64_t)blockIdx.y * (g_max + 1) + g) * M;
    for (int u = threadIdx.x; u < M; u += blockDim.x) out[u] = s[u];
}

// A value of f above 2^900 would leave the transform no room: such a segment is
// stored times 2^-200 and marked; big[S][col] = 1 if a segment up to S is marked.
constexpr double kDown = 0x1p-200;
constexpr int kBigHi = (1023 + 900) << 20;  // high word of 2^900

// (s, c) += v, the rounding error of the addition kept in c (TwoSum).
__device__ __forceinline__ void comp_add(double &s, double &c, double v)
{
    const double t = s + v, bv = t - s;
    c += (s - (t - bv)) + (v - bv);
    s = t;
}
// For superblock T, C columns per CTA (a power of two), 256 / C threads each:
// the sum of segment T-2 of every column (fsum, mark, big), then
// mid[kind][col] = sum over the segments S <= T-2 of w(n(T-S)+1) fsum[S], sum and
// error term.  All lanes at work until the trees; with a warp per column inside the transforms'
// kernels an LCR sweep of 256 x 2^13 took 9.0 instead of 8.5 ms.
__global__ void __launch_bounds__(kThreads)
    middle_sums_kernel(const double *__restrict__ F, int64_t ldF, int cols, int n, int64_t T,
                       const double *__restrict__ WB, const double *__restrict__ WA,
                       int64_t wstride, int dim, int C, double *fsum, unsigned char *mark,
                       unsigned char *big, double2 *__restrict__ mid)
{
    __shared__ double2 red[2][kThreads];
    __shared__ int over[kThreads];
    const int c = threadIdx.x % C, r = threadIdx.x / C, R = kThreads / C;
    const int col = blockIdx.x * C + c;
    const bool act = col < cols;
    const int64_t S = T - 2;
    auto tree = [&](int kinds) {  // over the R threads of a column, in a fixed order
        for (int off = R / 2; off > 0; off >>= 1) {
            __syncthreads();
            if (r < off)
                for (int k = 0; k < kinds; ++k) {
                    double2 x = red[k][threadIdx.x];
                    const double2 y = red[k][threadIdx.x + off * C];
                    comp_add(x.x, x.y, y.x);
                    x.y += y.y;
                    red[k][threadIdx.x] = x;
                }
        }
        __syncthreads();
    };
    if (r == 0) over[c] = 0;
    __syncthreads();
    auto column_sum = [&](double sc) {  // true if a value is of at least 2^900
        double t = 0.0, e = 0.0;
        bool ov = false;
        for (int j = r; act && j < n; j += R) {
            double f = F[(S * n + j) * ldF + col];
            ov = ov || (__double2hiint(f) & 0x7fffffff) >= kBigHi;
            if (sc != 1.0) f *= sc;
            comp_add(t, e, f);
        }
        red[0][threadIdx.x] = make_double2(t, e);
        return ov;
    };
    if (column_sum(1.0)) over[c] = 1;
    __syncthreads();
    if (over[c]) column_sum(kDown);
    tree(1);
    if (r == 0 && act) {
        fsum[S * cols + col] = red[0][c].x + red[0][c].y;
        mark[S * cols + col] = over[c] != 0;
        big[S * cols + col] = over[c] || (S > 0 && big[(S - 1) * cols + col]);
    }
    __syncthreads();
    double t[2] = {0.0, 0.0}, e[2] = {0.0, 0.0};
    if (act) {
        const bool scaled = big[S * cols + col];
        const double *W[2] = {WB + (col % dim) * wstride, WA + (col % dim) * wstride};
        for (int64_t q = r; q <= S; q += R) {
            double f = fsum[q * cols + col];
            if (scaled && !mark[q * cols + col]) f *= kDown;
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const double w = W[k][n * (T - q) + 1], v = w * f;
                e[k] += fma(w, f, -v);
                comp_add(t[k], e[k], v);
            }
        }
    }
    red[0][threadIdx.x] = make_double2(t[0], e[0]);
    red[1][threadIdx.x] = make_double2(t[1], e[1]);
    tree(2);
    if (r == 0 && act) mid[col] = red[0][c], mid[cols + col] = red[1][c];
}

// Spectrum of segment S (points nS .. nS+n-1) of column blockIdx.x.
__global__ void __launch_bounds__(kThreads)
    segment_spectrum_kernel(const double *__restrict__ F, int64_t ldF, int cols, int64_t rows, int n,
                            int64_t S, const double2 *__restrict__ tw,
                            const unsigned char *__restrict__ mark, double2 *__restrict__ Fhat)
{
    extern __shared__ double2 s[];
    const int M = 2 * n, col = blockIdx.x;
    const double sc = mark[S * cols + col] ? kDown : 1.0;
    for (int j = threadIdx.x; j < n; j += blockDim.x) {
        const int64_t k = S * n + j;
        s[j] = make_double2(k < rows ? F[k * ldF + col] * sc : 0.0, 0.0);
        s[j + n] = make_double2(0.0, 0.0);
    }
    __syncthreads();
    fft_forward(s, M, tw);
    double2 *out = Fhat + (S * cols + col) * M;
    for (int u = threadIdx.x; u < M; u += blockDim.x) out[u] = s[u];
}

// acc[chunk][col][u] = sum over the segments S of the chunk of Fhat[S] What[T-S];
// segments 0 .. T-2.  grid = (M / blockDim, chunks, cols).
__global__ void product_kernel(const double2 *__restrict__ Fhat, const double2 *__restrict__ What,
                               const unsigned char *__restrict__ mark,
                               const unsigned char *__restrict__ big, int cols, int dim, bool multi,
                               int M, int g_max, int64_t T, double2 *__restrict__ acc)
{
    const int u = blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t col = blockIdx.z, nseg = T - 1;
    const int64_t s0 = nseg * blockIdx.y / gridDim.y, s1 = nseg * (blockIdx.y + 1) / gridDim.y;
    const double2 *W = What + (multi ? (col % dim) * (int64_t)(g_max + 1) * M : 0) + u;
    const double2 *f = Fhat + col * M + u;
    const int64_t fs = (int64_t)cols * M;
    double2 r = make_double2(0.0, 0.0);
    if (!big[(T - 2) * cols + col]) {
#pragma unroll 4
        for (int64_t S = s0; S < s1; ++S) {
            const double2 x = f[S * fs], w = W[(T - S) * M];
            r.x = fma(x.x, w.x, r.x), r.y = fma(x.x, w.y, r.y);
            r.x = fma(-x.y, w.y, r.x), r.y = fma(x.y, w.x, r.y);
        }
    } else {
        for (int64_t S = s0; S < s1; ++S) {
            const double sc = mark[S * cols + col] ? 1.0 : kDown;
            const double2 x = make_double2(f[S * fs].x * sc, f[S * fs].y * sc), w = W[(T - S) * M];
            r.x = fma(x.x, w.x, r.x), r.y = fma(x.x, w.y, r.y);
            r.x = fma(-x.y, w.y, r.x), r.y = fma(x.y, w.x, r.y);
        }
    }
    acc[(blockIdx.y * (int64_t)cols + col) * M + u] = r;
}

// G[kind][a][col], a < n: the sums of the chunks in order, transformed back,
// plus the middle weights times the segments' sums (mid).
__global__ void __launch_bounds__(kThreads)
    inverse_kernel(const double2 *__restrict__ acc, const double2 *__restrict__ mid,
                   const unsigned char *__restrict__ big, int chunks, int cols, int n, int64_t T,
                   const double2 *__restrict__ tw, double *__restrict__ G)
{
    extern __shared__ double2 s[];
    const int M = 2 * n, col = blockIdx.x;
    for (int u = threadIdx.x; u < M; u += blockDim.x) {
        double2 r = acc[(int64_t)col * M + u];
        for (int c = 1; c < chunks; ++c) r = r + acc[((int64_t)c * cols + col) * M + u];
        s[u] = r;
    }
    __syncthreads();
    fft_backward(s, M, tw);
    const double up = big[(T - 2) * cols + col] ? 1.0 / kDown : 1.0;
    const double2 mP = mid[col], mC = mid[cols + col];
    for (int j = threadIdx.x; j < n; j += blockDim.x) {
        G[(int64_t)j * cols + col] = (mP.x + (mP.y + s[j].x)) * up;
        G[(int64_t)(n + j) * cols + col] = (mC.x + (mC.y + s[j].y)) * up;
    }
}

int fft_threads(int M) { return M / 4 < kThreads ? M / 4 : kThreads; }

}  // namespace

cudaError_t launch_fft_weights(const DevWeights &w, int sets, int n, int g_max, double2 *tw,
                               double2 *What, cudaStream_t st)
{
    const int M = 2 * n;
    twiddle_kernel<<<(M + 127) / 128, 128, 0, st>>>(M, tw);
    if (g_max >= 2)
        weight_spectra_kernel<<<dim3((unsigned)(g_max - 1), (unsigned)sets), fft_threads(M),
                                sizeof(double2) * M, st>>>(w.B, w.A, w.stride, n, g_max, tw, What);
    return cudaGetLastError();
}

int fft_chunks(int n, int cols, int64_t T)
{
    // enough CTAs of 128 threads to fill the FP64 units (four warps per SM
    // already do), at least eight segments each
    const int64_t per = (int64_t)cols * (2 * n / 128);
    const int64_t want = (152 * 2 + per - 1) / per, most = (T - 1 + 7) / 8;
    const int64_t c = want < most ? want : most;
    return (int)(c < 1 ? 1 : (c > 16 ? 16 : c));
}

cudaError_t launch_fft_segment(const DevBatch &bt, const DevWeights &w, int n, int64_t T,
                               const double2 *tw, const FarWork &f, cudaStream_t st)
{
    const int M = 2 * n;
    int C = 1;
    while (C < 8 && C < bt.cols) C *= 2;
    middle_sums_kernel<<<(unsigned)((bt.cols + C - 1) / C), kThreads, 0, st>>>(
        bt.F, bt.ldF, bt.cols, n, T, w.B, w.A, w.stride, bt.dim, C, f.fsum, f.mark, f.big, f.mid);
    segment_spectrum_kernel<<<(unsigned)bt.cols, fft_threads(M), sizeof(double2) * M, st>>>(
        bt.F, bt.ldF, bt.cols, bt.N + 1, n, T - 2, tw, f.mark, f.Fhat);
    return cudaGetLastError();
}

cudaError_t launch_fft_far(const DevBatch &bt, bool multi, int n, int g_max, int64_t T,
                           const double2 *tw, const double2 *What, const FarWork &f, double *G,
                           cudaStream_t st)
{
    const int M = 2 * n, chunks = fft_chunks(n, bt.cols, T);
    product_kernel<<<dim3((unsigned)(M / 128), (unsigned)chunks, (unsigned)bt.cols), 128, 0, st>>>(
        f.Fhat, What, f.mark, f.big, bt.cols, bt.dim, multi, M, g_max, T, f.acc);
    inverse_kernel<<<(unsigned)bt.cols, fft_threads(M), sizeof(double2) * M, st>>>(
        f.acc, f.mid, f.big, chunks, bt.cols, n, T, tw, G);
    return cudaGetLastError();
}

}  // namespace fabm
