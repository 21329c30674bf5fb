// a2 on CUDA cores in compensated single precision ("split" precision for
// narrow batches): the far part of the hereditary sums of Sec. 2 of
// arXiv:1710.01133 for one block of 32 targets, split over the points k in
// chunks, like the double-precision kernel but in fp32, which GB300 runs at
// 64 times the double rate.
//
// f (the recurrence's float copy of the double history) and the weights are
// in fp32 (2^-24 relative); each thread adds 16 products in plain fp32 and folds the
// group into a Kahan-compensated fp32 sum, so the rounding of a chunk's sum
// stays within a few units of 2^-24 of its magnitude.  Each chunk writes
// (sum, -compensation) pairs that the float-float combine adds up in a fixed
// order and rounds once to double.  This suits batches with few columns,
// where a 128-column tensor tile would be mostly padding; wide batches use
// the tensor-core kernel.
#include <algorithm>

#include "history_blocks.cuh"

namespace fabm {
namespace {

// grid = (ceil(n_chunks / PACK), ceil(cols / kColsPerCta)); block = PACK groups of
// 32 * kColsPerCta threads, one chunk each.  One group per CTA is a kernel of its
// own: with the groups' barriers and limits it took 79 instead of 56 registers (127
// instead of 96 with several orders): LCR of two orders, 1000 x 1000, 1.58 ms, now
// 1.39 (with the recurrence on the same SMs, recurrence.cu).
constexpr int kGroup = kWarp * hist::kColsPerCta;
constexpr int kPack = 3;  // groups per CTA where the launch leaves SMs free
template <bool MULTI, int PACK>
__global__ void __launch_bounds__(PACK *kGroup)
    hist_fp32c_kernel(const double *__restrict__ F, const float *__restrict__ Ff, int64_t ldF,
                      int cols, const float *__restrict__ WB, const float *__restrict__ WA,
                      int64_t c, int64_t kc, int64_t k_end, int n_chunks, float2 *__restrict__ part,
                      int64_t wstride, int dim)
{
    const int col0 = blockIdx.y * hist::kColsPerCta;
    if constexpr (PACK == 1) {
        __shared__ hist::f32c::Tiles<MULTI> tl;
        hist::f32c::hist_fp32c_chunk<MULTI>(F, Ff, ldF, cols, WB, WA, c, kc, k_end, part, blockIdx.x, col0,
                                            wstride, dim, threadIdx.x, tl, [] { __syncthreads(); });
    } else {
        extern __shared__ __align__(16) unsigned char smem[];
        const int g = threadIdx.x / kGroup, chunk = blockIdx.x * PACK + g;
        if (chunk >= n_chunks) return;
        hist::f32c::hist_fp32c_chunk<MULTI>(
            F, Ff, ldF, cols, WB, WA, c, kc, k_end, part, chunk, col0, wstride, dim,
            threadIdx.x % kGroup, reinterpret_cast<hist::f32c::Tiles<MULTI> *>(smem)[g],
            [g] { asm volatile("bar.sync %0, %1;" ::"r"(1 + g), "r"(kGroup) : "memory"); });
    }
}

__global__ void to_float_kernel(const double *__restrict__ x, int64_t n, float *__restrict__ y)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        y[i] = (float)x[i];
}

}  // namespace

cudaError_t launch_to_float(const double *x, int64_t n, float *y, cudaStream_t st)
{
    int64_t blocks = (n + 255) / 256;
    if (blocks > 152 * 16) blocks = 152 * 16;
    to_float_kernel<<<(unsigned)blocks, 256, 0, st>>>(x, n, y);
    return cudaGetLastError();
}

cudaError_t launch_hist_fp32c(const DevBatch &bt, const float *WBf, const float *WAf,
                              int64_t wstride, int64_t c, int lag, int n_chunks, int64_t kc,
                              bool alone, float2 *part, cudaStream_t st)
{
    const int64_t k_end = (c - lag) * hist::kL;
    if (lag < 1) return cudaErrorInvalidValue;
    if (k_end <= 0) return cudaSuccess;
    // The recurrence of the block before runs beside this launch on an SM per
    // trajectory, and a step's latency grows by a third where history warps share
    // its SM (Lorenz type 2^16: 724 cycles a step against 550 alone).  So where
    // three chunks per CTA leave SMs free (fp32c_alone), each CTA takes an SM of
    // its own, and so does the recurrence.  The chunks and their sums stay as
    // they are.
    const int groups = (bt.cols + hist::kColsPerCta - 1) / hist::kColsPerCta;
    auto run = [&]<bool MULTI, int PACK>(int64_t stride, int dim) -> cudaError_t {
        auto kernel = hist_fp32c_kernel<MULTI, PACK>;
        size_t smem = 0;
        if constexpr (PACK > 1) {
            smem = std::max(sizeof(hist::f32c::Tiles<MULTI>) * PACK, kAloneSmem);
            const cudaError_t e =
                cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            if (e != cudaSuccess) return e;
        }
        kernel<<<dim3((unsigned)((n_chunks + PACK - 1) / PACK), (unsigned)groups), PACK * kGroup, smem, st>>>(
            bt.F, bt.Ff, bt.ldF, bt.cols, WBf, WAf, c, kc, k_end, n_chunks, part, stride, dim);
        return cudaGetLastError();
    };
    if (wstride)
        return alone ? run.template operator()<true, kPack>(wstride, bt.dim)
                     : run.template operator()<true, 1>(wstride, bt.dim);
    return alone ? run.template operator()<false, kPack>(0, 1) : run.template operator()<false, 1>(0, 1);
}

bool fp32c_alone(int n_chunks, int cols, int B)
{
    const int groups = (cols + hist::kColsPerCta - 1) / hist::kColsPerCta;
    return (n_chunks + kPack - 1) / kPack * groups + B <= 148;
}

}  // namespace fabm
