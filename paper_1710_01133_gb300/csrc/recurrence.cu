// a4 + a5: kernels around recur_block / init_one (recurrence.cuh).
#include "recurrence.cuh"

namespace fabm {
namespace {

template <class Rhs, int D>
__global__ void init_kernel(DevBatch bt, bool f_pairs, FFInputs ff)
{
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b < bt.B) init_one<Rhs, D>(bt, b, f_pairs, ff);
}

template <class Rhs, int D, bool SPLIT, int LAG>
__global__ void __launch_bounds__((SPLIT ? D + 1 : D) * kWarp)
    recur_kernel(DevBatch bt, DevWeights w, StepConsts kc, int64_t c, const double *G)
{
    if constexpr (SPLIT) {
        __shared__ __align__(16) float smem_f[recur_split_smem_floats<D, LAG>()];
        recur_block_split<Rhs, D, LAG>(bt, blockIdx.x, w, kc, c, G, smem_f);
    } else {
        __shared__ double smem[recur_smem_doubles<D, 1, LAG>()];
        recur_block<Rhs, D, 1, LAG>(bt, blockIdx.x, w, kc, c, G, smem);
    }
}

// Share of an SM's memory that the driver gives to shared memory for the compensated
// fp32 history (132 of 228 KB).  Left to itself it gives this recurrence less where a
// CTA has few bytes or few warps, and kernels that want different shares do not run on
// one SM together (LCR of two orders, 200 x 4000: 4.5 ms without, 3.5 with).
constexpr int kHistCarveout = 57;

template <bool SPLIT, int LAG>
bool launch_recur_t(int rhs, const DevBatch &bt, const DevWeights &w, const StepConsts &k,
                    int64_t c, bool alone, const double *G, cudaStream_t st)
{
    bool set = true;
    const bool ok = dispatch_rhs(rhs, bt.dim, [&]<class R, int D>() {
        constexpr int warps = SPLIT ? recur_split_warps<R, D>() : D;
        auto kernel = recur_kernel<R, D, SPLIT, LAG>;
        const size_t smem = alone ? kAloneSmem : 0;
        if (SPLIT && !alone)
            set = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout,
                                       kHistCarveout) == cudaSuccess;
        if (alone)
            set = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem) == cudaSuccess;
        if (set) kernel<<<(unsigned)bt.B, warps * kWarp, smem, st>>>(bt, w, k, c, G);
    });
    return ok && set;
}

}  // namespace

cudaError_t launch_init(int rhs, const DevBatch &bt, cudaStream_t st, bool f_pairs, const FFInputs &ff)
{
    const int threads = 128;
    const unsigned blocks = (unsigned)((bt.B + threads - 1) / threads);
    bool ok = dispatch_rhs(rhs, bt.dim, [&]<class R, int D>() {
        init_kernel<R, D><<<blocks, threads, 0, st>>>(bt, f_pairs, ff);
    });
    return ok ? cudaGetLastError() : cudaErrorInvalidValue;
}

cudaError_t launch_recur(int rhs, const DevBatch &bt, const DevWeights &w, const StepConsts &k,
                         int64_t c, int L, int lag, bool split, bool alone, const double *G,
                         cudaStream_t st)
{
    bool ok = false;
    if (L == kWarp && lag == 1)
        ok = split ? launch_recur_t<true, 1>(rhs, bt, w, k, c, alone, G, st)
                   : launch_recur_t<false, 1>(rhs, bt, w, k, c, false, G, st);
    else if (L == kWarp && lag == 2)
        ok = split ? launch_recur_t<true, 2>(rhs, bt, w, k, c, alone, G, st)
                   : launch_recur_t<false, 2>(rhs, bt, w, k, c, false, G, st);
    return ok ? cudaGetLastError() : cudaErrorInvalidValue;
}

}  // namespace fabm
