// The three bf16 slices of f of the split path (number format: history_split.cu).
#pragma once

#include "fabm_internal.cuh"

namespace fabm {

__device__ __forceinline__ int exp_clamp(int e) { return e < -126 ? -126 : (e > 127 ? 127 : e); }
__device__ __forceinline__ float pow2f(int e) { return __int_as_float((exp_clamp(e) + 127) << 23); }

// Exponent of a column's segment whose largest |f| is m.
__device__ __forceinline__ int slice_exponent(float m)
{
    int E = 0;
    if (m > 0.f && m <= 3.0e38f) E = ilogbf(m) + 1;
    return E < -100 ? -100 : E;
}

// Eight values hi[q] + lo[q] on the grid of exponent E as packed bf16 per slice.
__device__ __forceinline__ void slice8(const float (&hi)[8], const float (&lo)[8], int E,
                                       uint32_t (&w)[3][4])
{
    const float sc = pow2f(8 - E);
#pragma unroll
    for (int k0 = 0; k0 < 8; k0 += 2) {
        float t[3][2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const float xh = hi[k0 + u] * sc, xl = lo[k0 + u] * sc;
            const float t0 = rintf(xh);
            const float r = ((xh - t0) + xl) * 256.f;
            const float t1 = rintf(r);
            const float t2 = rintf((r - t1) * 256.f);
            t[0][u] = t0, t[1][u] = t1 * 0x1p-8f, t[2][u] = t2 * 0x1p-16f;
        }
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            __nv_bfloat162 p = __floats2bfloat162_rn(t[q][0], t[q][1]);
            w[q][k0 / 2] = *reinterpret_cast<uint32_t *>(&p);
        }
    }
}

// Where column cloc of column tile ct has the slices of segment seg: slice q,
// points j' = 8 k1 .. 8 k1 + 7 (j' = 63 - j) at + q * 8192 + k1 * 1024 (bf16).
__device__ __forceinline__ __nv_bfloat16 *slice_base(__nv_bfloat16 *Fs, int64_t seg, int n_ct, int ct,
                                                     int cloc)
{
    return Fs + ((seg * n_ct + ct) * 3) * (int64_t)(128 * kSplitSeg) + cloc * 8;
}

}  // namespace fabm
