// combine.cuh -- the sum of a split row's segment partials, by one warp: the
// last warp to finish a segment of the row (rows_kernel.cuh), or the combine
// kernel (combine.cu, which says where).
#pragma once

#include "internal.h"

namespace spmm {

// lanes that share the columns of a row of k floats: the least power of two >= k, at most 32
__host__ __device__ __forceinline__ int combine_lanes_log2(int32_t k) {
    int lg = 0;
    while ((1 << lg) < k && lg < 5) ++lg;
    return lg;
}

// One warp per split row.  With k < 32 the warp is cut into SG = 32 / L
// segment groups of L lanes (L the smallest power of two >= k): group g adds
// segments g, g + SG, ... in order, then the groups' sums are added by a
// fixed xor-shuffle tree, so the result is the same on every run.
// Compensated partials are added in segment order by one group (SG = 1).
__device__ __forceinline__ void combine_row(const int4 sp, const float* __restrict__ partials, float* __restrict__ Y,
                                            int64_t ldy, int32_t k, int32_t lanes_log2,
                                            const float* __restrict__ pcomp, int lane) {
    if (pcomp) {                               // Neumaier summation of (sum, compensation) partials
        for (int c = lane; c < k; c += 32) {
            const int64_t base = (int64_t)sp.z * k + c;
            float acc = 0.f, cmp = 0.f;
            for (int q = 0; q < sp.y; ++q) {
                const float x = __ldcg(partials + base + (int64_t)q * k);
                const float t = acc + x;
                cmp += ((fabsf(acc) >= fabsf(x)) ? (acc - t) + x : (x - t) + acc) +
                       __ldcg(pcomp + base + (int64_t)q * k);
                acc = t;
            }
            Y[(int64_t)sp.x * ldy + c] = acc + cmp;
        }
        return;
    }
    const int L = 1 << lanes_log2, SG = 32 >> lanes_log2;
    const int g = lane >> lanes_log2, li = lane & (L - 1);
    for (int c0 = 0; c0 < k; c0 += L) {        // one pass unless k > 32
        const int c = c0 + li;
        const float* p = partials + (int64_t)sp.z * k + c;
        float acc = 0.f;
        if (c < k) {
            int q = g;
            for (; q + 7 * SG < sp.y; q += 8 * SG) {
                float v[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) v[u] = __ldcg(p + (int64_t)(q + u * SG) * k);
#pragma unroll
                for (int u = 0; u < 8; ++u) acc += v[u];
            }
            for (; q < sp.y; q += SG) acc += __ldcg(p + (int64_t)q * k);
        }
        for (int off = L; off < 32; off <<= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
        if (g == 0 && c < k) Y[(int64_t)sp.x * ldy + c] = acc;
    }
}

}  // namespace spmm
