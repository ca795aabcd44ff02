// combine.cu -- second pass for split (hub) rows: Y[row, :] = sum of the row's
// segment partials, added in a fixed order so the result is the same on every
// run.  It serves streaming handles (whose launches each hold some of a row's
// segments) and, on resident ones, task lists of more than kCombineInsideTasks,
// compensated products, the hot variant, and pattern rows on 16 or more lanes of
// one element (combines_inside, apply_resident); other launches, and the batched
// ones, add a row's partials themselves.  The partials of a call with k columns
// are packed k floats per slot (slot s at s * k), so a small k reads only the
// floats it needs.
#include "combine.cuh"

namespace spmm {

__global__ void __launch_bounds__(kWarpsPerBlock * 32)
combine_kernel(const int4* __restrict__ splits, int64_t n_splits, const float* __restrict__ partials,
               float* __restrict__ Y, int64_t ldy, int32_t k, int32_t lanes_log2, const float* __restrict__ pcomp) {
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t s = (int64_t)blockIdx.x * kWarpsPerBlock + w;
    if (s >= n_splits) return;                 // whole warps
    combine_row(splits[s], partials, Y, ldy, k, lanes_log2, pcomp, lane);
}

cudaError_t launch_combine(const int4* splits, int64_t n_splits, const float* partials, float* Y,
                           int64_t ldy, int32_t k, cudaStream_t s, const float* partials_comp) {
    if (n_splits <= 0) return cudaSuccess;
    const int lg = combine_lanes_log2(k);
    const dim3 block(kWarpsPerBlock * 32);
    const dim3 grid((unsigned)((n_splits + kWarpsPerBlock - 1) / kWarpsPerBlock));
    combine_kernel<<<grid, block, 0, s>>>(splits, n_splits, partials, Y, ldy, k, lg, partials_comp);
    return cudaGetLastError();
}

}  // namespace spmm
