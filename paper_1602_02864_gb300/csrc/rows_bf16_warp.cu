// rows_bf16_warp.cu -- row-task kernel instantiations for __nv_bfloat16 X with a whole
// warp per X row, in their own translation unit so they compile in parallel
// with the others.
#include "rows_kernel.cuh"

namespace spmm {

cudaError_t launch_rows_bf16_warp(const FwdArgs& a, int vmode, int vec, int ch, cudaStream_t s) {
    return launch_rows_t<__nv_bfloat16, false, 4>(a, vmode, vec, ch, s);
}

}  // namespace spmm
