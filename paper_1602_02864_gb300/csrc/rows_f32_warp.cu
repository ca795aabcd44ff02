// rows_f32_warp.cu -- row-task kernel instantiations for float X with a whole
// warp per X row, in their own translation unit so they compile in parallel
// with the others.
#include "rows_kernel.cuh"

namespace spmm {

cudaError_t launch_rows_f32_warp(const FwdArgs& a, int vmode, int vec, int ch, cudaStream_t s) {
    return launch_rows_t<float, false, 4>(a, vmode, vec, ch, s);
}

}  // namespace spmm
