// rows_bf16_mg.cu -- row-task kernel instantiations for __nv_bfloat16 X whose short-row
// runs are split into equal pieces per lane group (merge-based), in their own
// translation unit so they compile in parallel with the others.
#include "rows_kernel.cuh"

namespace spmm {

cudaError_t launch_rows_bf16_mg(const FwdArgs& a, int vmode, int vec, int ch, cudaStream_t s) {
    // rows on two lanes run faster with two blocks whatever X takes (k = 8, us with three / two: 256 K
    // vertices 53.8 / 49.7, 2 M 255 / 240, 4 M 550 / 463), wider ones on 8-byte lanes beyond kLargeXBytes
    // (k = 12, 1 M 167 / 188, 2 M 313 / 338, 3 M 476 / 476, 4 M 664 / 652)
    if (vmode != 0 && (vec < 4 || a.lanes_log2 == 1 || a.x_large)) return launch_rows_t<__nv_bfloat16, false, 3>(a, vmode, vec, ch, s);
    return launch_rows_t<__nv_bfloat16, false, 1>(a, vmode, vec, ch, s);
}

}  // namespace spmm
