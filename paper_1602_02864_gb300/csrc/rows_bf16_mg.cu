// rows_bf16_mg.cu -- row-task kernel instantiations for __nv_bfloat16 X whose short-row
// runs are split into equal pieces per lane group (merge-based), in their own
// translation unit so they compile in parallel with the others.
#include "rows_kernel.cuh"

namespace spmm {

cudaError_t launch_rows_bf16_mg(const FwdArgs& a, int vmode, int vec, int ch, cudaStream_t s) {
    if (vmode != 0 && (vec < 4 || a.x_large)) return launch_rows_t<__nv_bfloat16, false, 3>(a, vmode, vec, ch, s);
    return launch_rows_t<__nv_bfloat16, false, 1>(a, vmode, vec, ch, s);
}

}  // namespace spmm
