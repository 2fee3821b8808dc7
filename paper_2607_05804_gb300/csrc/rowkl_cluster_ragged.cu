// The row grids of rowkl_cluster.cuh for bf16 logits whose row stride is not a multiple of 8:
// a row's first and last vectors are masked in the statistics and written column by column.

#include "rowkl_cluster.cuh"

namespace turnopd {

cudaError_t launch_rows_bf16_ragged(const RowIn &p, bool fp32_grad, cudaStream_t stream)
{
    return launch_rows_t<__nv_bfloat16, kAny>(p, fp32_grad, stream);
}

}  // namespace turnopd
