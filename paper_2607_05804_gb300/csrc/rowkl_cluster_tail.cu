// The row grids of rowkl_cluster.cuh for bf16 logits whose row stride is a multiple of 8 and
// whose vocabulary is not: a row's last vector is masked in the statistics and written column
// by column.

#include "rowkl_cluster.cuh"

namespace turnopd {

cudaError_t launch_rows_bf16_tail(const RowIn &p, bool fp32_grad, cudaStream_t stream)
{
    return launch_rows_t<__nv_bfloat16, kTail>(p, fp32_grad, stream);
}

}  // namespace turnopd
