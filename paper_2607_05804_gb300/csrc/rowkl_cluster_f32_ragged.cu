// The row grids of rowkl_cluster.cuh for fp32 logits whose vocabulary or row stride is not
// a multiple of 4: a row's first and last vectors are masked in the statistics and
// written column by column.

#include "rowkl_cluster.cuh"

namespace turnopd {

cudaError_t launch_rows_f32_ragged(const RowIn &p, bool fp32_grad, cudaStream_t stream)
{
    return launch_rows_t<float, kAny>(p, fp32_grad, stream);
}

}  // namespace turnopd
