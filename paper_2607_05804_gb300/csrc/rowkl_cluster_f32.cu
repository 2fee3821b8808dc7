// The row grids of rowkl_cluster.cuh for fp32 logits whose vocabulary and row stride are
// multiples of 4.

#include "rowkl_cluster.cuh"

namespace turnopd {

cudaError_t launch_rows_f32(const RowIn &p, bool fp32_grad, cudaStream_t stream)
{
    return launch_rows_t<float, kWhole>(p, fp32_grad, stream);
}

}  // namespace turnopd
