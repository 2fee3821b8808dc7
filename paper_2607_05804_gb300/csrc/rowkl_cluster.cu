// The row path's entry, and the row grids of rowkl_cluster.cuh for bf16 logits whose
// vocabulary and row stride are multiples of 8.  The grids for other rows and for fp32
// logits are the same kernels, each set in its own translation unit, so that none slows
// another's build or changes its code.

#include "rowkl_cluster.cuh"

namespace turnopd {

cudaError_t launch_rows_bf16(const RowIn &p, bool fp32_grad, cudaStream_t stream)
{
    return launch_rows_t<__nv_bfloat16, kWhole>(p, fp32_grad, stream);
}

// *used = false (and nothing is launched) for arrays that are not 16-byte aligned.
cudaError_t launch_rows(const RowIn &p, bool bf16, bool fp32_grad, cudaStream_t stream, bool *used)
{
    auto al16 = [](const void *q) { return (reinterpret_cast<uintptr_t>(q) & 15u) == 0; };
    *used = al16(p.zs) && al16(p.zt) && (!p.grad || al16(p.grad)) && p.vocab <= (int64_t)INT32_MAX - 16;
    if (!*used)
        return cudaSuccess;
    const int n = bf16 ? 8 : 4;
    const bool whole = p.vocab % n == 0 && p.ld % n == 0;
    if (bf16)
        return whole ? launch_rows_bf16(p, fp32_grad, stream)
               : p.ld % n == 0 ? launch_rows_bf16_tail(p, fp32_grad, stream)
                               : launch_rows_bf16_ragged(p, fp32_grad, stream);
    return whole ? launch_rows_f32(p, fp32_grad, stream) : launch_rows_f32_ragged(p, fp32_grad, stream);
}

}  // namespace turnopd
