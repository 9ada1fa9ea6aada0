// Mixed-precision (FP32 cycles) instantiations of the discrete-adjoint kernel (V-cycle and
// cycle-index-gamma preconditioners), in a translation unit of their own so
// that they compile in parallel with the rest of the library.
#include "fused_adjoint.cuh"

namespace rich_fused {

const void* rich_adjoint_kernel32(bool wcycle) {
    return wcycle ? (const void*)k_adjoint<float, true> : (const void*)k_adjoint<float, false>;
}

void rich_adjoint_launch32(const FParams& P, int grid, size_t smem, cudaStream_t st) {
    if (P.gamma > 1) k_adjoint<float, true><<<grid, 512, smem, st>>>(P);
    else k_adjoint<float, false><<<grid, 512, smem, st>>>(P);
}

int rich_adjoint_cluster32(const FParams& P, size_t smem, int n, int clusters, cudaStream_t st, int* fit) {
    return cluster_call(k_adjoint_cluster<float>, P, smem, n, clusters, st, fit);
}

}  // namespace rich_fused
