// Adjoint block kernels for kernel width I = 4 (float64 fields).
#include "adjoint_kernel.cuh"

namespace trk {

cudaError_t launch_adjoint_i4(const AdjArgs& a, int64_t nblocks, int deg_hi, cudaStream_t st)
{
    if (deg_hi) return adj::dispatch_adjoint<4, 4 + 1>(a, nblocks, st);
    return adj::dispatch_adjoint<4, 4 - 1>(a, nblocks, st);
}

}  // namespace trk
