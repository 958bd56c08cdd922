// Block kernels for kernel width I = 4, weights of degree I - 1
// (all storages and modes).
#include "direct_kernel.cuh"

namespace trk {

cudaError_t launch_block_i4(int mode, const BlockArgs& a, const void* tmap, int64_t nblocks, cudaStream_t st)
{
    const CUtensorMap* m = static_cast<const CUtensorMap*>(tmap);
    if (mode == MODE_AB2_D) return launch_slabs<4, 3, MODE_AB2_D, 3>(a, *m, st);   // (batched sets)
    return dispatch_mode<4, 3>(mode, a.f, GoBlock<4, 3>{a, m, nblocks, st});
}

}  // namespace trk
