// Block kernels for kernel width I = 8, weights of degree I + 1 (spline with m = I / 2)
// (all storages and modes).
#include "direct_kernel.cuh"

namespace trk {

cudaError_t launch_block_i8h(int mode, const BlockArgs& a, const void* tmap, int64_t nblocks, cudaStream_t st)
{
    const CUtensorMap* m = static_cast<const CUtensorMap*>(tmap);
    if (mode == MODE_AB2_D) return launch_slabs<8, 9, MODE_AB2_D, 3>(a, *m, st);   // (batched sets)
    return dispatch_mode<8, 9>(mode, a.f, GoBlock<8, 9>{a, m, nblocks, st});
}

}  // namespace trk
