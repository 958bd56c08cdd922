// Adjoint of float32 and split-bf16 fields for kernel width I = 8.
#include "adjoint_scatter.cuh"

namespace trk {

cudaError_t launch_adj_particles_i8(const BlockArgs& a, const void* tmap, int deg_hi, cudaStream_t st)
{
    const CUtensorMap* m = static_cast<const CUtensorMap*>(tmap);
    if (deg_hi) return launch_adj_particles<8, 8 + 1>(a, m, st);
    return launch_adj_particles<8, 8 - 1>(a, m, st);
}

cudaError_t launch_adj_scatter_i8(const AdjScatterArgs& a, int64_t nblocks, int deg_hi, cudaStream_t st)
{
    if (deg_hi) return launch_adj_scatter<8, 8 + 1>(a, nblocks, st);
    return launch_adj_scatter<8, 8 - 1>(a, nblocks, st);
}

}  // namespace trk
