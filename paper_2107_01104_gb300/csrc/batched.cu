// Batched AB2 advection: many particle sets of uneven size and different
// kernels (I = 4, 6, 8; value or value + gradient outputs) advanced by one
// persistent launch per step (dense sets: the slab pipeline).  CTAs take work items from a per-set atomic
// counter, set after set: an item is a run of 128 grouped particles whose
// stencils are gathered from the field through L1 (run_direct).  Large sets
// come last in no particular order; the items are small, so the tail is
// shorter than an item.
#include <algorithm>

#include "direct_kernel.cuh"

namespace trk {

namespace {

__host__ __device__ constexpr size_t batched_warp_bytes()
{
    return std::max(WarpPlan<float, MODE_AB2_D, 3>::total, WarpPlan<float, MODE_AB2, 3>::total);
}

template <int I, int DEG>
__device__ __forceinline__ void run_item(const BatchSet& S, int64_t j0, int64_t j1, unsigned char* ws, int warp, int lane)
{
    if (S.deriv) run_direct<float, I, DEG, MODE_AB2_D, 3, ST_F32, 4>(S.a, j0, j1, ws, warp, NW, lane);
    else if constexpr (I == 8) run_direct_warp<DEG, MODE_AB2, 3>(S.a, j0, j1, ws, warp, NW, lane);
    else run_direct<float, I, DEG, MODE_AB2, 3, ST_F32, 4>(S.a, j0, j1, ws, warp, NW, lane);
}

__global__ void __launch_bounds__(NT, 4) k_batched(const BatchSet* __restrict__ sets, int nsets, int* ctr)
{
    __shared__ __align__(128) unsigned char smem[NW * batched_warp_bytes()];
    __shared__ int s_item;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned char* ws = smem + warp * batched_warp_bytes();
    for (int s = 0; s < nsets; ++s) {
        const BatchSet& S = sets[s];
        for (;;) {
            if (threadIdx.x == 0) s_item = atomicAdd(ctr + s, 1);
            __syncthreads();
            const int it = s_item;
            __syncthreads();
            if (it >= S.n_items) break;
            const int64_t j0 = (int64_t)it * PB, j1 = j0 + PB < S.a.np ? j0 + PB : S.a.np;
            switch (S.I * 2 + S.deg_hi) {
                case 8: run_item<4, 3>(S, j0, j1, ws, warp, lane); break;
                case 9: run_item<4, 5>(S, j0, j1, ws, warp, lane); break;
                case 12: run_item<6, 5>(S, j0, j1, ws, warp, lane); break;
                case 13: run_item<6, 7>(S, j0, j1, ws, warp, lane); break;
                case 16: run_item<8, 7>(S, j0, j1, ws, warp, lane); break;
                default: run_item<8, 9>(S, j0, j1, ws, warp, lane); break;
            }
        }
    }
}

}  // namespace

cudaError_t launch_batched(const BatchSet* sets, int nsets, int* ctr, int nsm, cudaStream_t st)
{
    static int ctas = 0;
    if (!ctas) {
        cudaError_t e = cudaFuncSetAttribute(k_batched, cudaFuncAttributePreferredSharedMemoryCarveout,
                                             carveout_percent(NW * batched_warp_bytes(), 4));
        if (e != cudaSuccess) return e;
        int occ = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_batched, NT, 0);
        if (e != cudaSuccess) return e;
        ctas = std::max(occ, 1);
    }
    k_batched<<<nsm * ctas, NT, 0, st>>>(sets, nsets, ctr);
    return cudaGetLastError();
}

}  // namespace trk
