// Direct kernel: a CTA takes a run of grouped particles and gathers every
// stencil from the field in global memory, through L1.  The order the
// particles are grouped in (cubes of cells, columns of cell blocks along x3,
// or none) only sets how much of the field the CTAs of an SM share in L1; any
// order gives the same results.
//
// Bound: the L1 data path.  A stencil is I^2 runs of I records (16 bytes), at
// about 1.2 cycles per run and SM on L1 hits: I = 6 44 cycles, I = 8 74.
#pragma once

#include <algorithm>

#include "block_kernel.cuh"

namespace trk {

// Warps of a CTA that fills an SM at the kernel's register cap; float64
// kernels, bound by the float64 pipe, four of 16.
template <typename T, int I, int MODE>
constexpr int direct_max_warps() { return sizeof(T) == 8 ? NW : 4 * min_ctas<T, I, MODE, SRC_GLOBAL>(); }

// shared-memory carveout (percent of the SM's 228 KB) that holds `ctas` CTAs of
// `smem` bytes each, with the 1 KB the system reserves per CTA
inline int carveout_percent(size_t smem, int ctas)
{
    const size_t per_cta = (smem + 1024 + 127) / 128 * 128;
    const size_t pct = (ctas * per_cta * 100 + 233471) / 233472;
    return (int)(pct < 100 ? pct : 100);
}

template <typename T, int I, int DEG, int MODE, int NC, int STORE, int RW>
__global__ void __launch_bounds__(32 * direct_max_warps<T, I, MODE>(),
                                  4 * min_ctas<T, I, MODE, SRC_GLOBAL>() / direct_max_warps<T, I, MODE>())
    k_direct(const __grid_constant__ BlockArgs a)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int64_t j0 = (int64_t)blockIdx.x * a.ppc;
    const int64_t j1 = j0 + a.ppc < a.np ? j0 + a.ppc : a.np;
    unsigned char* ws = smem_raw + warp * WarpPlan<T, MODE, NC>::total;
    if constexpr (sizeof(T) == 4 && I == 8 && RW == 4 && !is_deriv<MODE>())
        run_direct_warp<DEG, MODE, NC>(a, j0, j1, ws, warp, nw, lane);
    else
        run_direct<T, I, DEG, MODE, NC, STORE, RW>(a, j0, j1, ws, warp, nw, lane);
}

template <typename T, int I, int DEG, int MODE, int NC, int STORE, int RW>
cudaError_t launch_direct_t(BlockArgs a, cudaStream_t st)
{
    if (a.np <= 0) return cudaSuccess;
    constexpr size_t per_warp = WarpPlan<T, MODE, NC>::total;
    constexpr int maxw = direct_max_warps<T, I, MODE>(), ctas_sm = min_ctas<T, I, MODE, SRC_GLOBAL>();
    auto kern = k_direct<T, I, DEG, MODE, NC, STORE, RW>;
    static int nsm = 0;
    if (!nsm) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(maxw * per_warp));
        if (e != cudaSuccess) return e;
        // the gathers run through L1: ask for no more shared memory than the resident CTAs use
        e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout,
                                 carveout_percent(NW * per_warp, ctas_sm));
        if (e != cudaSuccess) return e;
        int dev = 0;
        if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
        if ((e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    }
    // a.ppc: a launch shape (every shape gives the same results); PPC_WIDE: CTAs that
    // fill an SM, whose warps share one neighbourhood of the field in L1; 0, by size:
    // 16 to 256 particles per CTA, so that small sets still reach every SM and larger
    // ones have eight CTAs per resident one.  On a field of many times the L2, at most
    // 64: concurrent CTAs close together share what they pull into L2 (512^3, I = 8, 9e5
    // tracers, AB2: 565 us per step against 675 with 128 and 743 with 256; not where two
    // CTAs hold an SM, I = 6 RK2: 1.5e6 tracers 901 with 64, 850 with 256).  I = 8 on
    // denser sets: wide (256^3, 1/16 per cell, RK2: 594 us against 638 with 256 by four
    // warps; 512^3, 1/33: 2479 against 2658 with 64).
    int nw = NW;
    if (a.ppc == 0) {
        const int64_t even = (a.np + (int64_t)nsm * ctas_sm - 1) / ((int64_t)nsm * ctas_sm);
        const int64_t n = a.f.NP - 2 * PAD, want = even <= 32 ? even : std::max<int64_t>(32, even / 8);
        const int64_t cap = ctas_sm > 2 && n * n * n * 4 * (int64_t)sizeof(T) > ((int64_t)1 << 30) ? 64 : 256;
        a.ppc = (int)std::min<int64_t>(cap, std::max<int64_t>(16, (want + 15) / 16 * 16));
        if (sizeof(T) == 4 && I == 8 && a.np >= 64 * 16 * (int64_t)nsm && 34 * a.np >= n * n * n) a.ppc = PPC_WIDE;
    }
    if (a.ppc == PPC_WIDE) {
        nw = maxw;
        a.ppc = 64 * nw;
    }
    kern<<<(unsigned)((a.np + a.ppc - 1) / a.ppc), 32 * nw, nw * per_warp, st>>>(a);
    return cudaGetLastError();
}

// Component chunk and record width of a mode: time steps contract three
// components; interpolation one (C = 1, 4-byte records), three (C = 2, 3) or
// chunks of four.
template <int I, int DEG, class F>
cudaError_t dispatch_mode(int mode, const FieldView& f, F&& go)
{
    const int s = f.storage;
#define TRK_STORE(M, NC, RW)                                             \
    if (s == ST_F64) return go.template run<double, M, NC, ST_F64, 4>(); \
    return go.template run<float, M, NC, ST_F32, RW>();
#define TRK_INTERP(M)                                      \
    if (f.C == 1) { TRK_STORE(M, 1, 1) }                   \
    if (f.C <= 3) { TRK_STORE(M, 3, 4) }                   \
    TRK_STORE(M, 4, 4)
    switch (mode) {
        case MODE_INTERP: TRK_INTERP(MODE_INTERP)
        case MODE_INTERP_DERIV: TRK_INTERP(MODE_INTERP_DERIV)
        case MODE_RK2: TRK_STORE(MODE_RK2, 3, 4)
        case MODE_AB2: TRK_STORE(MODE_AB2, 3, 4)
    }
#undef TRK_INTERP
#undef TRK_STORE
    return cudaErrorInvalidValue;
}

template <int I, int DEG>
struct GoDirect {
    const BlockArgs& a;
    cudaStream_t st;
    template <typename T, int MODE, int NC, int STORE, int RW>
    cudaError_t run() const
    {
        return launch_direct_t<T, I, DEG, MODE, NC, STORE, RW>(a, st);
    }
};

template <int I, int DEG>
struct GoBlock {
    const BlockArgs& a;
    const CUtensorMap* tmap;
    int64_t nblocks;
    cudaStream_t st;
    template <typename T, int MODE, int NC, int STORE, int RW>
    cudaError_t run() const
    {
        return launch_block_t<T, I, DEG, MODE, NC, STORE, RW>(a, tmap, nblocks, st);
    }
};

}  // namespace trk
