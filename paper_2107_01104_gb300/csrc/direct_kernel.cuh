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
constexpr int direct_max_warps() { return sizeof(T) == 8 ? NW : 4 * CTAS_SM; }

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
                                  4 * CTAS_SM / direct_max_warps<T, I, MODE>())
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
    constexpr int maxw = direct_max_warps<T, I, MODE>(), ctas_sm = CTAS_SM;
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
    // a.ppc: particles per CTA (every shape gives the same results); 0, by size (us per
    // step, float32 unless noted):
    //  - float64, bound by its pipe: an even share per resident CTA, so that every SM has its
    //    warps to the end, in rounds of a warp where that is less for the fullest SM (warps of a
    //    CTA that have none cost nothing; 128^3, I = 6, RK2, two steps with their binning: 4e4
    //    tracers 348, in rounds of a CTA 386; 1e5 762, 811; 2e5 1459, 1487), else of a CTA, whose
    //    warps then end together (32^3, I = 8, RK2, one step: 2e4 tracers 164, 169).
    //  - up to 64 each (I = 8: 32), the same (64^3, I = 4, 3.5e4: 12 with 64, 16 with 32,
    //    28 in CTAs of 1024).
    //  - then an eighth of an even share per resident CTA, so that the last wave is short,
    //    up to 256, which keeps a CTA's stencils close together (256^3, I = 4, AB2, 2^21: 235
    //    with 256, 356 with 64).
    //  - at most 64 on sets below 1/80 per cell in a field of many times the L2 (records above
    //    1 GB), whose concurrent CTAs then share what they pull into it (512^3, AB2, 64 and
    //    256: 1e6 I = 4 266, 288, I = 6 430, 468, I = 8 584, 641; but 3e6 492, 457 and 966, 846
    //    and 1406, 1353; 3e7 I = 4 4610, 2943; 1024^3, I = 6, 6e6 3191, 3541, 2e7 6437, 6189).
    //    In smaller fields for I = 8 (256^3, 5e5, RK2: 322, 352 with 256) and for RK2's
    //    sixteen lanes on sets below 1/12 per cell (256^3, 8e5: 314 with 64, 330 with 1024).
    //  - I = 8 from 1/20 per cell on (big fields 1/32), sets of at least one such CTA per SM: CTAs
    //    that fill an SM, whose warps share one neighbourhood of the field in L1 (PPC_WIDE;
    //    256^3, 2^21, RK2: 1126, 1229 with 256, 1258 with 64; 4e5 264, 244 with 64; 512^3, 4.5e6
    //    2504, 2585 with 256, 3e6 1800, 1763).
    int nw = NW;
    if (a.ppc == 0) {
        constexpr bool split = group_lanes<T, I, MODE, SRC_GLOBAL>() == 16, f32 = sizeof(T) == 4;
        const int64_t even = (a.np + (int64_t)nsm * ctas_sm - 1) / ((int64_t)nsm * ctas_sm);
        const int64_t n = a.f.NP - 2 * PAD, cells = n * n * n, one_wave = I < 8 ? 64 : 32;
        const int64_t want = !f32 || even <= one_wave ? even : std::max<int64_t>(one_wave, even / 8);
        const bool big = cells * 16 > (int64_t)1 << 30;
        const bool small = big ? 80 * a.np < cells : I == 8 || (split && 12 * a.np < cells);
        // whole rounds of the CTA, or (float64) of a warp where an SM then has fewer of these in all
        constexpr int round = 32 / group_lanes<T, I, MODE, SRC_GLOBAL>();
        const auto ceil_to = [](int64_t x, int64_t u) { return (x + u - 1) / u * u; };
        const auto per_sm = [&](int64_t p) { return ceil_to(ceil_to(a.np, p) / p, nsm) / nsm * ceil_to(p, round); };
        int64_t unit = f32 ? std::max(16, NW * round) : NW * round;
        if (!f32 && per_sm(ceil_to(want, round)) < per_sm(ceil_to(want, unit))) unit = round;
        a.ppc = (int)std::min<int64_t>(!f32 ? 1 << 20 : (small ? 64 : 256) / unit * unit, ceil_to(want, unit));
        if (f32 && I == 8 && a.np >= 64 * 16 * (int64_t)nsm && (big ? 32 : 20) * a.np >= cells) a.ppc = PPC_WIDE;
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
