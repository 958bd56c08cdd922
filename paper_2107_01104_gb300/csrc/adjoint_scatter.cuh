// Adjoint of one RK2 step for float32 and split-bf16 fields, in two kernels:
//
//   particles  MODE_ADJ of the interpolation kernels (k_slabs, or k_direct for
//              sparse sets): J(X), J(X*) and the float64 lambda recurrence;
//              leaves X*, mu and dt/2 lambda in grouped order (X* from a u summed
//              beside its derivatives: the forward step's up to rounding, contract);
//   scatter    gfield += W(X)^T mu + W(X*)^T (dt/2 lambda), here.
//
// (Float64 fields: adjoint_kernel.cuh.)
//
// Scatter of a dense set: one CTA per cell block; a warp keeps the sums of its
// x2 rows of the block's halo in registers -- lanes along x1, x3 planes in
// registers, two halves of eight planes where the halo is at most 16 wide --
// and adds, for every stencil that covers a row, the outer product of its x1
// weights, its x3 weights (zero outside the stencil) and w2 mu.  Warp w owns
// rows w and w + 8: the blocks are 8 rows high, so every warp meets the same
// number of stencils (I = 8: one row per warp).  The stencils' weights are
// expanded in shared memory once per batch, sorted by their first row, so a
// warp reads only those that cover its rows; the two stencils of a particle
// whose X and X* share a cell are added as one.  No atomics and no memory
// traffic per node: a stencil costs a warp about 25 instructions per row (12
// of them packed FMAs), where an atomic add per node and component cost 7 L2
// sectors per 32 adds, and a read-modify-write in shared memory about 100
// wavefronts per stencil.  The block's sums go to its slab of scratch once, to
// be added per node over the blocks in a fixed order (k_adj_gather), or by
// float64 atomics without one.
#pragma once

#include "direct_kernel.cuh"

namespace trk {

constexpr int SB = 128;           // particles per batch of the scatter, two stencils each

template <int I>
struct ScatterPlan {
    static constexpr int H = adj_halo(I);              // rows, columns and planes of the halo
    static constexpr bool HALVES = H <= 16;
    static constexpr int RPW = HALVES ? 2 : 1;         // rows per warp: w, w + 8
    static constexpr int WARPS = HALVES ? 8 : H;
    static constexpr int XE = HALVES ? 16 : 20;        // expanded x1 weights
    static constexpr int NZ = HALVES ? 8 : 20;         // planes per lane
    static constexpr int ZE = HALVES ? 16 : 20;        // expanded x3 weights
    static constexpr int E = 2 * SB;                   // stencils per batch
    static constexpr size_t w1 = 0;                                            // [E][XE]
    static constexpr size_t w3 = w1 + (size_t)E * XE * 4;                      // [E][ZE]
    static constexpr size_t wm = w3 + (size_t)E * ZE * 4;                      // [E][I] w2 mu (float4)
    static constexpr size_t cnt = wm + (size_t)E * I * 16;                     // [32] stencils per first row (pairs, singles), then offsets
    static constexpr size_t total = cnt + 256;
    static_assert(2 * (H - I + 1) < 32 && 32 * WARPS >= E, "counters; one thread per stencil");
};

__device__ __forceinline__ unsigned long long pack2(float a)
{
    unsigned long long r;
    asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(a));
    return r;
}
// two fused multiply-adds, acc += a * w elementwise
__device__ __forceinline__ void fma2(unsigned long long& acc, unsigned long long a, unsigned long long w)
{
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(w));
}
__device__ __forceinline__ unsigned long long mul2(unsigned long long a, unsigned long long b)
{
    unsigned long long r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ unsigned long long add2(unsigned long long a, unsigned long long b)
{
    unsigned long long r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ float2 unpack2(unsigned long long v)
{
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}

// the weight of node i of one axis at offset t
template <int I, int DEG>
__device__ __forceinline__ float axis_weight(const CoefTable<float>& tb, float t, int i)
{
    float acc = tb.c[i][DEG];
#pragma unroll
    for (int d = DEG - 1; d >= 0; --d) acc = fmaf(acc, t - 0.5f, tb.c[i][d]);
    return acc;
}

// the outer products of one stencil (e) or two (e, e + 1) of a row
template <int I, bool TWO>
__device__ __forceinline__ void add_row(const float* w1e, const float* w3e, const float4* wme, int e, int row, int x, int z0,
                                        unsigned long long (&acc)[3][ScatterPlan<I>::NZ / 2])
{
    using P = ScatterPlan<I>;
    const float4 m0 = wme[e * I + row], m1 = TWO ? wme[(e + 1) * I + row] : m0;
    const float wa = w1e[e * P::XE + x], wb = TWO ? w1e[(e + 1) * P::XE + x] : wa;
    const ulonglong2* za = reinterpret_cast<const ulonglong2*>(w3e + e * P::ZE + z0);
    const ulonglong2* zb = reinterpret_cast<const ulonglong2*>(w3e + (e + 1) * P::ZE + z0);
    const unsigned long long a[3] = {pack2(wa * m0.x), pack2(wa * m0.y), pack2(wa * m0.z)};
    const unsigned long long b[3] = {pack2(wb * m1.x), pack2(wb * m1.y), pack2(wb * m1.z)};
#pragma unroll
    for (int i = 0; i < P::NZ / 4; ++i) {
        const ulonglong2 u = za[i];
        if constexpr (TWO) {
            const ulonglong2 v = zb[i];
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                unsigned long long s = mul2(a[k], u.x), t = mul2(a[k], u.y);
                fma2(s, b[k], v.x);
                fma2(t, b[k], v.y);
                acc[k][2 * i] = add2(acc[k][2 * i], s);
                acc[k][2 * i + 1] = add2(acc[k][2 * i + 1], t);
            }
        } else {
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                fma2(acc[k][2 * i], a[k], u.x);
                fma2(acc[k][2 * i + 1], a[k], u.y);
            }
        }
    }
}

// SLAB: the block's sums into its slab of scratch, [3][H][H][H]; else float64 atomics into gfield
template <int I, int DEG, bool SLAB>
__global__ void __launch_bounds__(32 * ScatterPlan<I>::WARPS, ScatterPlan<I>::HALVES ? 3 : 1)
    k_adj_scatter(const __grid_constant__ AdjScatterArgs a)
{
    using P = ScatterPlan<I>;
    constexpr int H = P::H, G = I / 2, LO = I / 2 - 1, NZ = P::NZ, RPW = P::RPW;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    float* w1e = reinterpret_cast<float*>(smem_raw + P::w1);
    float* w3e = reinterpret_cast<float*>(smem_raw + P::w3);
    float4* wme = reinterpret_cast<float4*>(smem_raw + P::wm);
    int* cnt = reinterpret_cast<int*>(smem_raw + P::cnt);      // [32], then the offsets [33]
    int* off = cnt;
    const int b = blockIdx.x;
    const int j0 = a.offsets[b], j1 = a.offsets[b + 1];
    if (j0 >= j1) return;
    const int N = a.g.N, mask = a.g.mask;
    const int o1 = b % a.g.nb1 * BLK - G, o2 = b / a.g.nb1 % a.g.nb2 * BLK - G, o3 = b / (a.g.nb1 * a.g.nb2) * BLK - G;
    const int64_t NN3 = (int64_t)N * N * N;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int x = P::HALVES ? lane & 15 : min(lane, P::XE - 1), z0 = P::HALVES ? (lane >> 4) * 8 : 0;
    unsigned long long acc[RPW][3][NZ / 2] = {};
    for (int b0 = j0; b0 < j1; b0 += SB) {
        const int n = 2 * min(SB, j1 - b0);
        if (tid < 32) cnt[tid] = 0;
        __syncthreads();
        // one thread per stencil (a particle's two in adjacent lanes): where it goes
        float4 at = make_float4(0.f, 0.f, 0.f, 0.f), mu = at;
        int key = -1, slot = 0, n1 = 0, n2 = 0, n3 = 0;
        if (tid < n) {
            at = (tid & 1) ? a.adj[b0 + (tid >> 1)] : a.rec[b0 + (tid >> 1)];
            mu = a.adj[(1 + (tid & 1)) * a.np + b0 + (tid >> 1)];
        }
        const int c = __float_as_int(at.w);
        // a stencil with a non-finite factor (or one near the end of the range) is added node by
        // node: times the zeros that expand the weights it would put NaN into whole planes
        const bool tame = fabsf(mu.x) + fabsf(mu.y) + fabsf(mu.z) + at.x + at.y + at.z < 1e37f;
        const bool same = (__shfl_xor_sync(0xffffffffu, c, 1) == c) & tame & __shfl_xor_sync(0xffffffffu, (int)tame, 1);
        if (tid < n) {
            n1 = (((c & 1023) - o1) & mask) - LO;               // first node, relative to the halo
            n2 = (((c >> 10 & 1023) - o2) & mask) - LO;
            n3 = (((c >> 20 & 1023) - o3) & mask) - LO;
            if ((unsigned)n1 <= (unsigned)(H - I) && (unsigned)n2 <= (unsigned)(H - I) && (unsigned)n3 <= (unsigned)(H - I) && tame) {
                key = 2 * n2 + (same ? 0 : 1);
                if (!same) slot = atomicAdd(cnt + key, 1);
                else if (!(tid & 1)) slot = atomicAdd(cnt + key, 2);
            }
        }
        const int pair_slot = __shfl_sync(0xffffffffu, slot, lane & ~1);
        if (same) slot = pair_slot + (lane & 1);
        __syncthreads();
        if (tid < 32) {   // counts -> offsets
            const int v = cnt[lane];
            int inc = v;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int up = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o) inc += up;
            }
            off[lane] = inc - v;
        }
        __syncthreads();
        // its weights, expanded over the halo
        if (tid < n) {
            if (key >= 0) {
                const int e = off[key] + slot;
                float4* e1 = reinterpret_cast<float4*>(w1e + e * P::XE);
                float4* e3 = reinterpret_cast<float4*>(w3e + e * P::ZE);
#pragma unroll
                for (int i = 0; i < P::XE / 4; ++i) e1[i] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int i = 0; i < P::ZE / 4; ++i) e3[i] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int i = 0; i < I; ++i) {
                    w1e[e * P::XE + n1 + i] = axis_weight<I, DEG>(a.cf, at.x, i);
                    w3e[e * P::ZE + n3 + i] = axis_weight<I, DEG>(a.cf, at.z, i);
                    const float w2 = axis_weight<I, DEG>(a.cf, at.y, i);
                    wme[e * I + i] = make_float4(w2 * mu.x, w2 * mu.y, w2 * mu.z, 0.f);
                }
            } else {   // X* left the halo (flagged by the gathers), or not tame: straight into the gradient
#pragma unroll 1
                for (int q = 0; q < I * I * I; ++q) {
                    const int ix = q % I, iy = q / I % I, iz = q / (I * I);
                    const int64_t gi = ((int64_t)((o3 + n3 + iz) & mask) * N + ((o2 + n2 + iy) & mask)) * N + ((o1 + n1 + ix) & mask);
                    const float w = axis_weight<I, DEG>(a.cf, at.x, ix) * axis_weight<I, DEG>(a.cf, at.y, iy) *
                                    axis_weight<I, DEG>(a.cf, at.z, iz);
                    atomicAdd(a.gfield + gi, (double)(w * mu.x));
                    atomicAdd(a.gfield + NN3 + gi, (double)(w * mu.y));
                    atomicAdd(a.gfield + 2 * NN3 + gi, (double)(w * mu.z));
                }
            }
        }
        __syncthreads();
        // the stencils that cover row y have first rows max(0, y - I + 1) .. min(y, H - I)
#pragma unroll
        for (int r = 0; r < RPW; ++r) {
            const int y = warp + 8 * r;
            if (y >= H) continue;
            for (int f = max(0, y - I + 1); f <= min(y, H - I); ++f) {
                const int p0 = off[2 * f], p1 = off[2 * f + 1], p2 = off[2 * f + 2];
#pragma unroll 1
                for (int e = p0; e < p1; e += 2) add_row<I, true>(w1e, w3e, wme, e, y - f, x, z0, acc[r]);
#pragma unroll 1
                for (int e = p1; e < p2; ++e) add_row<I, false>(w1e, w3e, wme, e, y - f, x, z0, acc[r]);
            }
        }
        __syncthreads();   // the batch's weights are read before the next batch's
    }
    if (P::HALVES ? x >= H : lane >= H) return;
#pragma unroll
    for (int r = 0; r < RPW; ++r) {
        const int y = warp + 8 * r;
        if (y >= H) continue;
#pragma unroll
        for (int i = 0; i < NZ / 2; ++i)
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const float2 v = unpack2(acc[r][k][i]);
#pragma unroll
                for (int s = 0; s < 2; ++s) {
                    const int z = z0 + 2 * i + s;
                    const float val = s ? v.y : v.x;
                    if (z >= H) continue;
                    if constexpr (SLAB) {
                        a.gscratch[(((int64_t)b * 3 + k) * H + z) * H * H + y * H + x] = val;
                    } else if (val != 0.0f) {
                        const int64_t gi = ((int64_t)((o3 + z) & mask) * N + ((o2 + y) & mask)) * N + ((o1 + x) & mask);
                        atomicAdd(a.gfield + k * NN3 + gi, (double)val);
                    }
                }
            }
    }
}

// Scatter of a sparse set: four particles at a time per warp, I = 6 five (the lane
// maps of the interpolation), one float64 atomic per node and component, both
// stages in one where X and X* share a cell.  Each pass over the nodes is 3 I^2
// conversions and atomics per warp (the bound) whether its lanes are busy or
// not, so the CTA first adds its particles at X (with X* where they share a cell),
// then the X* left over, as many per warp again (256^3, I = 6, 1/32 per cell, the
// whole adjoint of four steps: 9158 -> 6560 us against passes for "shared", "X" and
// "X*" wherever one of the four differs).  Five particles of six lanes instead of four
// of eight, two of them idle, and few particles per CTA (its launch): 256^3, I = 6, us
// per call of two steps, 1e5 particles 1195 -> 893, 6.4e5 3790 -> 3401.
template <int I, int GL, bool TWO>
__device__ __forceinline__ void add_direct(const AdjScatterArgs& a, const LaneMap<I, GL>& m, int c, bool active,
                                           const Weights<float, I, false, GL>& wa, const float4& ma,
                                           const Weights<float, I, false, GL>& wb, const float4& mb)
{
    using M = LaneMap<I, GL>;
    constexpr int LO = I / 2 - 1;
    const int N = a.g.N, mask = a.g.mask;
    const int64_t NN3 = (int64_t)N * N * N;
    const int x1 = ((c & 1023) + m.x - LO) & mask, c2 = (c >> 10 & 1023) - LO, c3 = (c >> 20 & 1023) + m.z0 - LO;
    if (!active) return;
#pragma unroll
    for (int r = 0; r < M::NY; ++r) {
        const float ya = wa.w1 * wa.w2[r], yb = TWO ? wb.w1 * wb.w2[r] : 0.0f;
        double* row = a.gfield + (int64_t)((c2 + r) & mask) * N + x1;
#pragma unroll
        for (int z = 0; z < M::NZ; ++z) {
            const float va = ya * wa.w3[z], vb = TWO ? yb * wb.w3[z] : 0.0f;
            double* p = row + (int64_t)((c3 + z * M::ZS) & mask) * N * N;
            atomicAdd(p, (double)(TWO ? fmaf(va, ma.x, vb * mb.x) : va * ma.x));
            atomicAdd(p + NN3, (double)(TWO ? fmaf(va, ma.y, vb * mb.y) : va * ma.y));
            atomicAdd(p + 2 * NN3, (double)(TWO ? fmaf(va, ma.z, vb * mb.z) : va * ma.z));
        }
    }
}

template <int I>
struct SparseScatter {
    static constexpr int GL = I == 6 ? 6 : 8, P = 32 / GL;   // lanes per particle, particles at once
    static constexpr int ROUND = NW * P;                     // particles of a CTA's round
    static constexpr int ROUNDS = 2;                         // at most
};

template <int I, int DEG>
__global__ void __launch_bounds__(NT, 4) k_adj_scatter_direct(const __grid_constant__ AdjScatterArgs a, int rounds)
{
    using S = SparseScatter<I>;
    constexpr int GL = S::GL, P = S::P;
    __shared__ __align__(16) float wbuf[NW][2][P][24];
    __shared__ int rest[S::ROUNDS * S::ROUND], nrest;   // particles (from the CTA's first) whose X* lies in another cell
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int g = GL == 6 ? SixLanes(lane).group : lane / GL;
    const LaneMap<I, GL> m(lane);
    const bool act = m.act && lane < GL * P;
    Basis<float, I, DEG, false, GL> B;
    B.init(a.cf, m);
    const int64_t first = (int64_t)blockIdx.x * rounds * S::ROUND;
    if (threadIdx.x == 0) nrest = 0;
    __syncthreads();
    Weights<float, I, false, GL> w0, w1;
    for (int it = 0; it < rounds; ++it) {
        const int q = it * S::ROUND + warp * P + g;
        const int64_t j = first + q;
        const bool live = j < a.np;
        float4 at0{}, at1{}, m0{}, m1{};
        if (live) {
            at0 = a.rec[j];
            at1 = a.adj[j];
            m0 = a.adj[a.np + j];
            m1 = a.adj[2 * a.np + j];
        }
        const bool same = __float_as_int(at0.w) == __float_as_int(at1.w);
        if (live && !same && lane == GL * g) rest[atomicAdd(&nrest, 1)] = q;
        if (!same) m1.x = m1.y = m1.z = 0.0f;
        B.eval(at0.x - 0.5f, at0.y - 0.5f, at0.z - 0.5f, m, wbuf[warp][0][g], w0);
        B.eval(at1.x - 0.5f, at1.y - 0.5f, at1.z - 0.5f, m, wbuf[warp][1][g], w1);
        add_direct<I, GL, true>(a, m, __float_as_int(at0.w), live && act, w0, m0, w1, m1);
        __syncwarp();
    }
    __syncthreads();
    const int n = nrest;
    for (int k = warp * P, odd = 0; k < n; k += S::ROUND, odd ^= 1) {
        const bool live = k + g < n;
        float4 at1{}, m1{};
        if (live) {
            const int64_t j = first + rest[k + g];
            at1 = a.adj[j];
            m1 = a.adj[2 * a.np + j];
        }
        B.eval(at1.x - 0.5f, at1.y - 0.5f, at1.z - 0.5f, m, wbuf[warp][odd][g], w1);
        add_direct<I, GL, false>(a, m, __float_as_int(at1.w), live && act, w1, m1, w1, m1);
        __syncwarp();
    }
}

// particles: with tmap through the slab pipeline, else direct gathers
template <int I, int DEG>
cudaError_t launch_adj_particles(const BlockArgs& a, const CUtensorMap* tmap, cudaStream_t st)
{
    return tmap ? launch_slabs<I, DEG, MODE_ADJ, 3>(a, *tmap, st)
                : launch_direct_t<float, I, DEG, MODE_ADJ, 3, ST_F32, 4>(a, st);
}

template <int I, int DEG, bool SLAB>
cudaError_t launch_adj_scatter_t(const AdjScatterArgs& a, int64_t nblocks, cudaStream_t st)
{
    auto kern = k_adj_scatter<I, DEG, SLAB>;
    static bool attr_set = false;
    if (!attr_set) {
        const cudaError_t e =
            cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ScatterPlan<I>::total);
        if (e != cudaSuccess) return e;
        attr_set = true;
    }
    kern<<<(unsigned)nblocks, 32 * ScatterPlan<I>::WARPS, ScatterPlan<I>::total, st>>>(a);
    return cudaGetLastError();
}

// nblocks 0: the sparse scatter
template <int I, int DEG>
cudaError_t launch_adj_scatter(const AdjScatterArgs& a, int64_t nblocks, cudaStream_t st)
{
    if (nblocks == 0) {
        using S = SparseScatter<I>;
        static int nsm = 0;
        if (!nsm) {
            int dev = 0;
            cudaError_t e = cudaGetDevice(&dev);
            if (e != cudaSuccess || (e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
        }
        // two rounds while the part of the gradient that the resident CTAs work on at once stays
        // within half of the L2 (64 MB; the nodes' lines are otherwise fetched again by the next
        // row of blocks): 256^3, I = 6, us per call of two steps, one round and two: 1e5 891 and
        // 1005, 2.5e5 1589 and 1548, 6.4e5 3558 and 3401
        const double share = std::min(1.0, 2.0 * S::ROUND * 4 * nsm / (double)a.np);
        const int rounds = share * 24.0 * a.g.N * a.g.N * a.g.N <= (double)(1 << 26) ? 2 : 1;
        const int64_t cta = (int64_t)rounds * S::ROUND;
        k_adj_scatter_direct<I, DEG><<<(unsigned)((a.np + cta - 1) / cta), NT, 0, st>>>(a, rounds);
        return cudaGetLastError();
    }
    if (a.gscratch) return launch_adj_scatter_t<I, DEG, true>(a, nblocks, st);
    return launch_adj_scatter_t<I, DEG, false>(a, nblocks, st);
}

}  // namespace trk
