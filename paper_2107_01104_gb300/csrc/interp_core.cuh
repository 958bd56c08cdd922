// The per-particle arithmetic shared by every interpolation and step kernel:
// 1-D weights, stencil gather and separable contraction (Eq. triple_sum,
// Sec. 3.3), the RK2 stage-2 point, and the lane-dense float64 phases around
// them (cell split before, position update after).
//
// Work split.  A warp takes up to 32 particles at a time.  Their float64 work
// is lane-dense (one particle per lane).  The interpolation works on four
// particles at once, one per group of eight lanes: lane u of a group owns the
// stencil column x = u (I = 8; I = 6: x = u for u < 6, lanes 6 and 7 repeat
// lanes 0 and 1 with zero weight; I = 4: x = u mod 4, planes z = u / 4 and
// u / 4 + 2), walks its (y, z) rows with the node's components in one 16-byte
// record, and sums z, then y, in registers; the groups then add their lanes
// (three butterfly steps per value).
//
// Why: a warp-wide load is then four runs of I consecutive records, which L1
// (and shared memory) serve at about 1.2 cycles per run, and the work that
// does not depend on the stencil size (weights, reductions, the stage-2
// point, addresses) is shared by four particles.  One warp per particle, the
// split this replaced, spent about 145 instructions per stencil (I = 6) of
// which 24 were the contraction's, and read its rows through 8 loads of five
// rows each; this one spends about 60.  Texture fetches of the same rows take
// 2.1 cycles per row on this GPU against 1.23 for plain loads, and mixing the
// two adds their times (measured on an L1-resident region: 44 cycles per
// 216-node stencil with loads, 56 / 68 / 75 with 1/4, 1/2, all rows as texture
// fetches; shared memory 45), so every load is a plain one.
//
// Everything here gives the same bits whatever kernel runs it, with one
// exception: the order of the sums depends on the stencil and, for float32 I = 6
// and 8, on whether derivatives are summed beside u (contract).
#pragma once

#include <type_traits>

#include <cuda.h>   // CUtensorMap (type only; the library does not link the driver API)

#include "internal.cuh"
#include "six_lanes.h"

namespace trk {

constexpr int NT = 128;           // threads per CTA of the block and batched kernels
constexpr int NW = NT / 32;       // warps per CTA
constexpr int PB = NT;            // particles per batch (32 per warp)

// ---------------------------------------------------------------------------
// Weight polynomials
// ---------------------------------------------------------------------------
template <typename T, class A>
__device__ __forceinline__ const CoefTable<T>& table(const A& a)
{
    if constexpr (sizeof(T) == 4) return a.cf;
    else return a.cd;
}

template <typename T, int DEG>
struct Row {
    T c[DEG + 1];
};

template <typename T, int DEG>
__device__ __forceinline__ Row<T, DEG> load_row(const T (&tab)[TRK_TAB_MAX_I][TRK_TAB_MAX_DEG], int i)
{
    Row<T, DEG> r;
#pragma unroll
    for (int d = 0; d <= DEG; ++d) r.c[d] = tab[i][d];
    return r;
}

template <typename T, int DEG>
__device__ __forceinline__ T horner(const Row<T, DEG>& r, T s)
{
    T acc = r.c[DEG];
#pragma unroll
    for (int d = DEG - 1; d >= 0; --d) acc = fma(acc, s, r.c[d]);
    return acc;
}

// n consecutive weights of a group's buffer (the same for every lane of the
// group) by 16-byte loads where the run starts on a 16-byte boundary
template <int n, typename T>
__device__ __forceinline__ void bcast_load(const T* p, T (&w)[n])
{
    static_assert(n % 2 == 0, "runs of even length");
    if constexpr (sizeof(T) == 4) {
#pragma unroll
        for (int i = 0; i + 4 <= n; i += 4) {
            const float4 v = *reinterpret_cast<const float4*>(p + i);
            w[i] = v.x;
            w[i + 1] = v.y;
            w[i + 2] = v.z;
            w[i + 3] = v.w;
        }
        if constexpr (n % 4 == 2) {
            const float2 v = *reinterpret_cast<const float2*>(p + n - 2);
            w[n - 2] = v.x;
            w[n - 1] = v.y;
        }
    } else {
#pragma unroll
        for (int i = 0; i < n; i += 2) {
            const double2 v = *reinterpret_cast<const double2*>(p + i);
            w[i] = v.x;
            w[i + 1] = v.y;
        }
    }
}

// ---------------------------------------------------------------------------
// Lane map and weights of a group of eight lanes
// ---------------------------------------------------------------------------
// Sixteen lanes (RK2, I = 6 float32): the eight of a half h own the x columns
// of the rows y = h, h + 2, h + 4.  Six lanes (steps, I = 6 float64): five groups
// and two lanes that repeat lanes 24 and 25 (six_lanes.h).
template <int I, int GL = 8>
struct LaneMap {
    static_assert(GL == 8 || I == 6, "six or sixteen lanes: I = 6");
    static constexpr int YS = GL == 16 ? 2 : 1; // rows along y per lane: y0, y0 + YS, ...
    static constexpr int NY = I / YS;
    static constexpr int NZ = I == 4 ? 2 : I;   // planes along z per lane: z0, z0 + ZS, ...
    static constexpr int ZS = I == 4 ? 2 : 1;
    int x, y0, z0;
    bool act;                                   // false: a repeated column (zero weight)
    __device__ __forceinline__ explicit LaneMap(int lane)
    {
        const int u = GL == 6 ? SixLanes(lane).u : lane & 7;
        x = I == 8 ? u : (I == 6 ? (u < 6 ? u : u - 6) : (u & 3));
        y0 = GL == 16 ? (lane >> 3 & 1) : 0;
        z0 = I == 4 ? u >> 2 : 0;
        act = GL == 6 || I != 6 || u < 6;
    }
};

template <typename T, int I, bool D, int GL = 8>
struct Weights {
    static constexpr int NY = LaneMap<I, GL>::NY, NZ = LaneMap<I, GL>::NZ;
    T w1, dw1;
    T w2[GL == 16 ? 4 : NY], w3[NZ];
    T dw2[D ? NY : 1], dw3[D ? NZ : 1];
};

// Lane u evaluates the weight of node i = x for the three axes by Horner's
// rule; axes 2 and 3 are exchanged through the group's buffer wb (axis 2 at 0,
// axis 3 at 8, their derivatives at 16 and 24; I = 4: axis 3 in the order 0, 2,
// 1, 3, so that a lane's planes are adjacent).  Successive calls of a warp
// alternate between two buffers, so one __syncwarp per call orders them.
// Sixteen lanes: half 0 evaluates axis 2, half 1 axis 3; axis 2 is stored in the
// order 0, 2, 4, -, 1, 3, 5, so that a half's rows are adjacent.
template <typename T, int I, int DEG, bool D, int GL = 8>
struct Basis {
    Row<T, DEG> r, dr;
    __device__ __forceinline__ void init(const CoefTable<T>& tb, const LaneMap<I, GL>& m)
    {
        r = load_row<T, DEG>(tb.c, m.x);
        if (D) dr = load_row<T, DEG>(tb.d, m.x);
    }
    __device__ __forceinline__ void eval(T s1, T s2, T s3, const LaneMap<I, GL>& m, T* wb, Weights<T, I, D, GL>& w) const
    {
        if constexpr (GL == 16) {
            static_assert(!D, "values only");
            const T a1 = horner(r, s1);
            wb[m.y0 ? 8 + m.x : (m.x & 1) * 4 + (m.x >> 1)] = horner(r, m.y0 ? s3 : s2);
            w.w1 = m.act ? a1 : (T)0;
            __syncwarp();
            bcast_load(wb + 4 * m.y0, w.w2);
            bcast_load(wb + 8, w.w3);
            return;
        }
        const T a1 = horner(r, s1), a2 = horner(r, s2), a3 = horner(r, s3);
        // (repeated columns store the values their originals store)
        const int x3 = I == 4 ? (m.x & 1) * 2 + (m.x >> 1) : m.x;
        wb[m.x] = a2;
        wb[8 + x3] = a3;
        w.w1 = m.act ? a1 : (T)0;
        if constexpr (D) {
            const T d1 = horner(dr, s1);
            wb[16 + m.x] = horner(dr, s2);
            wb[24 + x3] = horner(dr, s3);
            w.dw1 = m.act ? d1 : (T)0;
        }
        __syncwarp();
        bcast_load(wb, w.w2);
        bcast_load(wb + 8 + 2 * m.z0, w.w3);
        if constexpr (D) {
            bcast_load(wb + 16, w.dw2);
            bcast_load(wb + 24 + 2 * m.z0, w.dw3);
        }
    }
};

// ---------------------------------------------------------------------------
// Stencil loaders: ld(r, z, v) = components of the lane's node in row r and its
// z-th plane
// ---------------------------------------------------------------------------
// Records in global memory.  A cell c in
// [0, N) plus one is at least PAD - 1 > I / 2 nodes inside the ghost-padded
// array, so a stencil is a box of fixed offsets from its first node.
template <int RW, int NC>
struct RecordLd {
    const float* p;        // the lane's first node
    int NP, NP2;           // record strides from row to row and from plane to plane of the lane
    __device__ __forceinline__ void operator()(int r, int z, float (&v)[NC]) const
    {
        const int off = z * NP2 + r * NP;
        if constexpr (RW == 4) {
            const float4 q = __ldg(reinterpret_cast<const float4*>(p) + off);
            const float w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
            for (int k = 0; k < NC; ++k) v[k] = w[k];
        } else {
            static_assert(NC == 1, "one component per 4-byte record");
            v[0] = __ldg(p + off);
        }
    }
};

// Component-major float64 field: components k >= kc read component kc - 1
template <int NC>
struct PlaneLd {
    const double* p;
    int64_t plane;
    int NP, NP2, kc;
    __device__ __forceinline__ void operator()(int r, int z, double (&v)[NC]) const
    {
        const int off = z * NP2 + r * NP;
#pragma unroll
        for (int k = 0; k < NC; ++k) v[k] = __ldg(p + (int64_t)(k < kc ? k : kc - 1) * plane + off);
    }
};

// Loader of the stencil whose first node has the padded index `base`, for the
// component chunk ch (NC components of it)
template <typename T, int I, int STORE, int RW, int NC, int GL>
__device__ __forceinline__ auto global_ld(const FieldView& f, int base, int ch, const LaneMap<I, GL>& m)
{
    constexpr int ZS = LaneMap<I, GL>::ZS, YS = LaneMap<I, GL>::YS;
    const int64_t n = (int64_t)base + m.x + m.y0 * f.NP + m.z0 * f.NP * f.NP;
    if constexpr (STORE == ST_F64)
        return PlaneLd<NC>{f.f64 + (int64_t)ch * NC * f.plane + n, f.plane, YS * f.NP, ZS * f.NP * f.NP, f.C - ch * NC};
    else
        return RecordLd<RW, NC>{f.rec + ((int64_t)ch * f.plane + n) * RW, YS * f.NP, ZS * f.NP * f.NP};
}

// A staged halo in shared memory: pitches P from row to row and PL from plane
// to plane of the lane (elements), float64: component pitch SC
template <typename T, int STORE, int RW, int NC, int P, int PL, int SC>
struct HaloLd {
    const void* p;         // the lane's first node
    __device__ __forceinline__ void operator()(int r, int z, T (&v)[NC]) const
    {
        if constexpr (STORE == ST_F64) {
#pragma unroll
            for (int k = 0; k < NC; ++k) v[k] = reinterpret_cast<const double*>(p)[k * SC + z * PL + r * P];
        } else if constexpr (RW == 4) {
            const float4 q = reinterpret_cast<const float4*>(p)[z * PL + r * P];
            const float w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
            for (int k = 0; k < NC; ++k) v[k] = w[k];
        } else {
            v[0] = reinterpret_cast<const float*>(p)[z * PL + r * P];
        }
    }
};

// A lane's stencil, its HR rows held in registers (re-used by RK2's second stage)
template <typename T, int I, int NC, int HR>
struct HeldLd {
    const T (&f)[HR][LaneMap<I>::NZ][NC];   // (NZ: the same for either group size)
    __device__ __forceinline__ void operator()(int r, int z, T (&v)[NC]) const
    {
#pragma unroll
        for (int k = 0; k < NC; ++k) v[k] = f[r][z][k];
    }
};

template <typename T, int I, int NC, int HR, class LD>
__device__ __forceinline__ void load_rows(const LD& ld, T (&f)[HR][LaneMap<I>::NZ][NC])
{
#pragma unroll
    for (int r = 0; r < HR; ++r)
#pragma unroll
        for (int z = 0; z < LaneMap<I>::NZ; ++z) ld(r, z, f[r][z]);
}

// ---------------------------------------------------------------------------
// Contraction: z then y in the lane, then x over the group.
//   D = false: out[k] = u_k
//   D = true:  out[k] = u_k, out[NC + 3k + j] = du_k / dt_j
// ---------------------------------------------------------------------------
// Sums v[0..n) over the group's eight lanes, in three exchanges that halve the
// values a lane carries (n = 12: 11 shuffles instead of 36; the shuffles share
// the data path the stencils come through).  The lane is left with the sums
// base .. base + count - 1 in v[0], v[1], ...
template <typename T, int n>
struct GroupSums {
    static constexpr int m1 = (n + 1) / 2, m2 = (m1 + 1) / 2, m3 = (m2 + 1) / 2;
    T v[m3];
    int base, count;

    template <int M, int O, int IN>
    __device__ __forceinline__ static void exchange(T (&x)[IN], int lane, int& base, int& count)
    {
        constexpr int h = (M + 1) / 2;
        const bool hi = lane & O;
#pragma unroll
        for (int i = 0; i < h; ++i) {
            const T a = x[i], b = i + h < M ? x[i + h < IN ? i + h : 0] : (T)0;
            x[i] = (hi ? b : a) + __shfl_xor_sync(0xffffffffu, hi ? a : b, O);
        }
        base += hi ? h : 0;
        count = hi ? max(count - h, 0) : min(count, h);
    }
    __device__ __forceinline__ GroupSums(T (&x)[n], int lane)
    {
        base = 0;
        count = n;
        exchange<n, 4>(x, lane, base, count);
        exchange<m1, 2>(x, lane, base, count);
        exchange<m2, 1>(x, lane, base, count);
#pragma unroll
        for (int i = 0; i < m3; ++i) v[i] = x[i];
    }
    // sum i in every lane of the group
    template <int i>
    __device__ __forceinline__ T all(int lane) const
    {
        constexpr bool h1 = i >= m1;
        constexpr int i1 = i - (h1 ? m1 : 0);
        constexpr bool h2 = i1 >= m2;
        constexpr int i2 = i1 - (h2 ? m2 : 0);
        constexpr bool h3 = i2 >= m3;
        return __shfl_sync(0xffffffffu, v[i2 - (h3 ? m3 : 0)], (lane & 24) | (h1 ? 4 : 0) | (h2 ? 2 : 0) | (h3 ? 1 : 0));
    }
    // the sums from `first` on to the particle's slots
    __device__ __forceinline__ void put(T* kb, int first, bool live) const
    {
#pragma unroll
        for (int i = 0; i < m3; ++i)
            if (live && i < count && base + i >= first) kb[base + i - first] = v[i];
    }
};

// the same for three values over a group of sixteen (after join_halves): half 0 is
// left with value 0 (lanes u < 4) or 1 (u >= 4), half 1 with value 2 (u < 4)
template <typename T>
struct HalfSums {
    T v;
    int which;   // -1: none
    __device__ __forceinline__ HalfSums(const T (&x)[3], int lane)
    {
        const bool hi = lane & 4, second = lane & 8;
        // half 1 adds value 2 in all its lanes
        const T give = second ? x[0] : (hi ? x[0] : x[1]), keep = second ? x[0] : (hi ? x[1] : x[0]);
        v = keep + __shfl_xor_sync(0xffffffffu, give, 4);
        v += __shfl_xor_sync(0xffffffffu, v, 2);
        v += __shfl_xor_sync(0xffffffffu, v, 1);
        which = lane & 3 ? -1 : (second ? (hi ? -1 : 2) : (hi ? 1 : 0));
    }
    template <int i>
    __device__ __forceinline__ T all(int lane) const
    {
        return __shfl_sync(0xffffffffu, v, (lane & 16) | (i == 0 ? 0 : (i == 1 ? 4 : 8)));
    }
    __device__ __forceinline__ void put(T* kb, int, bool live) const
    {
        if (live && which >= 0) kb[which] = v;
    }
};

// the same for three values over a group of six, in the order GroupSums has for
// I = 6, ((x0 + x4) + x2) + ((x1 + x5) + x3): lanes 2q and 2q + 1 add the even and
// the odd columns of value q
template <typename T>
struct TrioSums {
    SixLanes at;
    T v;
    __device__ __forceinline__ TrioSums(const T (&x)[3], int lane) : at(lane)
    {
        const int q = at.value();
        auto value = [&](int i) { return i == 0 ? x[0] : (i == 1 ? x[1] : x[2]); };
        const T own = value(q);
        const T c1 = __shfl_sync(0xffffffffu, value(at.next(2)), at.partner(1));
        const T c2 = __shfl_sync(0xffffffffu, value(at.next(1)), at.partner(2));
        v = (q == 1 ? c1 : own) + (q == 2 ? c1 : c2);
        v += q == 0 ? c1 : (q == 1 ? own : c2);
        v += __shfl_xor_sync(0xffffffffu, v, 1);
    }
    template <int i>
    __device__ __forceinline__ T all(int) const
    {
        return __shfl_sync(0xffffffffu, v, at.holder(i));
    }
    __device__ __forceinline__ void put(T* kb, int, bool live) const
    {
        if (live && (at.u & 1) == 0) kb[at.value()] = v;
    }
};

// i-th term of a sum over n nodes taken from the ends inwards (0, n-1, 1, ...):
// the small outer terms first, so that they are rounded while the partial sum is small
__host__ __device__ constexpr int inward(int i, int n) { return i % 2 == 0 ? i / 2 : n - 1 - i / 2; }

// a = w v (first) or a + w v, component-wise.  PACK: two float32 components per
// instruction, rounded as single ones are; for gradients of I = 4, 6 from slabs
// and for a warp per particle, whose registers hold the pairs (256^3, 2^21
// particles, gradients: I = 6 431 -> 419 us; I = 8 RK2, 2^20: 592 -> 582; values
// from slabs spill: I = 6 RK2 379 -> 462).
template <bool PACK, int NC>
__device__ __forceinline__ void axpy(bool first, float w, const float (&v)[NC], float (&a)[NC])
{
    if constexpr (PACK) {
#pragma unroll
        for (int k = 0; k + 1 < NC; k += 2) {
            if (first)
                asm("{.reg .b64 p, q, r;\n mov.b64 p, {%2, %2};\n mov.b64 q, {%3, %4};\n mul.rn.f32x2 r, p, q;\n"
                    "mov.b64 {%0, %1}, r;}"
                    : "=f"(a[k]), "=f"(a[k + 1])
                    : "f"(w), "f"(v[k]), "f"(v[k + 1]));
            else
                asm("{.reg .b64 p, q, r;\n mov.b64 p, {%2, %2};\n mov.b64 q, {%3, %4};\n mov.b64 r, {%0, %1};\n"
                    "fma.rn.f32x2 r, p, q, r;\n mov.b64 {%0, %1}, r;}"
                    : "+f"(a[k]), "+f"(a[k + 1])
                    : "f"(w), "f"(v[k]), "f"(v[k + 1]));
        }
        if constexpr (NC % 2) a[NC - 1] = first ? w * v[NC - 1] : fmaf(w, v[NC - 1], a[NC - 1]);
    } else {
#pragma unroll
        for (int k = 0; k < NC; ++k) a[k] = first ? w * v[k] : fmaf(w, v[k], a[k]);
    }
}
template <bool, int NC>
__device__ __forceinline__ void axpy(bool first, double w, const double (&v)[NC], double (&a)[NC])
{
#pragma unroll
    for (int k = 0; k < NC; ++k) a[k] = first ? w * v[k] : fma(w, v[k], a[k]);
}

// z sums of one row: pv (and pd with the derivative weights)
template <typename T, int I, int NC, bool D, int GL, bool PACK, class LD>
__device__ __forceinline__ void row_sums(const LD& ld, int r, const Weights<T, I, D, GL>& w, T (&pv)[NC], T (&pd)[NC])
{
    constexpr int NZ = LaneMap<I>::NZ;
#pragma unroll
    for (int zz = 0; zz < NZ; ++zz) {
        const int z = inward(zz, NZ);
        T v[NC];
        ld(r, z, v);
        axpy<PACK, NC>(zz == 0, w.w3[z], v, pv);
        if constexpr (D) axpy<PACK, NC>(zz == 0, w.dw3[z], v, pd);
    }
}

// the lane's column: out as above, to be summed over the group (GroupSums).
// The rows are summed from the ends inwards; float32 values of I = 8 in the
// order a whole warp on one particle sums them in (run_direct_warp): parts
// {0, 4}, {1, 5}, {6, 2}, {7, 3}, then (p0 + p2) + (p1 + p3); of I = 6 in the
// order of sixteen lanes: rows 0, 4, 2 plus rows 1, 5, 3.  With derivatives the
// order stays from the ends inwards.  So u of a step that also writes gradients, and
// the u that takes the adjoint to its stage-2 point, differ from the plain step's
// in the last bits (each is as far from the exact sum); X*, which is u times dt, can
// then lie on the other side of a face, where the interpolation has the other cell's
// polynomial.  Summing u in the value's order there as well was measured (256^3):
// batched sets 7.1 -> 7.7 ms and the gradients' error 5.1e-7 -> 5.4e-7, or, with the
// rows from the ends inwards and u in parts, 11.7 ms, and the adjoint 36 -> 60 ms.
template <typename T, int I, int NC, bool D, int GL, bool PACK, class LD>
__device__ __forceinline__ void contract(const LD& ld, const Weights<T, I, D, GL>& w, T (&out)[D ? 4 * NC : NC])
{
    constexpr int NY = LaneMap<I, GL>::NY;
    T a[NC], b[NC], c[NC], pv[NC], pd[NC];
    if constexpr (sizeof(T) == 4 && I == 6 && !D) {
        T half[NC];
#pragma unroll
        for (int h = 0; h < (GL == 16 ? 1 : 2); ++h) {
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                const int r = GL == 16 ? inward(q, 3) : h + 2 * inward(q, 3);
                row_sums<T, I, NC, D, GL, PACK>(ld, r, w, pv, pd);
                axpy<PACK, NC>(q == 0, w.w2[r], pv, half);
            }
#pragma unroll
            for (int k = 0; k < NC; ++k) a[k] = h ? a[k] + half[k] : half[k];
        }
    } else if constexpr (sizeof(T) == 4 && I == 8 && !D) {
        T part[NC], pair[NC];
#pragma unroll
        for (int q = 0; q < 2; ++q)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int p = q + 2 * h, r0 = h ? p + 4 : p, r1 = h ? p : p + 4;
                row_sums<T, I, NC, D, GL, PACK>(ld, r0, w, pv, pd);
#pragma unroll
                for (int k = 0; k < NC; ++k) part[k] = w.w2[r0] * pv[k];
                row_sums<T, I, NC, D, GL, PACK>(ld, r1, w, pv, pd);
#pragma unroll
                for (int k = 0; k < NC; ++k) {
                    part[k] = fma(w.w2[r1], pv[k], part[k]);
                    pair[k] = h ? pair[k] + part[k] : part[k];
                    if (h) a[k] = q ? a[k] + pair[k] : pair[k];
                }
            }
    } else {
#pragma unroll
        for (int rr = 0; rr < NY; ++rr) {
            const int r = inward(rr, NY);
            row_sums<T, I, NC, D, GL, PACK>(ld, r, w, pv, pd);
            axpy<PACK, NC>(rr == 0, w.w2[r], pv, a);
            if constexpr (D) {
                axpy<PACK, NC>(rr == 0, w.dw2[r], pv, b);
                axpy<PACK, NC>(rr == 0, w.w2[r], pd, c);
            }
        }
    }
#pragma unroll
    for (int k = 0; k < NC; ++k) {
        out[k] = GL == 16 ? a[k] : w.w1 * a[k];   // (sixteen lanes: join_halves multiplies)
        if constexpr (D) {
            out[NC + 3 * k] = w.dw1 * a[k];
            out[NC + 3 * k + 1] = w.w1 * b[k];
            out[NC + 3 * k + 2] = w.w1 * c[k];
        }
    }
}

// ---------------------------------------------------------------------------
// Per-warp shared memory
// ---------------------------------------------------------------------------
template <int MODE>
__host__ __device__ constexpr bool is_ab() { return MODE == MODE_AB2 || MODE == MODE_AB2_D; }
template <int MODE>
__host__ __device__ constexpr bool is_step() { return MODE == MODE_RK2 || is_ab<MODE>(); }
template <int MODE>
__host__ __device__ constexpr bool is_deriv()
{
    return MODE == MODE_INTERP_DERIV || MODE == MODE_AB2_D || MODE == MODE_ADJ;
}
// a second stage one step along (its halo has a margin of one cell)
template <int MODE>
__host__ __device__ constexpr bool two_stages() { return MODE == MODE_RK2 || MODE == MODE_ADJ; }

// values handed from the groups to the particle's lane: k1 and k2 (RK2), u
// (AB, interpolation), u and its derivatives; adjoint: J(X), J(X*), t*, the
// cell of X* (in units of the cell width)
template <int MODE, int NC>
__host__ __device__ constexpr int result_count()
{
    return MODE == MODE_RK2 ? 6 : (MODE == MODE_ADJ ? 22 : (is_deriv<MODE>() ? 4 * NC : NC));
}

__host__ __device__ constexpr size_t align32(size_t x) { return (x + 31) & ~size_t(31); }

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

template <int BYTES>
__device__ __forceinline__ void cp_async(void* dst, const void* src)
{
    if constexpr (BYTES == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(smem_addr(dst)), "l"(src) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(smem_addr(dst)), "l"(src), "n"(BYTES)
                     : "memory");
}

__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

template <typename T, int MODE, int NC>
struct WarpPlan {
    static constexpr int KS = (result_count<MODE, NC>() + 3) / 4 * 4;                      // values per particle
    static constexpr size_t rec = 0;                                                       // [2][32] records
    static constexpr size_t k = align32(rec + 2 * 32 * 4 * sizeof(T));                     // [32][KS]
    static constexpr size_t w = align32(k + 32 * KS * sizeof(T));                          // [2][NG groups][WB]
    static constexpr int WB = is_deriv<MODE>() ? 40 : 24;                                  // groups 8 banks apart
    static constexpr bool HAS_X = is_step<MODE>() || MODE == MODE_ADJ;
    static constexpr int NG = sizeof(T) == 8 ? 5 : 4;
    static constexpr size_t x = align32(w + 2 * NG * WB * sizeof(T));                       // [3][32] positions (steps), lambda
    static constexpr size_t rhs = align32(x + (HAS_X ? 3 * 32 * sizeof(double) : 0));      // [3 HIST][32] AB history
    static constexpr int HIST = MODE == MODE_AB2 ? AB_MAX_HIST : (MODE == MODE_AB2_D ? 1 : 0);   // entries (AB2_D: order 2)
    static constexpr size_t total = align32(rhs + 3 * HIST * 32 * sizeof(float));
};

// ---------------------------------------------------------------------------
// Halo of a cell block (block kernels): H^3 nodes from G nodes below the
// block's first cell, with one more layer on each side for RK2's stage-2 point.
// Dense rows (pitch P; float64 an even number of elements, the halo XOFF in,
// so that a tensor copy starts on 16 bytes).
// ---------------------------------------------------------------------------
template <typename T, int I, int MODE, int NC, int RW>
struct HaloGeom {
    static constexpr int MARGIN = two_stages<MODE>() ? 1 : 0;
    static constexpr HaloBox B = halo_box(I, MARGIN, sizeof(T) == 8);
    static constexpr int H = B.H, G = B.G, P = B.P, XOFF = B.XOFF;
    static constexpr int PL = P * H, SC = PL * H;
    static constexpr size_t bytes = align32(sizeof(T) == 8 ? (size_t)NC * SC * 8 : (size_t)SC * RW * 4);
};

// Slabs: the halo as k_slabs stages it, cut along x1 into slabs of SW nodes
// aligned to SW, each a dense box [H][H][SW] of 16-byte records.  A group's
// lanes read consecutive x1: eight banks groups apart whichever slabs they lie
// in (SW = 8: 128-byte rows; I = 4, whose groups read rows of two planes at
// once: 64-byte rows, and H is odd).
template <int I, int MODE>
struct SlabGeom {
    static constexpr HaloBox B = halo_box(I, two_stages<MODE>() ? 1 : 0, false);
    static constexpr int H = B.H, G = B.G;
    static constexpr int SW = slab_width(I), SPT = BLK / SW;       // slabs a block is wide
    static constexpr int X0 = -((G + SW - 1) / SW) * SW;          // first slab's x1 relative to the block
    static constexpr int NSL = (H - G - X0 + SW - 1) / SW;        // slabs a block's halo spans
    static constexpr size_t bytes = (size_t)H * H * SW * 16, slot = (bytes + 127) / 128 * 128;
    static_assert(SW == 8 || H % 2 == 1, "two planes in distinct banks");
};

// where a group's stencil comes from
enum { SRC_GLOBAL = 0, SRC_HALO = 1, SRC_SLABS = 2 };
struct Place {
    const unsigned char* halo;   // SRC_HALO: the staged halo; SRC_SLABS: slot 0 of the slab ring
    int slab;                    // SRC_SLABS: sequence number of the block's first slab
    int c[3];                    // the particle's cell
};

// ---------------------------------------------------------------------------
// P1: lane-dense.  The record of the lane's particle: the one the binning made
// (grouped position j), or split here from the position of particle src.
// ---------------------------------------------------------------------------
template <typename T>
__device__ __forceinline__ PRec<T> particle_record(const BlockArgs& a, int64_t j, int64_t src, bool valid)
{
    PRec<T> rec;
    rec.t[0] = rec.t[1] = rec.t[2] = (T)0;
    rec.cell = cell_as<T>(0);
    if (!valid) return rec;
    if (a.rec_in) return reinterpret_cast<const PRec<T>*>(a.rec_in)[j];
    return split_record<T>(a.g, a.np, a.pos_in, src, a.flags);
}

// The lane's particle state that the update needs, on its way to shared memory
// while the particle is interpolated (cp.async; the lane reads its own copies).
template <typename T, int MODE, int NC>
__device__ __forceinline__ void fetch_state(const BlockArgs& a, int64_t src, bool valid, unsigned char* ws, int lane)
{
    using WPl = WarpPlan<T, MODE, NC>;
    if constexpr (WPl::HAS_X) {   // (the adjoint's pos_in is lambda, src the caller index)
        if (!valid) return;
#pragma unroll
        for (int ax = 0; ax < 3; ++ax)
            cp_async<8>(ws + WPl::x + (ax * 32 + lane) * 8, a.pos_in + ax * a.np + src);
        if constexpr (is_ab<MODE>()) {   // the valid history rows
            const int rows = 3 * min(a.history_valid, a.ab_order - 1);
            for (int r = 0; r < rows; ++r) cp_async<4>(ws + WPl::rhs + (r * 32 + lane) * 4, a.rhs_in + r * a.np + src);
        }
    }
}

// Lanes per particle and rows of the RK2 stencil that a lane holds in registers
// between the stages: its second stage then gathers these only where X* left
// the cell.  I = 4 (8 nodes per lane): always.  I = 6 (36 nodes, 108 registers of
// values): gathered from global memory, by sixteen lanes that hold 18 nodes each,
// sixteen warps per SM (256^3 float32, RK2, us per step at 1/64 particle per cell:
// 120, against 145 with eight lanes and eight warps that hold 36 nodes, 158 with
// sixteen warps that gather twice; 512^3, 1.5e6: 671, 797); from slabs in shared
// memory eight lanes without held rows, which issue fewer instructions (1/8 per
// cell: 633 against 710 with sixteen lanes; 1/16: 377, 400, 12 warps with held
// rows 407).  I = 8 would take 256 registers (run_direct_warp holds them),
// float64 twice these: none.  float64 I = 6 steps are bound by the float64 pipe,
// which idle lanes hold as long as busy ones: six lanes per particle, five
// particles per warp (128^3, 4e5 tracers, RK2: 1410 us per step; eight lanes, two
// of them idle: 1770).
template <typename T, int I, int MODE, int SRC>
__host__ __device__ constexpr int group_lanes()
{
    if (I != 6 || SRC != SRC_GLOBAL) return 8;
    return sizeof(T) == 8 ? (MODE == MODE_RK2 || MODE == MODE_AB2 ? 6 : 8) : (MODE == MODE_RK2 ? 16 : 8);
}
template <typename T, int I, int MODE, int SRC>
__host__ __device__ constexpr int held_rows()
{
    if (group_lanes<T, I, MODE, SRC>() == 16) return 3;
    return sizeof(T) == 8 || I != 4 ? 0 : 4;
}

// The halves of a group of sixteen: half 0 goes on with values 0 and 1, half 1
// with value 2 (then 0), so that the sums over x take three shuffles, not four.
template <typename T>
__device__ __forceinline__ void join_halves(T (&k)[3], T w1, int lane)
{
    const bool hi = lane & 8;
    const T r = __shfl_xor_sync(0xffffffffu, hi ? k[0] : k[2], 8), r1 = __shfl_xor_sync(0xffffffffu, k[1], 8);
    k[0] = w1 * ((hi ? k[2] : k[0]) + r);
    k[1] = w1 * (k[1] + r1);
}

// One stage: contract the stencil of ld at the offsets s (less 1/2) from the
// cell's centre; the rows held in f are loaded if `fresh`.
template <typename T, int I, int DEG, int NC, bool D, int HR, int GL, class LD>
__device__ __forceinline__ void interpolate_stage(const LD& ld, T s1, T s2, T s3, T* wb, bool fresh,
                                                  const LaneMap<I, GL>& m, const Basis<T, I, DEG, D, GL>& B,
                                                  T (&f)[HR > 0 ? HR : 1][LaneMap<I>::NZ][NC], T (&k)[D ? 4 * NC : NC],
                                                  int lane)
{
    Weights<T, I, D, GL> w;
    if constexpr (HR > 0) {
        static_assert(HR == (LaneMap<I, GL>::NY), "all of the lane's rows");
        if (fresh) load_rows<T, I, NC, HR>(ld, f);
        __syncwarp();
        B.eval(s1, s2, s3, m, wb, w);
        contract<T, I, NC, D, GL, false>(HeldLd<T, I, NC, HR>{f}, w, k);
    } else {
        B.eval(s1, s2, s3, m, wb, w);
        contract<T, I, NC, D, GL, false>(ld, w, k);
    }
    if constexpr (GL == 16) join_halves(k, w.w1, lane);
}

// ---------------------------------------------------------------------------
// Q: a group interpolates its particle (offsets t, stencil at `at`), component
// chunk ch; the results go to the particle's slots kb.  live: false for an
// empty slot.
// ---------------------------------------------------------------------------
template <typename T, int I, int DEG, int MODE, int NC, int STORE, int RW, int SRC, int NS = 1>
__device__ __forceinline__ void interpolate_group(const BlockArgs& a, const Place& at, int ch, const T (&t)[3], bool live,
                                                  int lane,
                                                  const Basis<T, I, DEG, is_deriv<MODE>(), group_lanes<T, I, MODE, SRC>()>& B,
                                                  const LaneMap<I, group_lanes<T, I, MODE, SRC>()>& m, T* wb0, T* wb1,
                                                  bool odd, T* kb)
{
    constexpr int GL = group_lanes<T, I, MODE, SRC>(), YS = LaneMap<I, GL>::YS;
    using Sums = std::conditional_t<GL == 16, HalfSums<T>,
                                    std::conditional_t<GL == 6, TrioSums<T>, GroupSums<T, is_deriv<MODE>() ? 4 * NC : NC>>>;
    constexpr bool D = is_deriv<MODE>(), HALO = SRC != SRC_GLOBAL;
    constexpr int LO = I / 2 - 1, ZS = LaneMap<I>::ZS, G = LO + (two_stages<MODE>() ? 1 : 0);
    // the stencil of the cell displaced by d from the particle's, in the staged halo
    auto halo_ld = [&](int d1, int d2, int d3) {
        const int r1 = (at.c[0] & 7) + d1 + G - LO, r2 = (at.c[1] & 7) + d2 + G - LO + m.y0, r3 = (at.c[2] & 7) + d3 + G - LO + m.z0;
        if constexpr (SRC == SRC_SLABS) {   // the lane's slab and column
            using SG = SlabGeom<I, MODE>;
            const int x = r1 + m.x - SG::G - SG::X0;
            const int row = r3 * SG::H + r2;
            return HaloLd<T, STORE, RW, NC, YS * SG::SW, ZS * SG::H * SG::SW, 0>{
                at.halo + (unsigned)(at.slab + x / SG::SW) % NS * SG::slot + (row * SG::SW + x % SG::SW) * 16};
        } else {
            using HG = HaloGeom<T, I, MODE, NC, RW>;
            const int e = r3 * HG::PL + r2 * HG::P + (r1 + m.x) + HG::XOFF;
            return HaloLd<T, STORE, RW, NC, YS * HG::P, ZS * HG::PL, HG::SC>{at.halo + e * (STORE == ST_F64 ? 8 : 4 * RW)};
        }
    };
    auto node_of = [&](int c1, int c2, int c3) { return (int)padded_index(a.f.NP, c1 - LO, c2 - LO, c3 - LO); };
    auto glob_ld = [&](int node) { return global_ld<T, I, STORE, RW, NC, GL>(a.f, node, ch, m); };
    if constexpr (!two_stages<MODE>()) {
        Weights<T, I, D, GL> w;
        B.eval(t[0] - (T)0.5, t[1] - (T)0.5, t[2] - (T)0.5, m, odd ? wb1 : wb0, w);
        constexpr bool PACK = D && I <= 6 && SRC == SRC_SLABS;
        T out[D ? 4 * NC : NC];
        if constexpr (HALO) contract<T, I, NC, D, GL, PACK>(halo_ld(0, 0, 0), w, out);
        else contract<T, I, NC, D, GL, PACK>(glob_ld(node_of(at.c[0], at.c[1], at.c[2])), w, out);
        if constexpr (MODE == MODE_INTERP_DERIV) {   // the derivatives only
            T der[3 * NC];
#pragma unroll
            for (int i = 0; i < 3 * NC; ++i) der[i] = out[NC + i];
            GroupSums<T, 3 * NC>(der, lane).put(kb + NC, 0, live);
        } else {
            Sums(out, lane).put(kb, 0, live);
        }
    } else {
        const T dtid = (T)(a.dt * a.g.inv_delta);
        constexpr int HR = MODE == MODE_RK2 ? held_rows<T, I, MODE, SRC>() : 0;
        constexpr int NOUT = D ? 4 * NC : NC;
        T f[HR > 0 ? HR : 1][LaneMap<I>::NZ][NC];
        T k1[NOUT], k2[NOUT];
        if constexpr (HALO)
            interpolate_stage<T, I, DEG, NC, D, HR, GL>(halo_ld(0, 0, 0), t[0] - (T)0.5, t[1] - (T)0.5, t[2] - (T)0.5, wb0, true, m, B, f, k1, lane);
        else
            interpolate_stage<T, I, DEG, NC, D, HR, GL>(glob_ld(node_of(at.c[0], at.c[1], at.c[2])), t[0] - (T)0.5, t[1] - (T)0.5, t[2] - (T)0.5, wb0, true, m, B, f, k1, lane);
        const Sums s1(k1, lane);
        const T u1[3] = {s1.template all<0>(lane), s1.template all<1>(lane), s1.template all<2>(lane)};
        s1.put(kb, MODE == MODE_RK2 ? 0 : 3, live);
        // stage-2 point, cell-relative: t* = t + dt k1 / delta
        T ts[3];
        int d[3];
#pragma unroll
        for (int ax = 0; ax < 3; ++ax) {
            ts[ax] = fma(dtid, u1[ax], t[ax]);
            const T fl = floor(ts[ax]);
            d[ax] = (int)fl;
            ts[ax] -= fl;
        }
        // X* at most one cell away lies in the halo, or inside the ghost layers; farther
        // its cell is wrapped (unsigned: a saturated conversion is far as well)
        const bool moved = (d[0] | d[1] | d[2]) != 0;
        const bool far = (unsigned)d[0] + 1u > 2u || (unsigned)d[1] + 1u > 2u || (unsigned)d[2] + 1u > 2u;
        auto wrap = [&](int ax) { return (int)(((unsigned)at.c[ax] + (unsigned)d[ax]) & (unsigned)a.g.mask); };
        if (far && m.x == 0 && live) atomicOr(a.flags + FLAG_CFL, 1);
        if constexpr (HALO) {
            if (!__any_sync(0xffffffffu, far)) {
                interpolate_stage<T, I, DEG, NC, D, HR, GL>(halo_ld(d[0], d[1], d[2]), ts[0] - (T)0.5, ts[1] - (T)0.5, ts[2] - (T)0.5, wb1, moved, m, B, f, k2, lane);
            } else {   // rare: every group of the warp gathers from global memory (the same values)
                interpolate_stage<T, I, DEG, NC, D, HR, GL>(glob_ld(node_of(wrap(0), wrap(1), wrap(2))), ts[0] - (T)0.5, ts[1] - (T)0.5, ts[2] - (T)0.5, wb1, true, m, B, f, k2, lane);
            }
        } else {
            const int n2 = far ? node_of(wrap(0), wrap(1), wrap(2))
                               : node_of(at.c[0] + d[0], at.c[1] + d[1], at.c[2] + d[2]);
            interpolate_stage<T, I, DEG, NC, D, HR, GL>(glob_ld(n2), ts[0] - (T)0.5, ts[1] - (T)0.5, ts[2] - (T)0.5, wb1, moved, m, B, f, k2, lane);
        }
        const Sums s2(k2, lane);
        if constexpr (MODE == MODE_RK2) {
            s2.put(kb + 3, 0, live);
        } else {   // the Jacobians, t* and the cell of X*
            s2.put(kb + 9, 3, live);
            if (live && (lane & 7) == 0) {
#pragma unroll
                for (int ax = 0; ax < 3; ++ax) kb[18 + ax] = ts[ax];
                kb[21] = cell_as<T>(wrap(0) | wrap(1) << 10 | wrap(2) << 20);
            }
        }
    }
}

// ---------------------------------------------------------------------------
// P3: lane-dense.  Interpolation: write the chunk's outputs of the particle in
// the caller's order.  Steps: float64 update, new key, block counts.
// ---------------------------------------------------------------------------
template <typename T, int MODE, int NC>
__device__ __forceinline__ void write_outputs(const BlockArgs& a, int64_t id, int ch, const unsigned char* ws, int lane)
{
    using WPl = WarpPlan<T, MODE, NC>;
    const T* kb = reinterpret_cast<const T*>(ws + WPl::k) + lane * WPl::KS;
    auto put = [&](int64_t row, double v) {
        if (a.out_f64) reinterpret_cast<double*>(a.out)[row * a.np + id] = v;
        else reinterpret_cast<float*>(a.out)[row * a.np + id] = (float)v;
    };
#pragma unroll
    for (int k = 0; k < NC; ++k) {
        if (ch * NC + k >= a.f.C) continue;
        if constexpr (MODE == MODE_INTERP) {
            put(ch * NC + k, (double)kb[k]);
        } else {
#pragma unroll
            for (int j = 0; j < 3; ++j) put(3 * (ch * NC + k) + j, (double)kb[NC + 3 * k + j] * a.g.inv_delta);
        }
    }
}

// hold: the field did not arrive (FLAG_HALO_TIMEOUT).  The particle stays as it was,
// position and history, and writes no outputs; its key and block count are those of
// its position, so that the next binning still finds every particle once.
template <typename T, int MODE, int NC>
__device__ __forceinline__ void update_particle(const BlockArgs& a, int64_t j, int32_t id, bool valid,
                                                const unsigned char* ws, int lane, bool hold = false)
{
    using WPl = WarpPlan<T, MODE, NC>;
    const unsigned vm = __ballot_sync(0xffffffffu, valid);
    if (!valid) return;
    const T* kb = reinterpret_cast<const T*>(ws + WPl::k) + lane * WPl::KS;
    const double* xs = reinterpret_cast<const double*>(ws + WPl::x) + lane;
    int cn[3];
    bool ok = true;
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
        const double k1 = widen(kb[ax]);
        const double x0 = xs[ax * 32];
        double xn;
        if constexpr (MODE == MODE_RK2) {
            const double k2 = widen(kb[3 + ax]);
            xn = x0 + (0.5 * a.dt) * (k1 + k2);
        } else {   // ABk, order min(k, 1 + history)
            float h[AB_MAX_HIST];   // entries beyond the valid ones are zero
#pragma unroll
            for (int e = 0; e < AB_MAX_HIST; ++e)
                h[e] = e < a.history_valid && e < a.ab_order - 1
                           ? reinterpret_cast<const float*>(ws + WPl::rhs)[(3 * e + ax) * 32 + lane]
                           : 0.0f;
            const int q = min(a.ab_order, a.history_valid + 1);
            const double inc = ab_increment(q, k1, [&](int e) { return widen(h[e]); });
            xn = x0 + a.dt * inc;
            // new history: u_n, then the older entries shifted by one
            a.rhs_out[ax * a.np + j] = hold ? h[0] : (float)k1;
#pragma unroll
            for (int e = 1; e < AB_MAX_HIST; ++e)
                if (e < a.ab_order - 1) a.rhs_out[(3 * e + ax) * a.np + j] = hold ? h[e] : h[e - 1];
            if (MODE == MODE_AB2 && a.out && !hold) reinterpret_cast<float*>(a.out)[ax * a.np + id] = (float)k1;
        }
        if (hold) xn = x0;
        ok &= split_cell(xn, a.g.inv_delta, a.g.mask, cn[ax]);
        a.pos_out[ax * a.np + j] = xn;
    }
    if constexpr (MODE == MODE_AB2_D) {
        if (a.out && !hold) {
#pragma unroll
            for (int i = 0; i < 9; ++i)
                reinterpret_cast<float*>(a.out)[i * a.np + id] = (float)((double)kb[3 + i] * a.g.inv_delta);
        }
    }
    if (!ok) atomicOr(a.flags + FLAG_NONFINITE, 1);
    if (!a.key_out) return;   // a set that is not grouped
    a.id_out[j] = id;
    const uint32_t key = block_key(a.g, cn[0], cn[1], cn[2]);
    a.key_out[j] = key;
    if (a.counts) {   // block counts of the next binning, one add per group of equal keys
        const unsigned peers = __match_any_sync(vm, key);
        if (lane == __ffs(peers) - 1) atomicAdd(a.counts + key, (uint32_t)__popc(peers));
    }
}

// Adjoint of one RK2 step, lane-dense (float64): with J in units of u per
// cell (times inv_delta: per length),
//   lambda* = dt/2 J(X*)^T lambda,  mu = dt/2 lambda + dt lambda*,
//   lambda <- lambda + lambda* + J(X)^T mu;
// lambda (caller order) is read and written, and what the field gradient's
// scatter needs is left in grouped order: X* (offsets and cell), mu, dt/2 lambda.
template <typename T, int MODE, int NC>
__device__ __forceinline__ void adjoint_particle(const BlockArgs& a, int64_t j, int32_t id, bool valid,
                                                 const unsigned char* ws, int lane)
{
    using WPl = WarpPlan<T, MODE, NC>;
    if (!valid) return;
    const T* kb = reinterpret_cast<const T*>(ws + WPl::k) + lane * WPl::KS;
    const double* ls = reinterpret_cast<const double*>(ws + WPl::x) + lane;
    const double dt = a.dt, hdi = 0.5 * dt * a.g.inv_delta;
    const double lam[3] = {ls[0], ls[32], ls[64]};
    double lstar[3], mu[3];
#pragma unroll
    for (int jj = 0; jj < 3; ++jj) {
        double s = 0;
#pragma unroll
        for (int k = 0; k < 3; ++k) s = fma(widen(kb[9 + 3 * k + jj]), lam[k], s);
        lstar[jj] = hdi * s;
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) mu[k] = fma(dt, lstar[k], 0.5 * dt * lam[k]);
#pragma unroll
    for (int jj = 0; jj < 3; ++jj) {
        double s = 0;
#pragma unroll
        for (int k = 0; k < 3; ++k) s = fma(widen(kb[3 * k + jj]), mu[k], s);
        a.pos_out[jj * a.np + id] = lam[jj] + lstar[jj] + a.g.inv_delta * s;
    }
    if (a.adj) {
        float4* o = a.adj + j;
        o[0] = make_float4((float)kb[18], (float)kb[19], (float)kb[20], (float)kb[21]);
        o[a.np] = make_float4((float)mu[0], (float)mu[1], (float)mu[2], 0.0f);
        o[2 * a.np] = make_float4((float)(0.5 * dt * lam[0]), (float)(0.5 * dt * lam[1]), (float)(0.5 * dt * lam[2]), 0.0f);
    }
}

// the adjoint of a particle that is held (update_particle): lambda as it is, nothing for the field gradient
__device__ __forceinline__ void hold_adjoint(const BlockArgs& a, int64_t j, const PRec<float>& rec)
{
    if (!a.adj) return;
    a.adj[j] = make_float4(rec.t[0], rec.t[1], rec.t[2], rec.cell);
    a.adj[a.np + j] = a.adj[2 * a.np + j] = make_float4(0.f, 0.f, 0.f, 0.f);
}

// per-warp pointers into its shared memory
template <typename T, int MODE, int NC>
struct WarpMem {
    using WPl = WarpPlan<T, MODE, NC>;
    PRec<T>* recs;
    T *kbuf, *wb0, *wb1;
    __device__ __forceinline__ WarpMem(unsigned char* ws, int g)
        : recs(reinterpret_cast<PRec<T>*>(ws + WPl::rec)), kbuf(reinterpret_cast<T*>(ws + WPl::k)),
          wb0(reinterpret_cast<T*>(ws + WPl::w) + g * WPl::WB), wb1(wb0 + WPl::NG * WPl::WB)
    {
    }
};

// ---------------------------------------------------------------------------
// A CTA's particles [j0, j1) (grouped order) with stencils from global memory.
// The warps take the particles four at a time in turn, so that the CTA's
// gathers stay close together in the field (and in L1).
// ---------------------------------------------------------------------------
template <typename T, int I, int DEG, int MODE, int NC, int STORE, int RW>
__device__ __forceinline__ void run_direct(const BlockArgs& a, int64_t j0, int64_t j1, unsigned char* ws, int warp,
                                           int nw, int lane)
{
    constexpr int GL = group_lanes<T, I, MODE, SRC_GLOBAL>(), P = 32 / GL;   // P particles at once,
    constexpr int R = 32 / P, PB_W = P * R;                                // R rounds of them per batch
    const int g = GL == 6 ? SixLanes(lane).group : lane / GL;
    const LaneMap<I, GL> m(lane);
    Basis<T, I, DEG, is_deriv<MODE>(), GL> B;
    B.init(table<T>(a), m);
    const WarpMem<T, MODE, NC> wm(ws, g);
    for (int64_t b0 = j0; b0 < j1; b0 += PB_W * nw) {
        const int64_t j = b0 + (lane / P * nw + warp) * P + lane % P;
        const int left = (int)min(j1 - b0 - P * warp, (int64_t)PB_W * nw);   // particles from this warp's first on
        if (left <= 0) break;
        const bool valid = j < j1 && lane < PB_W;
        const int64_t src = !valid ? 0 : (a.perm ? a.perm[j] : j);
        const int32_t id = !valid ? 0 : (a.id_in ? a.id_in[src] : (int32_t)src);
        wm.recs[lane] = particle_record<T>(a, j, src, valid);
        fetch_state<T, MODE, NC>(a, MODE == MODE_ADJ ? id : src, valid, ws, lane);
        __syncwarp();
        for (int ch = 0; ch < (WarpPlan<T, MODE, NC>::HAS_X ? 1 : (a.f.C + NC - 1) / NC); ++ch) {
            for (int it = 0; it < R && it * P * nw < left; ++it) {
                const PRec<T> rec = wm.recs[P * it + g];
                Place at{};
                unpack_cell(cell_of(rec), at.c);
                interpolate_group<T, I, DEG, MODE, NC, STORE, RW, SRC_GLOBAL>(
                    a, at, ch, rec.t, it * P * nw + g < left && lane < GL * P, lane, B, m, wm.wb0, wm.wb1, it & 1,
                    wm.kbuf + (P * it + g) * WarpMem<T, MODE, NC>::WPl::KS);
            }
            __syncwarp();
            if constexpr (is_step<MODE>()) {
                cp_async_wait_all();
                update_particle<T, MODE, NC>(a, j, id, valid, ws, lane);
            } else if constexpr (MODE == MODE_ADJ) {
                cp_async_wait_all();
                adjoint_particle<T, MODE, NC>(a, j, id, valid, ws, lane);
            } else if (valid) write_outputs<T, MODE, NC>(a, id, ch, ws, lane);
            __syncwarp();
        }
    }
}

// ---------------------------------------------------------------------------
// I = 8, float32, values: a whole warp per particle where stencils come from
// beyond L1.  Lane (x, j) owns the rows y = j and j + 4 of column x: 16 nodes,
// which it holds for RK2's second stage (eight lanes per particle would hold
// 64, 256 registers, and gathering twice doubles the traffic beyond L1).  The
// sums are those of the eight-lane form, bit for bit.  256^3, 1/16 per cell,
// RK2, us per step: 690 with eight lanes at best; 512^3, 1.4e-2 per cell: 1717.
// ---------------------------------------------------------------------------
template <int DEG>
struct WarpBasis {
    Row<float, DEG> r;
    int ax, i;
    bool act;
    __device__ __forceinline__ void init(const CoefTable<float>& tb, int lane)
    {
        act = lane < 24;
        ax = act ? lane >> 3 : 0;
        i = lane & 7;
        r = load_row<float, DEG>(tb.c, i);
    }
    __device__ __forceinline__ void eval(float s1, float s2, float s3, float* wb) const
    {
        const float w = horner(r, ax == 0 ? s1 : (ax == 1 ? s2 : s3));
        if (act) wb[ax * 8 + i] = w;
        __syncwarp();
    }
};

// the warp's sum of component comp = 2 bit4 + bit3 of the lane, in the eight lanes that share it
template <int NC>
__device__ __forceinline__ float warp_contract(const float (&f)[2][8][NC], const float* wb, int lane)
{
    const int x = lane & 7, j = lane >> 3;
    float w3[8];
    bcast_load(wb + 16, w3);
    const float w1 = wb[x], w2[2] = {wb[8 + j], wb[12 + j]};
    float p[4] = {0.f, 0.f, 0.f, 0.f}, pv[2][NC];
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int zz = 0; zz < 8; ++zz) axpy<true, NC>(zz == 0, w3[inward(zz, 8)], f[h][inward(zz, 8)], pv[h]);
#pragma unroll
    for (int k = 0; k < NC; ++k) {
        // rows in contract's order: j, j + 4 for j < 2, else j + 4, j
        const bool up = j < 2;
        p[k] = fmaf(up ? w2[1] : w2[0], up ? pv[1][k] : pv[0][k], (up ? w2[0] : w2[1]) * (up ? pv[0][k] : pv[1][k]));
    }
    const bool b4 = lane & 16, b3 = lane & 8;
    float q0 = (b4 ? p[2] : p[0]) + __shfl_xor_sync(0xffffffffu, b4 ? p[0] : p[2], 16);
    float q1 = (b4 ? p[3] : p[1]) + __shfl_xor_sync(0xffffffffu, b4 ? p[1] : p[3], 16);
    float m = (b3 ? q1 : q0) + __shfl_xor_sync(0xffffffffu, b3 ? q0 : q1, 8);
    m *= w1;
    m += __shfl_xor_sync(0xffffffffu, m, 4);
    m += __shfl_xor_sync(0xffffffffu, m, 2);
    m += __shfl_xor_sync(0xffffffffu, m, 1);
    return m;
}

template <int NC>
__device__ __forceinline__ void warp_load(const FieldView& f, int node, int ch, int lane, float (&v)[2][8][NC])
{
    const RecordLd<4, NC> ld{f.rec + ((int64_t)ch * f.plane + node + (lane & 7) + (lane >> 3) * f.NP) * 4, f.NP, f.NP * f.NP};
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int z = 0; z < 8; ++z) ld(4 * h, z, v[h][z]);
}

template <int DEG, int MODE, int NC>
__device__ __forceinline__ void run_direct_warp(const BlockArgs& a, int64_t j0, int64_t j1, unsigned char* ws, int warp,
                                                int nw, int lane)
{
    using T = float;
    using WPl = WarpPlan<T, MODE, NC>;
    static_assert(!is_deriv<MODE>(), "values only");
    constexpr int LO = 3;
    WarpBasis<DEG> B;
    B.init(a.cf, lane);
    const WarpMem<T, MODE, NC> wm(ws, 0);
    const int comp = (lane & 16 ? 2 : 0) + (lane & 8 ? 1 : 0);
    const bool writer = (lane & 7) == 0 && comp < NC;
    const float dtid = (float)(a.dt * a.g.inv_delta);
    for (int64_t b0 = j0; b0 < j1; b0 += 32 * nw) {
        const int64_t j = b0 + lane * nw + warp;
        const int left = (int)min(j1 - b0 - warp, (int64_t)32 * nw);   // particles from this warp's first on
        if (left <= 0) break;
        const bool valid = j < j1;
        const int64_t src = !valid ? 0 : (a.perm ? a.perm[j] : j);
        const int32_t id = !valid ? 0 : (a.id_in ? a.id_in[src] : (int32_t)src);
        wm.recs[lane] = particle_record<T>(a, j, src, valid);
        fetch_state<T, MODE, NC>(a, src, valid, ws, lane);
        __syncwarp();
        for (int ch = 0; ch < (is_step<MODE>() ? 1 : (a.f.C + NC - 1) / NC); ++ch) {
            for (int it = 0; it * nw < left; ++it) {
                const PRec<T> rec = wm.recs[it];
                int c[3];
                unpack_cell(cell_of(rec), c);
                float f[2][8][NC];
                warp_load<NC>(a.f, (int)padded_index(a.f.NP, c[0] - LO, c[1] - LO, c[2] - LO), ch, lane, f);
                float* kb = wm.kbuf + it * WPl::KS;
                B.eval(rec.t[0] - 0.5f, rec.t[1] - 0.5f, rec.t[2] - 0.5f, MODE != MODE_RK2 && (it & 1) ? wm.wb1 : wm.wb0);
                const float m = warp_contract<NC>(f, MODE != MODE_RK2 && (it & 1) ? wm.wb1 : wm.wb0, lane);
                if (writer) kb[comp] = m;
                if constexpr (MODE == MODE_RK2) {
                    float ts[3];
                    int d[3];
#pragma unroll
                    for (int ax = 0; ax < 3; ++ax) {
                        const float u1 = __shfl_sync(0xffffffffu, m, ax == 0 ? 0 : (ax == 1 ? 8 : 16));
                        ts[ax] = fmaf(dtid, u1, rec.t[ax]);
                        const float fl = floorf(ts[ax]);
                        d[ax] = (int)fl;
                        ts[ax] -= fl;
                    }
                    if ((d[0] | d[1] | d[2]) != 0) {   // (the whole warp: one particle)
                        const bool far = (unsigned)d[0] + 1u > 2u || (unsigned)d[1] + 1u > 2u || (unsigned)d[2] + 1u > 2u;
                        if (far) {
                            if (lane == 0) atomicOr(a.flags + FLAG_CFL, 1);
#pragma unroll
                            for (int ax = 0; ax < 3; ++ax) c[ax] = (int)(((unsigned)c[ax] + (unsigned)d[ax]) & (unsigned)a.g.mask);
                        } else {
#pragma unroll
                            for (int ax = 0; ax < 3; ++ax) c[ax] += d[ax];
                        }
                        warp_load<NC>(a.f, (int)padded_index(a.f.NP, c[0] - LO, c[1] - LO, c[2] - LO), 0, lane, f);
                    }
                    B.eval(ts[0] - 0.5f, ts[1] - 0.5f, ts[2] - 0.5f, wm.wb1);
                    const float m2 = warp_contract<NC>(f, wm.wb1, lane);
                    if (writer) kb[3 + comp] = m2;
                }
            }
            __syncwarp();
            if constexpr (is_step<MODE>()) {
                cp_async_wait_all();
                update_particle<T, MODE, NC>(a, j, id, valid, ws, lane);
            } else if (valid) {
                write_outputs<T, MODE, NC>(a, id, ch, ws, lane);
            }
            __syncwarp();
        }
    }
}

// resident CTAs (of four warps) per SM the kernels are register-capped for
// (128 registers)
constexpr int CTAS_SM = 4;

}  // namespace trk
