// Block kernel: one CTA per cell block of BLK^3 cells (the block grouping of
// Sec. 3.3.1, with the paper's x3 slices generalised to cubes), the block's
// field halo staged in shared memory.  The arithmetic is interp_core.cuh's;
// here are the staging and the CTA's phases:
//
//   issue   the halo of a component chunk starts to land: one tensor copy
//           (cp.async.bulk.tensor, TMA) issued by one thread and awaited on an
//           mbarrier, or cp.async copies of one record (16 or 4 bytes; 8-byte
//           elements of a float64 field) each, in the same layout;
//   P1      each warp splits its particles (float64, lane-dense) meanwhile;
//   Q       the warps interpolate, four particles at a time, from shared memory;
//   P3      lane-dense outputs, or the position update.
//
// Particles beyond PB = 128 in a block take further batches.
#pragma once

#include "interp_core.cuh"

namespace trk {

enum { HC_ASYNC = 0, HC_TMA = 1 };

__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait_group()
{
    asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

__device__ __forceinline__ void mbar_init(uint64_t* bar)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_addr(bar)) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
}

// one thread: announce `bytes` for the barrier's current phase and start the copy of
// the box at tensor coordinates (x, y, z, k) into dst
__device__ __forceinline__ void tma_issue(void* dst, const CUtensorMap* map, int x, int y, int z, int k, uint64_t* bar,
                                          uint32_t bytes)
{
    // shared-memory reads of the previous halo (generic proxy) are ordered
    // before the copy's writes (async proxy)
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(smem_addr(bar)), "r"(bytes)
                 : "memory");
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], "
        "[%6];\n" ::"r"(smem_addr(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(k), "r"(smem_addr(bar))
        : "memory");
}

// Waits for the barrier's phase `parity` to complete; false after `limit` polls
// (each try_wait itself suspends for a bounded time).
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, int limit)
{
    const uint32_t a = smem_addr(bar);
    for (int it = 0; it < limit; ++it) {
        uint32_t done = 0;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(done)
            : "r"(a), "r"(parity)
            : "memory");
        if (done) return true;
    }
    return false;
}

// Copies the halo of component chunk ch into shared memory (cp.async, the
// caller waits).  Threads run along x1.
template <typename T, int I, int MODE, int NC, int STORE, int RW>
__device__ __forceinline__ void stage_halo_async(unsigned char* halo, const FieldView& f, int ch, int o1, int o2, int o3)
{
    using HG = HaloGeom<T, I, MODE, NC, RW>;
    constexpr int H = HG::H;
    const int64_t NP = f.NP;
    const int64_t n0 = ((int64_t)(o3 + PAD) * NP + (o2 + PAD)) * NP + (o1 + PAD);
    constexpr int COMPS = STORE == ST_F64 ? NC : 1;
    const int kc = STORE == ST_F64 ? min(NC, f.C - ch * NC) : 1;
    for (int e = threadIdx.x; e < COMPS * H * H * H; e += NT) {
        const int x = e % H, y = e / H % H, z = e / (H * H) % H, k = e / (H * H * H);
        const int64_t n = n0 + ((int64_t)z * NP + y) * NP + x;
        const int d = k * HG::SC + z * HG::PL + y * HG::P + x + HG::XOFF;
        if constexpr (STORE == ST_F64) {
            if (k < kc) cp_async<8>(reinterpret_cast<double*>(halo) + d, f.f64 + (int64_t)(ch * NC + k) * f.plane + n);
        } else {
            cp_async<4 * RW>(halo + (size_t)d * 4 * RW, f.rec + ((int64_t)ch * f.plane + n) * RW);
        }
    }
}

template <typename T, int I, int MODE, int NC, int RW>
struct BlockPlan {
    static constexpr size_t mbar = HaloGeom<T, I, MODE, NC, RW>::bytes;
    static constexpr size_t warp = mbar + 32;
    static constexpr size_t total = warp + NW * WarpPlan<T, MODE, NC>::total;
    static_assert(total <= 232448, "block shared-memory plan exceeds the per-block limit");
};

// One CTA per cell block: cp.async halos, and the tensor-copy halos of float64
// fields (whose arithmetic, not the staging, sets the time).
template <typename T, int I, int DEG, int MODE, int NC, int STORE, int RW, int HC>
__global__ void __launch_bounds__(NT, 4)
    k_block(const __grid_constant__ BlockArgs a, const __grid_constant__ CUtensorMap tmap)
{
    using HG = HaloGeom<T, I, MODE, NC, RW>;
    using PL = BlockPlan<T, I, MODE, NC, RW>;
    constexpr bool STEP = is_step<MODE>();
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const int b = blockIdx.x;
    const int j0 = a.offsets[b], j1 = a.offsets[b + 1];
    if (j0 >= j1) return;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 3;
    Place at{};
    at.halo = smem_raw;
    const int o1 = b % a.g.nb1 * BLK - HG::G, o2 = b / a.g.nb1 % a.g.nb2 * BLK - HG::G,
              o3 = b / (a.g.nb1 * a.g.nb2) * BLK - HG::G;
    uint64_t* mbar = reinterpret_cast<uint64_t*>(smem_raw + PL::mbar);
    unsigned char* ws = smem_raw + PL::warp + warp * WarpPlan<T, MODE, NC>::total;
    const WarpMem<T, MODE, NC> wm(ws, g);
    const LaneMap<I> m(lane);
    Basis<T, I, DEG, is_deriv<MODE>()> B;
    B.init(table<T>(a), m);
    const int nchunks = STEP ? 1 : (a.f.C + NC - 1) / NC;

    uint32_t phase = 0;
    bool hold = false;
    if constexpr (HC == HC_TMA) {
        static_assert(STORE == ST_F64, "node records are staged by k_slabs");
        if (tid == 0) mbar_init(mbar);
        __syncthreads();
    }
    auto issue_halo = [&](int ch) {
        if constexpr (HC == HC_TMA) {
            if (tid == 0)
                tma_issue(smem_raw, &tmap, o1 + PAD - HG::XOFF, o2 + PAD, o3 + PAD, NC * ch, mbar,
                          (uint32_t)(NC * HG::SC * sizeof(double)));
        } else {
            stage_halo_async<T, I, MODE, NC, STORE, RW>(smem_raw, a.f, ch, o1, o2, o3);
        }
    };
    for (int b0 = j0; b0 < j1; b0 += PB) {
        if (b0 == j0) issue_halo(0);   // lands while P1 runs
        const int j = b0 + ((lane >> 2) * NW + warp) * 4 + (lane & 3);
        const int left = min(j1 - b0 - 4 * warp, PB);
        const bool valid = j < j1;
        const int64_t src = !valid ? 0 : (a.perm ? a.perm[j] : j);
        const int32_t id = !valid ? 0 : (a.id_in ? a.id_in[src] : (int32_t)src);
        wm.recs[lane] = particle_record<T>(a, j, src, valid);
        fetch_state<T, MODE, NC>(a, src, valid, ws, lane);
        __syncwarp();
        for (int ch = 0; ch < nchunks; ++ch) {
            // a chunk is staged for this (batch, chunk) unless the only chunk is still in place
            const bool issued = (b0 == j0 && ch == 0) || nchunks > 1;
            if (issued && !(b0 == j0 && ch == 0)) {
                __syncthreads();   // the previous halo's readers are done
                issue_halo(ch);
            }
            if (issued) {
                if constexpr (HC == HC_TMA) {
                    // if the copy did not land within the limit (all threads agree) the block's
                    // particles are held and the host is told; the shared memory is not
                    // given up while the copy may still write to it
                    const bool ok = mbar_wait(mbar, phase, a.wait_limit);
                    if (__syncthreads_or(!ok)) {
                        hold = true;
                        if (tid == 0) atomicOr(a.flags + FLAG_HALO_TIMEOUT, 1);
                        mbar_wait(mbar, phase, kWaitLimit);
                    }
                    phase ^= 1u;
                } else {
                    cp_async_wait_all();
                    __syncthreads();
                }
            }
            for (int it = 0; it < 8 && it * 4 * NW < left; ++it) {
                const PRec<T> rec = wm.recs[4 * it + g];
                unpack_cell(cell_of(rec), at.c);   // (a particle lies in its own block)
                interpolate_group<T, I, DEG, MODE, NC, STORE, RW, SRC_HALO>(
                    a, at, ch, rec.t, it * 4 * NW + g < left, lane, B, m, wm.wb0, wm.wb1, it & 1,
                    wm.kbuf + (4 * it + g) * WarpMem<T, MODE, NC>::WPl::KS);
            }
            __syncwarp();
            if constexpr (!STEP) {
                if (valid && !hold) write_outputs<T, MODE, NC>(a, id, ch, ws, lane);
                __syncwarp();
            }
        }
        if constexpr (STEP) {
            cp_async_wait_all();
            update_particle<T, MODE, NC>(a, j, id, valid, ws, lane, hold);
            __syncwarp();
        }
    }
}

// ---------------------------------------------------------------------------
// Pipelined form for node records: one persistent CTA per SM takes a
// contiguous range of the grouped particles and walks their cell blocks in
// key order, i.e. along rows of blocks in x1 (TRK_STEP_COLUMN: rows stacked along
// x3 in segments first).  The field passes through shared
// memory as a ring of NS slabs (SlabGeom): moving one block along x1 brings in
// only the slabs it does not share with the previous block, copied (TMA) NS
// slabs ahead while earlier blocks are interpolated.
//
// The slabs of the CTA's blocks are numbered in the order they are needed
// (SPT per block and NSL - SPT more per row of blocks); slab q goes to slot
// q mod NS.  The warps take the particles four at a time in turn, as in
// run_direct, and never wait for each other: a warp waits for the slabs its
// four particles need (full[slot], an mbarrier), and when it moves past a slab
// it counts itself off (done[slot]); the last of the CTA's warps to do so
// starts the copy of slab q + NS into the slot.  A warp holds the slabs of at
// most two adjacent blocks of a row at a time (an iteration whose particles
// span more takes further rounds) and every warp passes through every slab in
// order, so with NS >= NSL + SPT the slowest warp never waits for another one.
//
// Bound: the shared-memory data path, I^2 runs of I records per stencil (one
// wavefront each; I = 4 two runs per wavefront) plus about ten wavefronts for
// weights and reductions; sparse sets: the copies, at about 6.6 TB/s from L2
// (a slab of I = 6, RK2, is 29 KB where a box of H^3 nodes is 54 KB: 256^3, 1/64
// particle per cell, 227 against 315 us per step).  256^3 float32, us per call,
// against one CTA and one box per block with a warp per particle: I = 8, u, 2^21
// tracers 804 -> 530; I = 6, RK2, 2^20 tracers 533 -> 380.
// ---------------------------------------------------------------------------
template <int I, int MODE, int NC>
struct SlabPlan {
    using SG = SlabGeom<I, MODE>;
    // (the adjoint hands 22 values per particle over: fewer warps leave room for the slabs)
    static constexpr int warps = MODE == MODE_ADJ ? (I == 8 ? 8 : 12) : 4 * CTAS_SM;
    static constexpr size_t slab = SG::slot;
    static constexpr size_t per_warp = WarpPlan<float, MODE, NC>::total;
    static constexpr size_t room = 232448 - 256 - warps * per_warp;
    static constexpr int NS = room / slab < 12 ? (int)(room / slab) : 12;
    static constexpr size_t full = NS * slab;                // [NS] mbarriers
    static constexpr size_t done = full + 128;               // [NS] counters
    static constexpr size_t issued = done + 64;              // [NS] the last slab copied into the slot
    static constexpr size_t warp = issued + 64;
    static constexpr size_t total = warp + warps * per_warp;
    static_assert(NS >= SG::NSL + SG::SPT && NS <= 16, "slabs of two adjacent blocks; counters");
    static_assert(total <= 232448, "slab shared-memory plan exceeds the per-block limit");
};

// the CTA's slabs as one warp sees them
template <int I, int MODE, int NC>
struct Slabs {
    using SP = SlabPlan<I, MODE, NC>;
    using SG = typename SP::SG;
    static constexpr int NS = SP::NS;
    unsigned char* smem;
    const BlockArgs& a;
    const CUtensorMap* map;
    int ch;                      // component chunk
    int b_first, b_last;         // the CTA's cell blocks
    int l1, per_row, q0, count;  // log2 nb1; slabs per row of blocks; number of b_first's first slab; slabs of the CTA
    int held = 0, ready = -1;    // this warp: first slab not counted off; last slab waited for
    bool dead = false;           // (this lane's) a wait ran out: no further waits, nothing counted off (give_up)

    __device__ __forceinline__ void init()
    {
        l1 = __ffs(a.g.nb1) - 1;   // block counts are powers of two
        per_row = SG::SPT * a.g.nb1 + SG::NSL - SG::SPT;
        q0 = 0;
        q0 = first_slab(b_first);
        count = first_slab(b_last) + SG::NSL;
    }
    // number of cell block b's first slab
    __device__ __forceinline__ int first_slab(int b) const
    {
        return (b >> l1) * per_row + (b & (a.g.nb1 - 1)) * SG::SPT - q0;
    }
    __device__ __forceinline__ uint64_t* full(int q) const
    {
        return reinterpret_cast<uint64_t*>(smem + SP::full) + q % NS;
    }
    __device__ __forceinline__ int* issued(int q) const { return reinterpret_cast<int*>(smem + SP::issued) + q % NS; }
    // rows of blocks: x3 inside a segment of 2^lseg blocks, then x2, the segments along x3
    __device__ __forceinline__ void row_origin(int row, int& o2, int& o3) const
    {
        const int ls = a.g.lseg, l2 = __ffs(a.g.nb2) - 1;
        o2 = (row >> ls & (a.g.nb2 - 1)) * BLK - SG::G;
        o3 = ((row >> (ls + l2) << ls) + (row & ((1 << ls) - 1))) * BLK - SG::G;
    }
    // one thread: start slab q's copy.  A sparse set's slab that no occupied block of
    // the CTA uses is left out (its barrier's phase is only completed); with four
    // particles per block on average nearly every slab is used, and reading the offsets
    // first would add their latency to every copy
    __device__ __forceinline__ void issue(int q) const
    {
        if (q >= count) return;
        *issued(q) = q;
        const int row = (q + q0) / per_row, pos = (q + q0) - row * per_row;
        const int lo = max(max(pos - SG::NSL + SG::SPT, 0) / SG::SPT + (row << l1), b_first);
        const int hi = min(min(pos / SG::SPT, a.g.nb1 - 1) + (row << l1), b_last);
        if (a.np >= 4 * ((int64_t)a.g.nb3 * a.g.nb2 << l1) || (hi >= lo && a.offsets[hi + 1] > a.offsets[lo])) {
            int o2, o3;
            row_origin(row, o2, o3);
            tma_issue(smem + q % NS * SP::slab, map, 4 * (SG::X0 + pos * SG::SW + PAD), o2 + PAD, o3 + PAD, ch, full(q),
                      (uint32_t)SG::bytes);
        } else {
            asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(smem_addr(full(q))) : "memory");
        }
    }
    __device__ __forceinline__ void need(int q)
    {
        while (ready < q) {
            ++ready;
            if (!dead && !mbar_wait(full(ready), (uint32_t)(ready / NS) & 1u, a.wait_limit)) {
                dead = true;
                atomicOr(a.flags + FLAG_HALO_TIMEOUT, 1);
            }
        }
    }
    // A lane whose wait runs out waits no more, and lane 0, if it is the one, counts no
    // more slabs off: none is copied over before every warp has seen it land (the other
    // warps' waits for what then never comes run out too).  The warp's particles stay as
    // they are from that batch on (its lanes go on over whatever the slots hold), and
    // before it leaves it waits, up to the full limit, for the copies on their way, those
    // that it issued itself among them: the shared memory is not given up under them.
    __device__ __forceinline__ void give_up()
    {
        for (int s = 0; s < NS; ++s) {
            const int q = *static_cast<volatile int*>(issued(s));
            // (one that does not land leaves the others no less time)
            if (q >= 0 && !mbar_wait(full(q), (uint32_t)(q / NS) & 1u, kWaitLimit)) break;
        }
    }
    // count this warp off the slabs before q (their reads are consumed)
    __device__ __forceinline__ void release_to(int q, int lane, int nw)
    {
        while (held < q) {
            need(held);
            __syncwarp();
            if (lane == 0 && !dead) {
                int* d = reinterpret_cast<int*>(smem + SP::done) + held % NS;
                int old;
                asm volatile("atom.acq_rel.cta.shared::cta.add.s32 %0, [%1], 1;\n"
                             : "=r"(old)
                             : "r"(smem_addr(d))
                             : "memory");
                if (old == nw - 1) {
                    *d = 0;
                    issue(held + NS);
                }
            }
            __syncwarp();
            ++held;
        }
    }
};

template <int I, int DEG, int MODE, int NC>
__global__ void __launch_bounds__(32 * SlabPlan<I, MODE, NC>::warps, 1)
    k_slabs(const __grid_constant__ BlockArgs a, const __grid_constant__ CUtensorMap tmap)
{
    using T = float;
    using SP = SlabPlan<I, MODE, NC>;
    using SG = typename SP::SG;
    constexpr int nw = SP::warps;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int GL = group_lanes<T, I, MODE, SRC_SLABS>(), P = 32 / GL;   // P particles at once
    const int g = lane / GL;
    const int64_t j0 = (int64_t)blockIdx.x * a.ppc;
    const int64_t j1 = j0 + a.ppc < a.np ? j0 + a.ppc : a.np;
    const PRec<T>* recs_in = reinterpret_cast<const PRec<T>*>(a.rec_in);
    Slabs<I, MODE, NC> slabs{smem_raw, a, &tmap, (int)blockIdx.y};
    {   // cell blocks of the first and the last particle (lanes 0 and 1)
        int c[3];
        unpack_cell(cell_of(recs_in[lane == 0 ? j0 : j1 - 1]), c);
        const int b = (int)block_key(a.g, c[0], c[1], c[2]);
        slabs.b_first = __shfl_sync(0xffffffffu, b, 0);
        slabs.b_last = __shfl_sync(0xffffffffu, b, 1);
        slabs.init();
    }
    if (tid == 0) {
        for (int s = 0; s < SP::NS; ++s) {
            mbar_init(slabs.full(s));
            reinterpret_cast<int*>(smem_raw + SP::done)[s] = 0;
            *slabs.issued(s) = -1;
        }
        for (int s = 0; s < SP::NS; ++s) slabs.issue(s);
    }
    __syncthreads();
    unsigned char* ws = smem_raw + SP::warp + warp * SP::per_warp;
    const WarpMem<T, MODE, NC> wm(ws, g);
    const LaneMap<I, GL> m(lane);
    Basis<T, I, DEG, is_deriv<MODE>(), GL> B;
    B.init(a.cf, m);
    // A batch is GL rounds of P particles per warp; the warps' first batches have 1/8
    // to 8/8 of these rounds, so that their float64 phases do not all meet on that pipe at once.
    // The records of the next batch and the state of this one are copied to shared
    // memory (cp.async) while this one is interpolated.
    int rounds = (1 + (warp & 7)) * (GL / 8), odd = 0, buf = 0;
    auto my_index = [&](int64_t b0) { return b0 + (lane / P * nw + warp) * P + lane % P; };
    auto fetch_records = [&](int64_t b0, int nrounds, int to) {
        const int64_t j = my_index(b0);
        if (j < j1 && lane / P < nrounds) cp_async<16>(wm.recs + to * 32 + lane, recs_in + j);
    };
    fetch_records(j0, rounds, 0);
    cp_async_commit();
    for (int64_t b0 = j0; b0 < j1; buf ^= 1) {
        const int64_t bn = b0 + (int64_t)P * nw * rounds;
        const int64_t j = my_index(b0);
        // (the same number; how it is formed, and the two calls of update_particle below, tip the
        // register allocation: gradients 482 and 528 us per step of 2^21 particles at 256^3, RK2
        // 402 and 385 per 2^20)
        using Left = std::conditional_t<MODE == MODE_RK2, int64_t, int>;
        const int left = (int)min((Left)(j1 - b0) - P * warp, (Left)(P * nw * rounds));
        if (left <= 0) break;
        const bool valid = j < j1 && lane / P < rounds;
        int32_t id = 0;   // (loaded where it is needed: a register less meanwhile)
        if (MODE == MODE_ADJ && valid) id = a.id_in[j];
        fetch_state<T, MODE, NC>(a, MODE == MODE_ADJ ? id : j, valid, ws, lane);
        fetch_records(bn, GL, buf ^ 1);
        cp_async_commit();
        cp_async_wait_group<1>();
        __syncwarp();
        for (int it = 0; it < rounds && it * P * nw < left; ++it) {
            const bool live = it * P * nw + g < left;
            const PRec<T> rec = wm.recs[buf * 32 + P * it + g];
            int c[3] = {0, 0, 0};
            if (live) unpack_cell(cell_of(rec), c);
            // (a particle lies in one of the CTA's blocks; the clamp only keeps corrupted
            // records inside them)
            const int block = min(max((int)block_key(a.g, c[0], c[1], c[2]), slabs.b_first), slabs.b_last);
            const int q = slabs.first_slab(block);
            bool todo = live;
            do {   // one round, unless the particles lie in more than two adjacent blocks of a row
                const int lo = (int)__reduce_min_sync(0xffffffffu, todo ? (unsigned)q : 0x7fffffffu);
                const bool now = todo && q - lo <= SG::SPT;
                Place at{};
                at.c[0] = c[0], at.c[1] = c[1], at.c[2] = c[2];
                at.slab = now ? q : lo;
                slabs.release_to(lo, lane, nw);
                slabs.need((int)__reduce_max_sync(0xffffffffu, (unsigned)at.slab) + SG::NSL - 1);
                at.halo = smem_raw;
                interpolate_group<T, I, DEG, MODE, NC, ST_F32, 4, SRC_SLABS, SP::NS>(
                    a, at, slabs.ch, rec.t, now, lane, B, m, wm.wb0, wm.wb1, odd & 1,
                    wm.kbuf + (P * it + g) * WarpMem<T, MODE, NC>::WPl::KS);
                ++odd;
                todo = todo && !now;
            } while (__any_sync(0xffffffffu, todo));
        }
        if (MODE != MODE_ADJ && valid) id = a.id_in ? a.id_in[j] : (int32_t)j;
        __syncwarp();
        const bool dead = __any_sync(0xffffffffu, slabs.dead);
        if constexpr (is_step<MODE>()) {
            cp_async_wait_all();
            if (MODE == MODE_RK2 && !dead) update_particle<T, MODE, NC>(a, j, id, valid, ws, lane);
            else update_particle<T, MODE, NC>(a, j, id, valid, ws, lane, dead);
        } else if constexpr (MODE == MODE_ADJ) {
            cp_async_wait_all();
            if (!dead) adjoint_particle<T, MODE, NC>(a, j, id, valid, ws, lane);
            else if (valid) hold_adjoint(a, j, wm.recs[buf * 32 + lane]);
        } else if (valid && !dead) {
            write_outputs<T, MODE, NC>(a, id, slabs.ch, ws, lane);
        }
        __syncwarp();
        b0 = bn;
        rounds = GL;
    }
    cp_async_wait_all();
    slabs.release_to(slabs.count, lane, nw);   // every copy has landed before the CTA ends
    if (__any_sync(0xffffffffu, slabs.dead)) slabs.give_up();
}

template <typename T, int I, int DEG, int MODE, int NC, int STORE, int RW, int HC>
cudaError_t launch_block_hc(const BlockArgs& a, const CUtensorMap& tmap, int64_t nblocks, cudaStream_t st)
{
    constexpr size_t smem = BlockPlan<T, I, MODE, NC, RW>::total;
    auto kern = k_block<T, I, DEG, MODE, NC, STORE, RW, HC>;
    static bool attr_set = false;
    if (!attr_set) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        attr_set = true;
    }
    if (nblocks <= 0) return cudaSuccess;
    kern<<<(unsigned)nblocks, NT, smem, st>>>(a, tmap);
    return cudaGetLastError();
}

template <int I, int DEG, int MODE, int NC>
cudaError_t launch_slabs(BlockArgs a, const CUtensorMap& tmap, cudaStream_t st)
{
    using SP = SlabPlan<I, MODE, NC>;
    auto kern = k_slabs<I, DEG, MODE, NC>;
    static int nsm = 0;
    if (!nsm) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SP::total);
        if (e != cudaSuccess) return e;
        int dev = 0;
        if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
        if ((e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    }
    if (a.np <= 0) return cudaSuccess;
    // one contiguous run of particles per SM, whole fours
    a.ppc = (int)(((a.np + nsm - 1) / nsm + 3) / 4 * 4);
    const dim3 grid((unsigned)((a.np + a.ppc - 1) / a.ppc), WarpPlan<float, MODE, NC>::HAS_X ? 1 : (unsigned)((a.f.C + NC - 1) / NC));
    kern<<<grid, 32 * SP::warps, SP::total, st>>>(a, tmap);
    return cudaGetLastError();
}

// tmap: the tensor map of the field for this mode's box (halo_box), or null
// for cp.async copies
template <typename T, int I, int DEG, int MODE, int NC, int STORE, int RW>
cudaError_t launch_block_t(const BlockArgs& a, const CUtensorMap* tmap, int64_t nblocks, cudaStream_t st)
{
    if constexpr (STORE == ST_F64) {
        if (tmap) return launch_block_hc<T, I, DEG, MODE, NC, STORE, RW, HC_TMA>(a, *tmap, nblocks, st);
    } else if constexpr (RW == 4) {
        if (tmap) return launch_slabs<I, DEG, MODE, NC>(a, *tmap, st);
    }
    const CUtensorMap none{};
    return launch_block_hc<T, I, DEG, MODE, NC, STORE, RW, HC_ASYNC>(a, none, nblocks, st);
}

}  // namespace trk
