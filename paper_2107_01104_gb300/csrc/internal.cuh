// Internal declarations shared by the CUDA translation units of libtracker.
// Not part of the public ABI (see include/tracker.h).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "coeffs.inc"

namespace trk {

// ---------------------------------------------------------------------------
// Device error flags (one int each in a small device array owned by the
// tracker).  Set with atomicOr, read and cleared by tracker_sync().
// ---------------------------------------------------------------------------
// FLAG_BINNING: a counting-sort scatter found a block fuller than its count
// (cannot happen when every step counts what it writes; guarded anyway).
// FLAG_HALO_TIMEOUT: a tensor copy of a block's halo or of a slab did not
// complete within the wait limit (the particles that needed it stay as they
// were; reported as an internal error).
enum { FLAG_NONFINITE = 0, FLAG_CFL = 1, FLAG_BINNING = 2, FLAG_HALO_TIMEOUT = 3, NUM_FLAGS = 4 };

// Storage codes (same values as trk_storage in tracker.h).
enum { ST_F64 = 0, ST_F32 = 1, ST_BF16X2 = 2 };

// Block-kernel modes.
// MODE_AB2_D: AB2 step that also writes du_k/dX_j at the step's start.
// MODE_ADJ: the adjoint of an RK2 step (Jacobians at X and X*, lambda recurrence).
enum { MODE_INTERP = 0, MODE_INTERP_DERIV = 1, MODE_RK2 = 2, MODE_AB2 = 3, MODE_AB2_D = 4, MODE_ADJ = 5 };

constexpr int BLK = 8;        // cell-block edge used by the block kernels
constexpr int LBLK = 3;       // log2(BLK)

// The stored field is ghost-padded: PAD periodic copies on each side of every
// axis, so a block's halo is a plain box (no wrap) and its rows can be read
// with aligned 16-byte vector loads.  Component k, node (x1, x2, x3) with
// x in [-PAD, N + PAD) lives at k * plane + ((x3 + PAD) * NP + (x2 + PAD)) * NP + (x1 + PAD).
constexpr int PAD = 8;

//
// Float64 fields are stored component-major, [C][NP^3].  Float32 and split-bf16
// fields are stored as node records, the layout every kernel gathers: four
// components per 16-byte record (C = 1: one per 4-byte record), chunk ch
// holding components 4 ch .. 4 ch + 3 of every node, absent components zero,
// [chunks][NP^3] records.  One stencil row of I nodes is then one contiguous
// run whatever the component.  A split-bf16 value is kept as the float32 sum
// of its two halves, which is what every use of the pair begins with (four
// bytes either way; unpacking pairs in the gathers took 12 of the 17
// instructions per node of a four-component chunk).
struct FieldView {
    int storage;              // ST_*
    int C;                    // components
    int NP;                   // padded extent N + 2 PAD
    int64_t plane;            // NP^3 nodes
    const double* f64;        // [C][NP^3]                        (ST_F64)
    const float* rec;         // [chunks][NP^3][4] (C = 1: [NP^3]) (ST_F32, ST_BF16X2)
};

__host__ __device__ constexpr int record_width(int C) { return C == 1 ? 1 : 4; }
__host__ __device__ constexpr int record_chunks(int C) { return (C + 3) / 4; }

__host__ __device__ __forceinline__ int64_t padded_index(int NP, int x1, int x2, int x3)
{
    return ((int64_t)(x3 + PAD) * NP + (x2 + PAD)) * NP + (x1 + PAD);
}

// ---------------------------------------------------------------------------
// Halo of an 8^3 cell block for kernel width I and stage-2 margin (0, or 1 for
// RK2): H^3 nodes from G nodes before the block.  P is the row pitch of its
// dense copy in shared memory (plane pitch P H): records, H; float64
// elements, even, the halo starting XOFF elements into the row so that a
// tensor copy starts on a 16-byte boundary.  Host: the tensor map's box;
// device: the lane offsets.
// ---------------------------------------------------------------------------
struct HaloBox {
    int H, G, P, XOFF;
};

__host__ __device__ constexpr HaloBox halo_box(int I, int margin, bool f64)
{
    const int H = BLK + I - 1 + 2 * margin;
    const int G = I / 2 - 1 + margin;
    const int xoff = f64 ? (PAD - G) & 1 : 0;
    const int P = f64 ? (H + xoff + 1) / 2 * 2 : H;
    return HaloBox{H, G, P, xoff};
}

// x1 extent of the slabs the pipelined block kernel stages the halos of node records in
__host__ __device__ constexpr int slab_width(int I) { return I == 4 ? 4 : 8; }

// components per chunk of an interpolation (the steps take three)
__host__ __device__ constexpr int chunk_components(int C) { return C == 1 ? 1 : (C <= 3 ? 3 : 4); }

// Kernel weights beta_i(s), s = t - 1/2, as polynomial coefficients, passed by
// value so that the kernels read them as constant-bank operands.
template <typename T>
struct CoefTable {
    T c[TRK_TAB_MAX_I][TRK_TAB_MAX_DEG];   // beta_i
    T d[TRK_TAB_MAX_I][TRK_TAB_MAX_DEG];   // beta_i' (d/dt)
};

struct GridGeom {
    int N, mask;
    int lb1, lb2, lb3;        // log2 of the binning block edges
    int nb1, nb2, nb3;        // blocks per axis
    int lseg;                 // log2 of the blocks along x3 whose rows of keys follow each other (0: x2 next)
    double inv_delta;         // fl(N / L)
};

// Arguments of the block and direct kernels (interpolation, RK2 step, AB step).
struct BlockArgs {
    GridGeom g;
    FieldView f;
    CoefTable<float> cf;      // weights for float32 arithmetic
    CoefTable<double> cd;     // weights for float64 arithmetic
    int64_t np;               // particle count (stride of the [3][np] arrays)
    const int32_t* offsets;   // [nblocks + 1]
    const int32_t* perm;      // sorted position j -> index into the *_in arrays, or null (identity)
    const double* pos_in;     // [3][np]
    const int32_t* id_in;     // [np] or null (then id = perm[j])
    const void* rec_in;       // [np] PRec (grouped) or null (then split from pos_in)
    const float* rhs_in;      // [ab_order-1][3][np] AB history (u_{n-1} first) or null
    double* pos_out;          // [3][np], written at j
    int32_t* id_out;          // [np], written at j
    float* rhs_out;           // [ab_order-1][3][np], written at j
    uint32_t* key_out;        // [np], written at j, or null (a set that is not grouped: no id_out, counts)
    uint32_t* counts;         // [nblocks] block counts of the new keys (added into) or null
    void* out;                // interpolation outputs [nout][np], written at id
    int out_f64;
    int history_valid;        // AB: valid history entries on entry, 0 .. ab_order-1
    int ab_order;             // AB order k (2, 3, 4); the history holds k-1 entries
    int ppc;                  // direct kernel: particles per CTA (a multiple of 16), 0 (by size) or PPC_WIDE
    double dt;
    int* flags;
    int wait_limit;           // polls of a tensor copy's barrier before a wait gives up
    float4* adj;              // MODE_ADJ: [3][np] X* (offsets, cell), mu, dt/2 lambda (grouped) or null
};

constexpr int PPC_WIDE = -1;
// polls after which a wait for a tensor copy gives up, so that a copy that never
// lands cannot hang a kernel: a poll of a phase that does not complete takes 1.47 us
// on this GPU, the limit 1.5 s (a slab CTA then ends within three of these: the
// first wait, the other warps', and the copies on their way)
constexpr int kWaitLimit = 1 << 20;
constexpr int AB_MAX_HIST = 3;   // history entries of the highest supported order (AB4)

// dt-free Adams-Bashforth increment of order q (1..4): sum_j beta^q_j u_{n-j}
// with u_n = f0 and u_{n-j} = hist(j - 1), summed newest first; beta^q are the
// textbook weights (integrals over one step of the Lagrange basis on the past
// steps).
template <class HIST>
__device__ __forceinline__ double ab_increment(int q, double f0, const HIST& hist)
{
    switch (q) {
        case 1: return f0;
        case 2: return 1.5 * f0 + (-0.5) * hist(0);
        case 3: return (23.0 / 12.0) * f0 + (-16.0 / 12.0) * hist(0) + (5.0 / 12.0) * hist(1);
        default:
            return (55.0 / 24.0) * f0 + (-59.0 / 24.0) * hist(0) + (37.0 / 24.0) * hist(1) +
                   (-9.0 / 24.0) * hist(2);
    }
}

// Arguments of the adjoint block kernel (one RK2 step, backwards).
struct AdjArgs {
    GridGeom g;
    FieldView f;
    CoefTable<float> cf;
    CoefTable<double> cd;
    int64_t np;
    const int32_t* offsets;   // [nblocks + 1] of the binned positions
    const int32_t* perm;      // sorted position j -> particle index
    const double* pos;        // [3][np] X at the start of the step, particle order
    const double* lam_in;     // [3][np] dLoss/dX' (particle order)
    double* lam_out;          // [3][np] dLoss/dX   (particle order)
    double* gfield;           // [3][N^3] dLoss/dfield (dense, added into) or null
    void* gscratch;           // [nblocks][3][H^3] per-block W^T partial sums (float, or double for
                              // float64 storage), or null: float64 atomics instead
    double dt;
    int* flags;
};

// Arguments of the field-gradient scatter (float32 / split-bf16 fields).
struct AdjScatterArgs {
    GridGeom g;
    CoefTable<float> cf;
    int64_t np;
    const int32_t* offsets;   // [nblocks + 1] of the grouped particles
    const float4* rec;        // [np] records of X
    const float4* adj;        // [3][np] X*, mu, dt/2 lambda (BlockArgs::adj)
    double* gfield;           // [3][N^3] dLoss/dfield (added into)
    float* gscratch;          // [nblocks][3][H^3] per-block sums, or null: float64 atomics instead
};

// One particle set of a batched step, resident in device memory.
struct BatchSet {
    BlockArgs a;              // set's step arguments (field, weights, state buffers)
    int n_items;              // work items of 128 particles
    int I, deg_hi, deriv;
};

constexpr int MAXSEG = 64;    // largest column segment (blocks along x3)

// ---------------------------------------------------------------------------
// Cell split (Sec. 2.2 steps 1-3), bit-exact with the float64 reference:
//   g = X * fl(N/L), c0 = floor(g), t = g - c0, c = c0 mod N.
// __dmul_rn/__dsub_rn forbid fused multiply-adds.  Positions beyond 2^51
// cells are rejected (returned false) together with NaN/Inf.
// ---------------------------------------------------------------------------
// |g| < 2^51, false for NaN and Inf: the biased exponent of g is below
// 1023 + 51 (an integer test, which keeps it off the float64 pipe)
__device__ __forceinline__ bool cell_in_range(double g)
{
    return ((__double2hiint(g) >> 20) & 0x7ff) < 1074;
}

__device__ __forceinline__ bool split_axis(double X, double inv_delta, int mask, int& c, double& t)
{
    const double g = __dmul_rn(X, inv_delta);
    if (!cell_in_range(g)) {
        c = 0;
        t = 0.0;
        return false;
    }
    const double c0 = floor(g);
    t = __dsub_rn(g, c0);
    c = (int)(__double2ll_rz(c0) & (long long)mask);
    return true;
}

// The same cell, and the offset t as a 32-bit fraction (truncated; the offset
// of the float32 kernels, whose weights it enters with 24 bits): one float64
// multiply, then integer shifts of the product's bits.  This GPU runs about
// 1.7 float64 operations per clock and SM, so the floor, difference and
// conversions of split_axis cost a particle ten clocks of that pipe, these
// shifts one and a half issue slots.  |g| in [2^-11, 2^21), which is where
// positions lie, is shifted; other products take the float64 operations.
__device__ __forceinline__ bool split_fixed(double X, double inv_delta, int mask, int& c, uint32_t& frac)
{
    const double g = __dmul_rn(X, inv_delta);
    const int hi = __double2hiint(g);
    const uint32_t lo = (uint32_t)__double2loint(g);
    const int s = 1043 - ((hi >> 20) & 0x7ff);        // |g| 2^32 = m >> s, m the 53-bit significand
    if ((unsigned)s < 32u) {
        const uint32_t mh = ((uint32_t)hi & 0xfffffu) | 0x100000u;
        uint32_t f = __funnelshift_r(lo, mh, s), n = mh >> s;
        if (hi < 0) {   // floor: -m, rounded down where bits were dropped
            const uint32_t exact = (lo & ((1u << s) - 1u)) == 0u ? 1u : 0u;
            f = ~f + exact;
            n = ~n + (f == 0u ? exact : 0u);
        }
        c = (int)(n & (uint32_t)mask);
        frac = f;
        return true;
    }
    c = 0;
    frac = 0;
    if (!cell_in_range(g)) return false;
    const double c0 = floor(g);
    c = (int)(__double2ll_rz(c0) & (long long)mask);
    frac = __double2uint_rz(__dsub_rn(g, c0) * 4294967296.0);   // saturates at t = 1
    return true;
}

// The cell only (for block keys).
__device__ __forceinline__ bool split_cell(double X, double inv_delta, int mask, int& c)
{
    uint32_t frac;
    return split_fixed(X, inv_delta, mask, c, frac);
}

// the offset as the kernels of type T use it
__device__ __forceinline__ bool split_offset(double X, double inv_delta, int mask, int& c, float& t)
{
    uint32_t frac;
    const bool ok = split_fixed(X, inv_delta, mask, c, frac);
    t = __uint2float_rn(frac) * 2.3283064365386963e-10f;   // 2^-32
    return ok;
}
__device__ __forceinline__ bool split_offset(double X, double inv_delta, int mask, int& c, double& t)
{
    return split_axis(X, inv_delta, mask, c, t);
}

// Record of a particle: where it is, as the interpolation reads it.
template <typename T>
struct alignas(4 * sizeof(T)) PRec {
    T t[3];         // offsets in the cell (Sec. 2.2 step 3, normalised by delta)
    T cell;         // c1 | c2 << 10 | c3 << 20, bit-cast into T's storage
};
template <typename T>
__device__ __forceinline__ T cell_as(int c)
{
    if constexpr (sizeof(T) == 4) return __int_as_float(c);
    else return __longlong_as_double((long long)c);
}
__device__ __forceinline__ int cell_of(const PRec<float>& r) { return __float_as_int(r.cell); }
__device__ __forceinline__ int cell_of(const PRec<double>& r) { return (int)__double_as_longlong(r.cell); }
__device__ __forceinline__ void unpack_cell(int p, int (&c)[3])
{
    c[0] = p & 1023, c[1] = p >> 10 & 1023, c[2] = p >> 20 & 1023;
}

// the record of the position pos[3][np] of particle j (non-finite: cell 0, flagged)
template <typename T>
__device__ __forceinline__ PRec<T> split_record(const GridGeom& g, int64_t np, const double* pos, int64_t j, int* flags)
{
    PRec<T> rec;
    int c[3];
    bool ok = true;
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) ok &= split_offset(pos[ax * np + j], g.inv_delta, g.mask, c[ax], rec.t[ax]);
    if (!ok) atomicOr(flags + FLAG_NONFINITE, 1);
    rec.cell = cell_as<T>(c[0] | c[1] << 10 | c[2] << 20);
    return rec;
}

// float32 -> float64 by integer operations for normal numbers (exact)
__device__ __forceinline__ double widen(float x)
{
    const uint32_t b = __float_as_uint(x), e = (b >> 23) & 0xffu;
    if (e - 1u < 254u) return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + (896u << 20))), (int)(b << 29));
    return (double)x;
}
__device__ __forceinline__ double widen(double x) { return x; }

__device__ __forceinline__ uint32_t block_key(const GridGeom& g, int c1, int c2, int c3)
{
    const int b1 = c1 >> g.lb1, b2 = c2 >> g.lb2, b3 = c3 >> g.lb3;
    // rows of blocks along x1; x3 inside a segment of 2^lseg blocks, then x2, the segments along x3
    const int row = ((((b3 >> g.lseg) * g.nb2 + b2) << g.lseg) + (b3 & ((1 << g.lseg) - 1)));
    return (uint32_t)(row * g.nb1 + b1);
}

// ---------------------------------------------------------------------------
// Host-side launchers (defined in the .cu files).  All take a stream and
// return a cudaError_t.
// ---------------------------------------------------------------------------
cudaError_t launch_keys(const GridGeom& g, int64_t np, const double* pos, uint32_t* keys, int* flags,
                        cudaStream_t st);

// Scratch layout for the radix sort of n keys.
size_t radix_scratch_bytes(int64_t n);
// Stable LSD radix sort of (keys, index) by the low `bits` bits of keys.
// keys_sorted and perm receive the result; scratch is radix_scratch_bytes(n).
cudaError_t radix_sort(const uint32_t* keys, int64_t n, int bits, uint32_t* keys_sorted, int32_t* perm,
                       void* scratch, cudaStream_t st, int64_t* launches);

cudaError_t launch_offsets(const uint32_t* keys_sorted, int64_t n, int64_t nblocks, int32_t* offsets,
                           cudaStream_t st);

// Scatter sorted state back to the caller's order: dst[a][id[j]] = src[a][j].
cudaError_t launch_unpermute_pos(int64_t np, const double* src, const int32_t* id, double* dst, cudaStream_t st);
cudaError_t launch_unpermute_rhs(int64_t np, const float* src, const int32_t* id, float* dst, int rows, cudaStream_t st);

// Fill the ghost-padded storage from a dense field src[C][N][N][N] (periodic ghosts).
cudaError_t launch_convert_field(int storage, int src_f64, const void* src, int C, int N, void* dst, cudaStream_t st);
// dLoss/dfield from the per-block partial sums: every node adds, in a fixed
// order, the partials of the non-empty blocks whose halo holds it
cudaError_t launch_adjoint_gather(int I, const AdjArgs& a, cudaStream_t st);
// halo edge of the adjoint kernel for kernel width I (stage-2 margin included)
constexpr int adj_halo(int I) { return BLK + I - 1 + 2; }
cudaError_t launch_adj_particles_i4(const BlockArgs& a, const void* tmap, int deg_hi, cudaStream_t st);
cudaError_t launch_adj_particles_i6(const BlockArgs& a, const void* tmap, int deg_hi, cudaStream_t st);
cudaError_t launch_adj_particles_i8(const BlockArgs& a, const void* tmap, int deg_hi, cudaStream_t st);
cudaError_t launch_adj_scatter_i4(const AdjScatterArgs& a, int64_t nblocks, int deg_hi, cudaStream_t st);
cudaError_t launch_adj_scatter_i6(const AdjScatterArgs& a, int64_t nblocks, int deg_hi, cudaStream_t st);
cudaError_t launch_adj_scatter_i8(const AdjScatterArgs& a, int64_t nblocks, int deg_hi, cudaStream_t st);
// float64 fields
cudaError_t launch_adjoint_i4(const AdjArgs& a, int64_t nblocks, int deg_hi, cudaStream_t st);
cudaError_t launch_adjoint_i6(const AdjArgs& a, int64_t nblocks, int deg_hi, cudaStream_t st);
cudaError_t launch_adjoint_i8(const AdjArgs& a, int64_t nblocks, int deg_hi, cudaStream_t st);

// Exclusive scan of a uint32 array in place; scratch is scan_scratch_bytes_u32(len).
size_t scan_scratch_bytes_u32(int64_t len);
cudaError_t scan_exclusive_u32(uint32_t* data, int64_t len, uint32_t* scratch, cudaStream_t st, int64_t* launches);

// One persistent launch over all sets (float32 or split-bf16 storage).
cudaError_t launch_batched(const BatchSet* sets, int nsets, int* ctr, int nsm, cudaStream_t st);

// Sets the thread-local message returned by tracker_last_error().
void set_error_message(const char* msg);

// True if p points into memory of device dev (or managed memory): the check
// the binning entry points make on caller arrays that their kernels write.
bool device_pointer_ok(const void* p, int dev);

// Block kernels, one entry per kernel width I (block_i4.cu, block_i6.cu, block_i8.cu).
// deg_hi selects the degree-(I+1) instantiation (spline with m = I/2).
// counting-sort binning of the step path: keys with block counts; counts ->
// offsets + cursors (counts zeroed); scatter of the state into its blocks
cudaError_t launch_keys_count(const GridGeom& g, int64_t np, const double* pos, uint32_t* keys, uint32_t* counts,
                              int* flags, cudaStream_t st);
// Small grids are scanned by one CTA (one launch); larger grids take two
// launches over all SMs with count_scan_scratch_bytes of scratch.
size_t count_scan_scratch_bytes(int64_t nblocks);
cudaError_t launch_count_scan(uint32_t* counts, int64_t nblocks, int32_t* offsets, int32_t* cursor,
                              uint32_t* scratch, cudaStream_t st, int64_t* launches);
// counting-sort permutation of keys (cursor from launch_count_scan): perm[d] = j, and the
// records PRec<float or double> rec[d] of pos (null: none)
cudaError_t launch_scatter_perm(const GridGeom& g, int64_t np, const uint32_t* keys, int32_t* cursor, const double* pos,
                                int32_t* perm, void* rec, int rec_f64, int* flags, cudaStream_t st);
// the same for the particle state, with its records
cudaError_t launch_scatter_state(const GridGeom& g, int64_t np, const uint32_t* keys, int32_t* cursor,
                                 const double* pos_in, const int32_t* id_in, const float* rhs_in, int rhs_rows,
                                 double* pos_out, int32_t* id_out, float* rhs_out, void* rec, int rec_f64, int* flags,
                                 cudaStream_t st);
// Block kernels: a.rec_in must hold the records of the grouped particles.
// tmap: a CUtensorMap of the padded field for halo_box(I, margin of the mode) for
// tensor-copy staging, or null for cp.async copies
cudaError_t launch_block_i4(int mode, const BlockArgs& a, const void* tmap, int64_t nblocks, cudaStream_t st);
cudaError_t launch_block_i4h(int mode, const BlockArgs& a, const void* tmap, int64_t nblocks, cudaStream_t st);
cudaError_t launch_block_i6(int mode, const BlockArgs& a, const void* tmap, int64_t nblocks, cudaStream_t st);
cudaError_t launch_block_i6h(int mode, const BlockArgs& a, const void* tmap, int64_t nblocks, cudaStream_t st);
cudaError_t launch_block_i8(int mode, const BlockArgs& a, const void* tmap, int64_t nblocks, cudaStream_t st);
cudaError_t launch_block_i8h(int mode, const BlockArgs& a, const void* tmap, int64_t nblocks, cudaStream_t st);
// direct path: a.np grouped particles, a.ppc per CTA, stencils from global memory
cudaError_t launch_direct_i4(int mode, const BlockArgs& a, int deg_hi, cudaStream_t st);
cudaError_t launch_direct_i6(int mode, const BlockArgs& a, int deg_hi, cudaStream_t st);
cudaError_t launch_direct_i8(int mode, const BlockArgs& a, int deg_hi, cudaStream_t st);

}  // namespace trk
