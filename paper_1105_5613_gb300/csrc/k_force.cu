// Pair forces of the truncated Lennard-Jones / soft-sphere mixture (Sec. 2.1, Eqs. lj0,
// sc0, mod0) over the cell stencil (Sec. 2.2), and the Verlet-list build.
//
// Work unit: one CTA per block of cells; its warps take the block's items in turn (list-mode
// forces: chunks of 32 own particles of one species across the block's cells; stencil forces:
// cells; list build: a cell's first 32 particles, and the rest).  The CTA stages the cells of the
// block and one cell around it -- the union of their 27-cell stencils -- into shared memory
// as float4 {x, y, z, species} in one frame (the block's centre).  The raw
// frame-relative records of each cell arrive by one TMA bulk copy per cell (cells are
// contiguous after the counting sort); the exact frame offsets are then added in shared
// memory.  Each lane owns one particle i and accumulates its force in registers: a full
// list, one writer per i, no atomics (the paper applies Newton's third law to halve the
// pair work on a CPU; here every pair is visited from both sides so that each force has
// a single owner and a fixed summation order).
//
// The Verlet list stores, per particle, uint16 offsets into the block's staged array,
// laid out as [kb][npad][8] so a warp reads 8 entries per lane with one coalesced 16-byte
// load.  Padding entries point to a sentinel far outside every cutoff.
//
// Mixed precision: distances and forces in FP32 from block-frame coordinates.  A pair is
// taken as interacting when its FP32 r^2 is below rc^2 (1 - 1e-5); a pair within that
// relative band of the cutoff is decided by the exact FP64 rule in a rare fix-up after
// each batch of 8 pairs, so the interacting set equals the FP64 definition.
//
// This file is compiled once per block shape, code BBMD_BLOCK_Z = 1, 2 or 4 (2 x 2 x Z
// cells) or 8 (4 x 4 x 2 cells), into namespace bbmd::z<BBMD_BLOCK_Z>; the handle picks one
// shape at creation.
#include <climits>
#include <cstddef>

#include "bbmd_internal.cuh"
#include "stage_loop.cuh"

#ifndef BBMD_BLOCK_Z
#error "k_force.cu is compiled once per block shape: define BBMD_BLOCK_Z (code 1, 2, 4 or 8)"
#endif
// warps per CTA and resident CTAs per SM targeted by the force and list kernels, per shape
#if BBMD_BLOCK_Z == 1
#define BBMD_SHAPE_WARPS 4
#define BBMD_SHAPE_FORCE_MIN 6
#define BBMD_SHAPE_LIST_MIN 6
#elif BBMD_BLOCK_Z == 2
#define BBMD_SHAPE_WARPS 8
#define BBMD_SHAPE_FORCE_MIN 3
#define BBMD_SHAPE_LIST_MIN 3
#elif BBMD_BLOCK_Z == 4
#define BBMD_SHAPE_WARPS 8
#define BBMD_SHAPE_FORCE_MIN 2
#define BBMD_SHAPE_LIST_MIN 3
#elif BBMD_BLOCK_Z == 8
#define BBMD_SHAPE_WARPS 8
#define BBMD_SHAPE_FORCE_MIN 2
#define BBMD_SHAPE_LIST_MIN 2
#else
#error "BBMD_BLOCK_Z must be 1, 2, 4 or 8"
#endif
// BBMD_WIDE (with shape 1): only the one-launch kernels, with eight warps a CTA, in namespace
// z1w -- for systems so small that a block has an SM to itself
#ifndef BBMD_WIDE
#define BBMD_WIDE 0
#endif
#ifndef BBMD_BLOCK_WARPS
#define BBMD_BLOCK_WARPS (BBMD_WIDE ? 8 : BBMD_SHAPE_WARPS)
#endif
#ifndef BBMD_FORCE_MIN_BLOCKS
#define BBMD_FORCE_MIN_BLOCKS BBMD_SHAPE_FORCE_MIN
#endif
// the stencil (cell-mode) force kernel of a 2 x 2 x 4 block fits three CTAs per SM in
// shared memory; bounded to them it compiles to 80 registers
#ifndef BBMD_CELL_MIN_BLOCKS
#define BBMD_CELL_MIN_BLOCKS (BBMD_BLOCK_Z == 4 ? 3 : BBMD_FORCE_MIN_BLOCKS)
#endif
#ifndef BBMD_LIST_MIN_BLOCKS
#define BBMD_LIST_MIN_BLOCKS BBMD_SHAPE_LIST_MIN
#endif
#define BBMD_CAT2(a, b) a##b
#define BBMD_CAT(a, b) BBMD_CAT2(a, b)

namespace bbmd {
#if BBMD_WIDE
namespace z1w {
#else
namespace BBMD_CAT(z, BBMD_BLOCK_Z) {
#endif

namespace {

constexpr unsigned FULL = 0xffffffffu;
constexpr float kFar = 1.0e15f;
constexpr int kBlockXY = block_xy_of(BBMD_BLOCK_Z);  // cells of a block along x and y
constexpr int kBlockZ = block_zc_of(BBMD_BLOCK_Z);   // cells of a block along z
constexpr int kRXY = kBlockXY + 2;                   // region cells along x and y
constexpr int kBW = BBMD_BLOCK_WARPS;                // warps per CTA
constexpr int kCells = block_cells_of(BBMD_BLOCK_Z);   // cells per block
constexpr int kRegion = region_cells_of(BBMD_BLOCK_Z);  // cells staged per block
static_assert(kRegion <= kBW * 32, "one thread per staged region cell");
#ifndef BBMD_LIST_AHEAD
#define BBMD_LIST_AHEAD 2
#endif
constexpr int kListAhead = BBMD_LIST_AHEAD;  // list rows in flight ahead of the pair loop
#ifndef BBMD_LIST_PREFETCH
#define BBMD_LIST_PREFETCH 4
#endif
// list rows prefetched into L2 this many rows ahead of the pair loop (0: none), so that
// the register loads two rows ahead find them in L2 rather than in DRAM
constexpr int kListPrefetch = BBMD_LIST_PREFETCH;

__device__ __forceinline__ float rcp_approx(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// The region of cells staged for one block: (X + 2) x (Y + 2) x (Z + 2) cells, index
// q = (z * (Y + 2) + y) * (X + 2) + x.
struct Region {
    int off[kRegion + 1];      // prefix of staged counts (clamped to smax); off[kRegion] = total
    int start[kRegion];        // first particle of each region cell
    int cnt[kRegion];          // particles of each region cell
    int nstaged;
    // used while a block is staged (and by the FP64 staging); free for the block's own work
    alignas(16) float hi[kRegion][3];  // frame offset of each cell (FP32 rounding of the exact value)
    float lo[kRegion][3];      // exact residual of that rounding (non-zero across the seam)
    long long fr[kRegion][3];  // FP64 form: frame point + seam image of each cell
};

// ------------------------------------------------ TMA bulk copies and mbarriers ----

__device__ __forceinline__ void prefetch_l2(const void* p) {
    asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(uint64_t* mbar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(mbar)), "r"(count)
                 : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

// (the memory may then be initialised again, or used for something else)
__device__ __forceinline__ void mbar_inval(uint64_t* mbar) {
    asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(smem_u32(mbar)) : "memory");
}

__device__ __forceinline__ void fence_proxy_async_smem() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* mbar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(mbar)),
                 "r"(bytes)
                 : "memory");
}

// Bulk copy of `bytes` (multiple of 16, both addresses 16-byte aligned) global -> shared,
// completion counted on the mbarrier.
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes,
                                         uint64_t* mbar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
            "r"(smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(mbar))
        : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* mbar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok)
        : "r"(smem_u32(mbar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Wait for the current phase, kStageTries tries at most (LIMIT: s.stage_tries).  On expiry raise
// ST_TIMEOUT, wait once more (again bounded) for the copies still in flight, and return false.
template <bool LIMIT>
__device__ __forceinline__ bool mbar_wait_bounded(const DevSim& s, uint64_t* mbar, uint32_t parity) {
    const uint32_t tries = LIMIT ? s.stage_tries : kStageTries;
    for (uint32_t it = 0; it < tries; ++it)
        if (mbar_try_wait(mbar, parity)) return true;
    set_status(s, ST_TIMEOUT);
    for (uint32_t it = 0; it < kStageTries; ++it)
        if (mbar_try_wait(mbar, parity)) break;
    return false;
}

// ------------------------------------------------------------------ blocks ----

struct BlockPos {
    int a0[3];  // first cell of the block per axis
};

__device__ __forceinline__ BlockPos block_pos(const DevSim& s, int64_t blk) {
    const int nbx = (s.nc[0] + kBlockXY - 1) / kBlockXY, nby = (s.nc[1] + kBlockXY - 1) / kBlockXY;
    BlockPos b;
    b.a0[0] = (int)(blk % nbx) * kBlockXY;
    b.a0[1] = (int)((blk / nbx) % nby) * kBlockXY;
    b.a0[2] = (int)(blk / ((int64_t)nbx * nby)) * kBlockZ;
    return b;
}

// Describe the region of block b (threads 0..kRegion-1 take one region cell each): counts,
// frame offsets relative to the block frame, prefix.
__device__ void region_info(const DevSim& s, const BlockPos& b, Region& R) {
    __shared__ int wtot[(kRegion + 31) / 32];
    const int tid = threadIdx.x, lane = tid & 31;
    int cnt = 0;
    if (tid < kRegion) {
        const int r[3] = {tid % kRXY, (tid / kRXY) % kRXY, tid / (kRXY * kRXY)};
        int a[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            int aa = b.a0[d] - 1 + r[d];
            long long wrap = 0;
            if (aa < 0) {
                aa += s.nc[d];
                wrap = -s.Lfix[d];
            } else if (aa >= s.nc[d]) {
                aa -= s.nc[d];
                wrap = s.Lfix[d];
            }
            a[d] = aa;
            // block frame: the cell boundary at the middle of the block (along z, the centre
            // of the cell when the block is one cell high)
            const long long fb = d < 2 ? (long long)(b.a0[d] + kBlockXY / 2) * s.D[d]
                                 : kBlockZ == 1 ? frame_axis(b.a0[d], s.D[d])
                                                : (long long)(b.a0[d] + kBlockZ / 2) * s.D[d];
            const long long fr = frame_axis(aa, s.D[d]) + wrap;
            const long long delta = fr - fb;
            const float hi = i64_to_f32(delta) * s.sx;
            const long long rest = delta - f32_to_i64(hi * pow2f(s.kexp));
            R.hi[tid][d] = hi;
            R.lo[tid][d] = i64_to_f32(rest) * s.sx;
            R.fr[tid][d] = fr;
        }
        const int nb = (a[2] * s.nc[1] + a[1]) * s.nc[0] + a[0];
        const int st = s.cell_start[nb];
        cnt = cell_count(st, s.cell_start[nb + 1], s.smax);
        R.start[tid] = st;
        R.cnt[tid] = cnt;
    }
    // every lane of the warps that cover the region takes part in the scan (lanes past the
    // region carry a count of zero)
    int incl = cnt;
    if (tid < ((kRegion + 31) & ~31)) {
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int t = __shfl_up_sync(FULL, incl, o);
            if (lane >= o) incl += t;
        }
        if (lane == 31) wtot[tid >> 5] = incl;
    }
    __syncthreads();
    if (tid < kRegion) {
        int base = 0;
        for (int k = 0; k < (tid >> 5); ++k) base += wtot[k];
        int ex = base + incl - cnt;
        R.off[tid] = min(ex, s.smax);
        if (tid == kRegion - 1) {
            int total = base + incl;
            R.off[kRegion] = min(total, s.smax);
            R.nstaged = min(total, s.smax);
            if (total > s.smax)
                set_status(s, s.sums_role == kSumsSmaller ? ST_SUMS_SHORT : ST_STENCIL_OVERFLOW);
        }
    }
    __syncthreads();
}

// Start staging block b into sm (mixed precision): describe its region, then one TMA bulk
// copy per region cell of the raw frame-relative records, counted on mbar.  Does not wait.
// All threads of the CTA call it; the previous reads of sm must be complete (barrier).
__device__ void issue_block(const DevSim& s, const BlockPos& b, Region& R, float4* sm,
                            uint64_t* mbar) {
    fence_proxy_async_smem();  // earlier generic accesses of sm before the async writes
    region_info(s, b, R);
    const int tid = threadIdx.x;
    if (tid == 0) mbar_arrive_expect_tx(mbar, (uint32_t)R.nstaged * 16u);
    __syncthreads();
    if (tid < kRegion) {
        const int n = R.off[tid + 1] - R.off[tid];
        if (n > 0) bulk_g2s(sm + R.off[tid], s.rel + R.start[tid], (uint32_t)n * 16u, mbar);
    }
}

// Wait for the copies of a block issued with issue_block, add the frame offsets of every
// region cell (exact residual first), write the sentinel sm[smax] and synchronise.
// Returns false on every thread of the CTA if some thread's wait gave up.
template <bool LIMIT>
__device__ bool finish_block(const DevSim& s, const Region& R, float4* sm, uint64_t* mbar,
                             uint32_t parity) {
    const bool ok = mbar_wait_bounded<LIMIT>(s, mbar, parity);
    if (__syncthreads_or(!ok)) return false;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    for (int q = w; q < kRegion; q += kBW) {
        const int o0 = R.off[q], cq = R.off[q + 1] - o0;
        const float hx = R.hi[q][0], hy = R.hi[q][1], hz = R.hi[q][2];
        const float lx = R.lo[q][0], ly = R.lo[q][1], lz = R.lo[q][2];
        for (int t = lane; t < cq; t += 32) {
            float4 v = sm[o0 + t];
            v.x = (v.x + lx) + hx;
            v.y = (v.y + ly) + hy;
            v.z = (v.z + lz) + hz;
            sm[o0 + t] = v;
        }
    }
    if (tid == 0) sm[s.smax] = make_float4(kFar, kFar, kFar, 0.f);
    __syncthreads();
    return true;
}

#ifndef BBMD_STAGE_BUFFERS
#define BBMD_STAGE_BUFFERS 1  // 2: stage block i+1 while block i is computed
#endif
constexpr int kStageBuffers = BBMD_STAGE_BUFFERS;

// LIMIT: staging waits take the handle's limit (s.stage_tries), in the kernels of several phases,
// which must not go on after one that gave up.  Those of one phase keep the default (a limit that
// is looked up costs their list-mode forces up to 1.8 %).
template <bool LIMIT>
struct StageOps {
    float4* smem;
    int stride;  // records of a buffer
    Region* R;
    uint64_t* mbar;

    __device__ __forceinline__ void open() {
        if (threadIdx.x == 0)
            for (int k = 0; k < kStageBuffers; ++k) mbar_init(&mbar[k], 1);
        __syncthreads();
    }
    __device__ __forceinline__ BlockPos position(const DevSim& s, int64_t blk) { return block_pos(s, blk); }
    __device__ __forceinline__ void issue(const DevSim& s, const BlockPos& pos, int b) {
        issue_block(s, pos, R[b], smem + b * stride, &mbar[b]);
    }
    __device__ __forceinline__ bool finish(const DevSim& s, int b, uint32_t parity) {
        return finish_block<LIMIT>(s, R[b], smem + b * stride, &mbar[b], parity);
    }
    template <class Body>
    __device__ __forceinline__ void compute(const BlockPos& pos, int b, Body& body) {
        body(pos, R[b], smem + b * stride, b);
    }
    __device__ __forceinline__ void drain(const DevSim& s, int b, uint32_t parity) {
        mbar_wait_bounded<LIMIT>(s, &mbar[b], parity);
    }
    __device__ __forceinline__ void sync() { __syncthreads(); }
    __device__ __forceinline__ void close() {
        if (threadIdx.x == 0)
            for (int k = 0; k < kStageBuffers; ++k) mbar_inval(&mbar[k]);
    }
};

// Blocks of this CTA in order (grid-stride): body(pos, R, sm, b) computes one staged block,
// from buffer b, and must not synchronise the CTA.  False (on every thread) if a staging wait
// gave up (see staged_blocks).
template <bool LIMIT, class Body>
__device__ __forceinline__ bool for_each_block(const DevSim& s, int lb, int lg, float4* smem, int stride,
                                               Region* R, uint64_t* mbar, Body body) {
    return staged_blocks<kStageBuffers>(s, StageOps<LIMIT>{smem, stride, R, mbar}, lb, lg, body);
}

// Particles of region cell q that were staged: all of them unless the region overflowed
// the staged capacity (flagged, the results are then discarded), so a lane never reads
// past the staged records.
__device__ __forceinline__ int staged_count(const Region& R, int q) {
    return min(R.cnt[q], R.off[q + 1] - R.off[q]);
}

// Global index of staged entry t (rare path).
__device__ __forceinline__ int64_t staged_global(const Region& R, int t) {
    return staged_particle(R.start, R.off, kRegion, t);
}

// The warp's own cell: its region index and whether it exists (odd nc leaves some warps of
// the last block along an axis idle).
struct WarpCell {
    int c;      // cell id
    int rq;     // region index of the cell
    int wr[3];  // region coordinates of the stencil's first cell per axis
    bool valid;
};

__device__ __forceinline__ WarpCell warp_cell(const DevSim& s, const BlockPos& b, int w) {
    WarpCell wc;
    const int o[3] = {w % kBlockXY, (w / kBlockXY) % kBlockXY, w / (kBlockXY * kBlockXY)};
    int a[3];
    wc.valid = true;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        a[d] = b.a0[d] + o[d];
        if (a[d] >= s.nc[d]) wc.valid = false;
        wc.wr[d] = o[d];
    }
    wc.c = wc.valid ? (a[2] * s.nc[1] + a[1]) * s.nc[0] + a[0] : 0;
    wc.rq = ((1 + o[2]) * kRXY + (1 + o[1])) * kRXY + (1 + o[0]);
    return wc;
}

// Per-lane pair constants for the lane's species; field suffix = species of j.  Kept as
// scalars and picked with selects so that nothing is indexed at run time.
struct LaneTab {
    float rlo0, rlo1, rhi0, rhi1, sig20, sig21, e480, e481;
    float e40, e41, vsh0, vsh1, fc0, fc1, rc0, rc1, sgl0, sgl1;
    float cpot;   // 0.5 for LJ force, 0 for soft sphere
    float cpe;    // 1 for LJ energy, 0 for soft sphere
    float rm0, rm1, hw;  // list mode: middle of the band around rc^2, half-width (both j)
    int si;
};

__device__ __forceinline__ void load_tab(const DevSim& s, int si, LaneTab& T) {
    const int k = si * 2;
    T.rlo0 = s.pt.rc2lo[k];      T.rlo1 = s.pt.rc2lo[k + 1];
    T.rhi0 = s.pt.rc2hi[k];      T.rhi1 = s.pt.rc2hi[k + 1];
    T.rm0 = 0.5f * (T.rlo0 + T.rhi0);
    T.rm1 = 0.5f * (T.rlo1 + T.rhi1);
    T.hw = 0.5f * fmaxf(T.rhi0 - T.rlo0, T.rhi1 - T.rlo1);
    T.sig20 = s.pt.sig2[k];      T.sig21 = s.pt.sig2[k + 1];
    T.sgl0 = s.pt.sig2lo[k];     T.sgl1 = s.pt.sig2lo[k + 1];
    T.e480 = s.pt.eps48[k];      T.e481 = s.pt.eps48[k + 1];
    T.e40 = s.pt.eps4[k];        T.e41 = s.pt.eps4[k + 1];
    T.vsh0 = s.pt.vshift[k];     T.vsh1 = s.pt.vshift[k + 1];
    T.fc0 = s.pt.fcut[k];        T.fc1 = s.pt.fcut[k + 1];
    T.rc0 = s.pt.frc[k];         T.rc1 = s.pt.frc[k + 1];
    T.cpot = s.pt.potential == BBMD_POT_LJ ? 0.5f : 0.0f;
    T.cpe = s.pt.potential == BBMD_POT_LJ ? 1.0f : 0.0f;
    T.si = si;
}

struct Acc {
    float fx, fy, fz;
};

// Force of one pair; contributes only when `in`.  d = x_j - x_i.  (Pair energies and the
// virial are evaluated by the FP64 energy pass, from exact integer positions.)
template <bool FSHIFT>
__device__ __forceinline__ void pair_add(const LaneTab& T, bool b, float dx, float dy, float dz,
                                         float r2, bool in, Acc& a) {
    float ir2 = rcp_approx(r2);
    float s2 = (b ? T.sig21 : T.sig20) * ir2;
    float s6 = s2 * s2 * s2;
    float f = (b ? T.e481 : T.e480) * ir2 * s6 * (s6 - T.cpot);
    if (FSHIFT) f = fmaf(b ? T.fc1 : T.fc0, rsqrtf(r2), f);
    f = in ? f : 0.f;
    a.fx = fmaf(f, dx, a.fx);
    a.fy = fmaf(f, dy, a.fy);
    a.fz = fmaf(f, dz, a.fz);
}

// Scalar forces f of two interacting pairs with the constants of their species pair given
// (the stencil kernel loads them per candidate stream); the arithmetic of pair_add.
template <bool FSHIFT>
__device__ __forceinline__ float2 pair_f2(float sig2, float e48, float cpot, float fc, float2 r2) {
    const float2 ir2 = make_float2(rcp_approx(r2.x), rcp_approx(r2.y));
    const float2 s2 = __fmul2_rn(make_float2(sig2, sig2), ir2);
    const float2 s6 = __fmul2_rn(__fmul2_rn(s2, s2), s2);
    float2 f = __fmul2_rn(__fmul2_rn(__fmul2_rn(make_float2(e48, e48), ir2), s6),
                          __fadd2_rn(s6, make_float2(-cpot, -cpot)));
    if (FSHIFT) f = __ffma2_rn(make_float2(fc, fc), make_float2(rsqrtf(r2.x), rsqrtf(r2.y)), f);
    return f;
}

// Fast path of one list pair (i, staged t), classified by d = r^2 - (middle of the band
// around rc^2 for the species of j): interacting iff d <= -hw; |d| < hw is the band,
// left to the exact fix-up; the smallest |d| of a batch tells whether it has band pairs.
template <bool FSHIFT>
__device__ __forceinline__ void pair_fast(const LaneTab& T, float4 me, float4 p, Acc& a, float& near) {
    float dx = p.x - me.x, dy = p.y - me.y, dz = p.z - me.z;
    float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
    const bool b = p.w != 0.f;
    const float d = r2 - (b ? T.rm1 : T.rm0);
    near = fminf(near, fabsf(d));
    pair_add<FSHIFT>(T, b, dx, dy, dz, r2, d <= -T.hw, a);
}

// A staged copy is usable only in the minimum image (the 4x4x4 region holds a cell twice
// when nc = 3; the two copies are at least a cell side apart from any tile particle).
__device__ __forceinline__ bool min_image_copy(const DevSim& s, float dx, float dy, float dz) {
    return fabsf(dx) < s.halfL[0] && fabsf(dy) < s.halfL[1] && fabsf(dz) < s.halfL[2];
}

// Exact decision for a band pair; adds its force if the FP64 rule says it interacts.  It
// runs for a few pairs per million.  Called out of line (pair_band_call), it keeps the
// lane's pair constants and accumulators in local memory (a stack frame); inline, it
// costs registers.  Inline is faster where the list kernel has 128 registers a thread
// (shapes 4 and 8: 6 % at 2 M particles); out of line where it has fewer (2 x 2 x 1 and
// 2 x 2 x 2: inline is 20 % slower there), and in the persistent batch
// kernel, whose other phases share the register budget (inline, some of its forms spill).
#ifndef BBMD_BAND_INLINE
#define BBMD_BAND_INLINE (BBMD_BLOCK_Z >= 4)
#endif
constexpr bool kBandInline = BBMD_BAND_INLINE;
template <bool FSHIFT>
__device__ __forceinline__ void pair_band(const DevSim& s, const Region& R, const LaneTab& T, float4 me, float4 p,
                          int t, int64_t gi, bool valid, Acc& a) {
    float dx = p.x - me.x, dy = p.y - me.y, dz = p.z - me.z;
    float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
    const bool b = p.w != 0.f;
    if (!valid || !(fabsf(r2 - (b ? T.rm1 : T.rm0)) < T.hw)) return;
    if (!min_image_copy(s, dx, dy, dz)) return;
    int64_t gj = staged_global(R, t);
    if (r2_exact(s, gi, gj) < s.pt.rc2[T.si * 2 + (b ? 1 : 0)])
        pair_add<FSHIFT>(T, b, dx, dy, dz, r2, true, a);
}

template <bool FSHIFT>
__device__ __noinline__ void pair_band_call(const DevSim& s, const Region& R, const LaneTab& T, float4 me,
                                            float4 p, int t, int64_t gi, bool valid, Acc& a) {
    pair_band<FSHIFT>(s, R, T, me, p, t, gi, valid, a);
}

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(FULL, v, o);
    return v;
}

// Sum of the lanes' kinetic energies k in units of 2^-32, rounded once.  Where every lane's is
// zero or in [2^-17, 2^18): the lanes' values in units of 2^-40, which hold them exactly, summed
// as three limbs by the warp's integer reduction.  Else (a system far colder than any liquid, or
// flying apart) the sum in FP64, which takes the FP64 pipe 8 x 16 clocks a chunk (forces at
// 16.4 M particles, 4 x 4 x 2: 2.95 -> 2.90 ms without it).
__device__ __forceinline__ unsigned long long chunk_energy(float k) {
    const bool exact = k < 0x1p18f && (k >= 0x1p-17f || k == 0.f);
    if (!__all_sync(FULL, exact)) return __double2ull_rn(warp_sum_d((double)k) * 0x1p32);
    const unsigned long long q = (unsigned long long)f32_to_i64(k * 0x1p40f);
    const unsigned s0 = __reduce_add_sync(FULL, (unsigned)q & 0x3ffffffu);
    const unsigned s1 = __reduce_add_sync(FULL, (unsigned)(q >> 26) & 0x3ffffffu);
    const unsigned s2 = __reduce_add_sync(FULL, (unsigned)(q >> 52));
    const unsigned long long t = s0 + ((unsigned long long)s1 << 26) + ((unsigned long long)s2 << 52);
    return (t + 0x7f + ((t >> 8) & 1)) >> 8;  // to nearest, ties to even
}

// Block reduction of per-warp doubles wv[0 .. nq) (lane 0 of each warp) into
// partials[(q0 + q) * kMaxPartials + lb], in a fixed order.
__device__ void block_partials(const DevSim& s, int lb, const double* wv, int q0, int nq) {
    __shared__ double red[kBW][4];
    int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (lane == 0)
        for (int q = 0; q < nq; ++q) red[w][q] = wv[q];
    __syncthreads();
    if (threadIdx.x < nq) {
        double t = 0.0;
        for (int k = 0; k < kBW; ++k) t += red[k][threadIdx.x];
        s.partials[(q0 + threadIdx.x) * kMaxPartials + lb] = t;
    }
}

__device__ __forceinline__ unsigned lo16(unsigned w) { return w & 0xffffu; }
__device__ __forceinline__ unsigned hi16(unsigned w) { return w >> 16; }

// Contiguous staged range of stencil row (dy, dz) of the warp's cell: three consecutive
// region cells along x.
__device__ __forceinline__ void stencil_run(const Region& R, const WarpCell& wc, int row, int& rs,
                                            int& re) {
    const int ry = wc.wr[1] + row % 3, rz = wc.wr[2] + row / 3;
    const int q0 = (rz * kRXY + ry) * kRXY + wc.wr[0];
    rs = R.off[q0];
    re = R.off[q0 + 3];
}

// ------------------------------------------------------- stencil compaction ----
// A stencil candidate farther than the reach from the bounding box of the warp's particles
// pairs with none of them.  Such candidates are dropped, 32 at a time, before the per-lane
// tests. The survivors keep their stencil order within their species' stream (below). The
// lists and force sums therefore hold exactly the pairs that testing every candidate finds.
// The reach carries a relative margin of 2^-9. Against it, FP32 rounding of the staged
// coordinates and of the box distance (about 1e-6 relative) is negligible. A dropped
// candidate lies beyond the upper edge of the exact-test band for every lane.

struct WarpBox {
    float lo[3], hi[3];
};

// Shared memory that the force and list bodies use in turn: the staged region's
// description and its mbarriers, and the per-warp candidate rings.  One instance per
// kernel, whichever bodies it runs (a kernel running several bodies, such as the
// persistent batch step, does not pay for each body's own copy).
struct StageShared {
    Region R[kStageBuffers];
    uint64_t mbar[kStageBuffers];
    // the block's work items (cells, or chunks of 32 particles) are handed to the warps in
    // turn as they come free (a count per block parity: one in use, the other reset for
    // the next block)
    int next_cell[2];
    // list-mode chunks of the block: the own particles, species A first then B (each cell
    // holds its A particles first), 32 to a chunk across the block's cells.  Per own cell
    // (in cell order): staged offset, first particle, count, A count; prefixes of the A
    // and B counts; the number of A chunks and of all chunks.
    int c_off[kCells], c_i0[kCells], c_n[kCells], c_nA[kCells];
    int prefA[kCells + 1], prefB[kCells + 1];
    int nchA, nch;
    // kinetic energy of the CTA's chunks in 2^-32 fixed point: integer sums do not depend
    // on which warp added which chunk when
    unsigned long long ke_fix;
};

// Lane `lane` of list-mode chunk `item` of the block: the particle's ordinal o among the
// block's particles of the chunk's species, its cell q (the last whose prefix is <= o: a
// cell with particles), its global index gi and staged index self.
__device__ __forceinline__ void chunk_lane(const StageShared& ss, int item, int lane, bool& act,
                                           int64_t& gi, int& self) {
    const bool isB = item >= ss.nchA;
    const int o = (isB ? item - ss.nchA : item) * 32 + lane;
    const int* pref = isB ? ss.prefB : ss.prefA;
    act = o < pref[kCells];
    int q = 0, hi = kCells - 1;
    while (q < hi) {
        const int mid = (q + hi + 1) >> 1;
        if (pref[mid] <= o) q = mid;
        else hi = mid - 1;
    }
    const int li = (isB ? ss.c_nA[q] : 0) + (o - pref[q]);
    gi = act ? (int64_t)ss.c_i0[q] + li : 0;
    self = act ? ss.c_off[q] + li : 0;
}

// The cell (within the block) of lane `lane`'s particle of chunk `item`.
__device__ __forceinline__ int chunk_cell(const StageShared& ss, int item, int lane) {
    const bool isB = item >= ss.nchA;
    const int o = (isB ? item - ss.nchA : item) * 32 + lane;
    const int* pref = isB ? ss.prefB : ss.prefA;
    int q = 0, hi = kCells - 1;
    while (q < hi) {
        const int mid = (q + hi + 1) >> 1;
        if (pref[mid] <= o) q = mid;
        else hi = mid - 1;
    }
    return q;
}

// Describe the block's chunks (ss.c_*, ss.pref*, ss.nchA, ss.nch).  is_A(t): staged particle
// t is of species A.  Every thread of the CTA calls it; it synchronises.
template <class IsA>
__device__ __forceinline__ void own_chunks(const DevSim& s, const BlockPos& bp, const Region& Rc,
                                           StageShared& ss, IsA is_A) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int cw = w; cw < kCells; cw += kBW) {
        const WarpCell wc = warp_cell(s, bp, cw);
        const int cnt = wc.valid ? staged_count(Rc, wc.rq) : 0;
        const int off = Rc.off[wc.rq];
        int nA = 0;  // the cell's A particles come first
        for (int t = 0; t < cnt; t += 32) {
            const unsigned b = __ballot_sync(FULL, t + lane < cnt && is_A(off + t + lane));
            nA += __popc(b);
            if (b != FULL) break;
        }
        if (lane == 0) {
            ss.c_off[cw] = off;
            ss.c_i0[cw] = wc.valid ? Rc.start[wc.rq] : 0;
            ss.c_n[cw] = cnt;
            ss.c_nA[cw] = nA;
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        int na = 0, nb = 0;
        for (int c = 0; c < kCells; ++c) {
            ss.prefA[c] = na;
            ss.prefB[c] = nb;
            na += ss.c_nA[c];
            nb += ss.c_n[c] - ss.c_nA[c];
        }
        ss.prefA[kCells] = na;
        ss.prefB[kCells] = nb;
        ss.nchA = (na + 31) >> 5;
        ss.nch = ss.nchA + ((nb + 31) >> 5);
    }
    __syncthreads();
}

// The next work item of the block for this warp (at least the item count when none is
// left).
__device__ __forceinline__ int take_cell(StageShared& ss, int par, int lane) {
    int cw = 0;
    if (lane == 0) cw = atomicAdd(&ss.next_cell[par], 1);
    return __shfl_sync(0xffffffffu, cw, 0);
}

__device__ __forceinline__ StageShared& stage_shared() {
    __shared__ __align__(16) StageShared ss;
    return ss;
}

// Bounding box of the active lanes' positions.
__device__ __forceinline__ WarpBox warp_box(float4 me, bool act) {
    WarpBox b;
    b.lo[0] = act ? me.x : kFar;
    b.lo[1] = act ? me.y : kFar;
    b.lo[2] = act ? me.z : kFar;
    b.hi[0] = act ? me.x : -kFar;
    b.hi[1] = act ? me.y : -kFar;
    b.hi[2] = act ? me.z : -kFar;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            b.lo[d] = fminf(b.lo[d], __shfl_xor_sync(FULL, b.lo[d], o));
            b.hi[d] = fmaxf(b.hi[d], __shfl_xor_sync(FULL, b.hi[d], o));
        }
    }
    return b;
}

// Position in the warp's 27-cell stencil: row (dy, dz) and the next group start g0 in the
// row's staged range [., re).
struct StencilScan {
    int row, g0, re;
};

// Advance to the next non-empty row if the current one is exhausted; false at the end.
__device__ __forceinline__ bool scan_next(const Region& R, const WarpCell& wc, StencilScan& sc) {
    while (sc.g0 >= sc.re) {
        if (++sc.row == 9) return false;
        stencil_run(R, wc, sc.row, sc.g0, sc.re);
    }
    return true;
}

// Squared reach from the box for a candidate of species 0 / 1: the largest upper band edge
// over the lane species, widened by 2^-9.
__device__ __forceinline__ float keep_reach(const float* hi4, int sj) {
    return fmaxf(hi4[sj], hi4[2 + sj]) * (1.0f + 0x1p-9f);
}

// ------------------------------------------------- species-split candidate streams ----
// The list build compacts the stencil candidates within reach of the warp's box into two
// streams, one per species of the candidate.  An entry holds the candidate relative to the
// box centre c, p' = p - c, and q = |p'|^2; a parallel ring holds its staged index.  A
// lane (m' = its own position - c) then tests a candidate of stream S as
//     r^2 - R^2(s_i, S) = q + (|m'|^2 - R^2(s_i, S)) - 2 p'.m'
// (an add and three FMAs after one broadcast load; the threshold is the same for the
// whole stream).  Relative to the box centre, |p'| stays below the box half-diagonal plus
// the reach (about 6 cell sides' worth of r^2 at most), so the FP32 error of this form is
// about 1e-5 in r^2, below the margin of the exact-test band (the band's edges lie at a
// relative 1e-5 and 3e-5 from R^2, about 8e-5 and 2.4e-4 at the bench's R^2 = 7.84).
// The band test uses the same form, so the candidates it sends to the exact rule are
// exactly those whose FP32 value could be on the wrong side.
constexpr int kSRing = 64;  // entries per stream ring (two 32-entry words; a power of two)

// One array per component, so that four (two pairs of) candidates come with one 16-byte
// broadcast read per component, and a lane that picks one entry of a word reads one of 32
// consecutive words per component (no bank conflicts among the lanes).
struct StreamRings {
    float x[2][kSRing], y[2][kSRing], z[2][kSRing], q[2][kSRing];  // p' = p - c, |p'|^2
    uint16_t idx[2][kSRing];   // staged index
    float4 box[2];             // (c, reach^2 of species A), (half-extents, reach^2 of B)
};

// The word of 32 entries of stream S that starts at cq (a multiple of 32).
struct StreamWord {
    const float *x, *y, *z, *q;
};

__device__ __forceinline__ StreamWord stream_word(const StreamRings& SR, int S, int cq) {
    const int o = cq & (kSRing - 1);
    return {SR.x[S] + o, SR.y[S] + o, SR.z[S] + o, SR.q[S] + o};
}

__device__ __forceinline__ StreamRings& warp_streams(int w) {
    __shared__ __align__(16) StreamRings rings_all[kBW];
    return rings_all[w];
}

// The warp's box as centre and half-extents, kept with the reaches in the warp's
// shared-memory slot (the compaction reads them there: fewer live registers); returns the
// centre.
__device__ __forceinline__ float4 warp_frame(const WarpBox& b, float keepA, float keepB, StreamRings& SR,
                                             int lane) {
    const float4 c = make_float4(0.5f * (b.lo[0] + b.hi[0]), 0.5f * (b.lo[1] + b.hi[1]),
                                 0.5f * (b.lo[2] + b.hi[2]), keepA);
    if (lane == 0) {
        SR.box[0] = c;
        SR.box[1] = make_float4(0.5f * (b.hi[0] - b.lo[0]), 0.5f * (b.hi[1] - b.lo[1]),
                                0.5f * (b.hi[2] - b.lo[2]), keepB);
    }
    __syncwarp();
    return c;
}

// Candidates g0 + lane (below re) go through the box test (against the centred box, with
// the reach of the candidate's species); survivors are appended to their species' stream
// at positions fill[S], fill[S] + 1, ... in candidate order.  cself receives the stream
// position of the lane's own particle (in the stream of its own species) when its group
// passes.
__device__ __forceinline__ void compact_streams(const float4* sm, int g0, int re, StreamRings& SR,
                                                int fill[2], int self, int& cself, int lane) {
    const int t = g0 + lane;
    bool keep = false;
    int sj = 0;
    float x = 0.f, y = 0.f, z = 0.f;
    if (t < re) {
        const float4 p = sm[t];
        const float4 c = SR.box[0], h = SR.box[1];
        x = p.x - c.x;
        y = p.y - c.y;
        z = p.z - c.z;
        const float ex = fmaxf(fabsf(x) - h.x, 0.f);
        const float ey = fmaxf(fabsf(y) - h.y, 0.f);
        const float ez = fmaxf(fabsf(z) - h.z, 0.f);
        sj = p.w != 0.f ? 1 : 0;
        keep = fmaf(ez, ez, fmaf(ey, ey, ex * ex)) < (sj ? h.w : c.w);
    }
    const unsigned bA = __ballot_sync(FULL, keep && sj == 0);
    const unsigned bB = __ballot_sync(FULL, keep && sj == 1);
    const unsigned lt = (1u << lane) - 1u;
    const int pos = sj ? fill[1] + __popc(bB & lt) : fill[0] + __popc(bA & lt);
    if (keep) {
        const int o = pos & (kSRing - 1);
        SR.x[sj][o] = x;
        SR.y[sj][o] = y;
        SR.z[sj][o] = z;
        SR.q[sj][o] = fmaf(z, z, fmaf(y, y, x * x));
        SR.idx[sj][o] = (uint16_t)t;
    }
    const int src = self - g0;
    const int sp = __shfl_sync(FULL, pos, src & 31);
    // (a group's lanes past the end of its row belong to other rows: with few particles a
    // cell, the lane's own may be among them)
    if (src >= 0 && src < 32 && self < re) cself = sp;
    fill[0] += __popc(bA);
    fill[1] += __popc(bB);
}

// After the last group: the rest of stream S's last word holds far records (q huge, so
// every test is positive) pointing at the sentinel.
__device__ __forceinline__ void stream_pad(StreamRings& SR, int S, int fill, int lane, int sentinel) {
    const int pe = (fill + 31) & ~31;
    if (fill + lane < pe) {
        const int o = (fill + lane) & (kSRing - 1);
        SR.x[S][o] = SR.y[S][o] = SR.z[S][o] = kFar;
        SR.q[S][o] = 3.0f * kFar * kFar;
        SR.idx[S][o] = (uint16_t)sentinel;
    }
}

// r^2 - R^2 of entry u of a stream word for a lane: m2 = -2 m', cst = |m'|^2 - R^2(s_i, S).
__device__ __forceinline__ float stream_d(const StreamWord& W, int u, float m2x, float m2y, float m2z,
                                          float cst) {
    return fmaf(W.z[u], m2z, fmaf(W.y[u], m2y, fmaf(W.x[u], m2x, W.q[u] + cst)));
}

// The signs of stream_d over a word (entry u in bit 31 - u: set where negative) and the
// smallest |stream_d|.  Two-wide FP32 (each half rounds like the scalar operation), four
// entries per 16-byte read of a component: 5.5 instructions an entry against 7.
__device__ __forceinline__ unsigned word_signs(const StreamWord& W, float m2x, float m2y, float m2z,
                                               float cst, float& near) {
    const float2 mx = make_float2(m2x, m2x), my = make_float2(m2y, m2y), mz = make_float2(m2z, m2z),
                 cc = make_float2(cst, cst);
    unsigned in = 0u;
#pragma unroll
    for (int u = 0; u < 32; u += 4) {
        const float4 x = *reinterpret_cast<const float4*>(W.x + u);
        const float4 y = *reinterpret_cast<const float4*>(W.y + u);
        const float4 z = *reinterpret_cast<const float4*>(W.z + u);
        const float4 q = *reinterpret_cast<const float4*>(W.q + u);
        const float2 d0 = __ffma2_rn(make_float2(z.x, z.y), mz, __ffma2_rn(make_float2(y.x, y.y), my,
                          __ffma2_rn(make_float2(x.x, x.y), mx, __fadd2_rn(make_float2(q.x, q.y), cc))));
        const float2 d1 = __ffma2_rn(make_float2(z.z, z.w), mz, __ffma2_rn(make_float2(y.z, y.w), my,
                          __ffma2_rn(make_float2(x.z, x.w), mx, __fadd2_rn(make_float2(q.z, q.w), cc))));
        in = __funnelshift_l(__float_as_uint(d0.x), in, 1);
        in = __funnelshift_l(__float_as_uint(d0.y), in, 1);
        in = __funnelshift_l(__float_as_uint(d1.x), in, 1);
        in = __funnelshift_l(__float_as_uint(d1.y), in, 1);
        near = fminf(near, fminf(fabsf(d0.x), fabsf(d0.y)));
        near = fminf(near, fminf(fabsf(d1.x), fabsf(d1.y)));
    }
    return in;
}

// Which force kernel runs: in cell mode the stencil kernel (MODE 1); in Verlet mode the
// list kernel (MODE 0), or the stencil kernel while the stored lists are cut at the
// capacity (exact forces until the host has grown the lists).
template <int MODE>
__device__ __forceinline__ bool force_selected(const DevSim& s) {
    if (s.nbr_mode != BBMD_NBR_VERLET) return MODE == 1;
    return (s.sc->list_short != 0) == (MODE == 1);
}

// MODE 0: Verlet list.  MODE 1: every particle of the 27-cell stencil (no stored list).
// BAND_INL: the band fix-up inline (else called out of line).  LIMIT: see StageOps.  False (on every thread of the
// CTA) if a staging wait gave up: the CTA must not stage again (staged_blocks).
template <int MODE, bool KE, bool FSHIFT, bool BAND_INL = kBandInline, bool LIMIT = false>
__device__ __forceinline__ bool force_body(const DevSim& s, int lb, int lg) {
    if (!force_selected<MODE>(s)) return true;  // CTA-uniform, before any barrier
    extern __shared__ float4 smem[];
    StageShared& ss = stage_shared();
    Region* const R = ss.R;
    uint64_t* const mbar = ss.mbar;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (threadIdx.x == 0) {
        ss.next_cell[0] = ss.next_cell[1] = 0;
        ss.ke_fix = 0ull;
    }
    int blk_it = 0;  // blocks of this CTA so far (the parity selects the counter)
    float hdt0 = 0.f, hdt1 = 0.f;
    if (KE) {
        hdt0 = s.sc->hdt[0];
        hdt1 = s.sc->hdt[1];
    }
    const float m0 = s.pt.mass[0], m1 = s.pt.mass[1];
    const float far = kFar;
    const unsigned sv = (unsigned)s.smax | ((unsigned)s.smax << 16);
    const uint4 sent = make_uint4(sv, sv, sv, sv);
    StreamRings* SRp = nullptr;  // candidate streams of the stencil mode
    if constexpr (MODE == 1) SRp = &warp_streams(w);
    const bool staged = for_each_block<LIMIT>(s, lb, lg, smem, s.smax + 1, R, mbar,
                                              [&](const BlockPos& bp, const Region& Rc, const float4* sm, int) {
        const int par = blk_it & 1;
        if (threadIdx.x == 0) ss.next_cell[par ^ 1] = 0;  // for the next block
        ++blk_it;
        // the block's work items: in list mode its chunks of one species (a lane's list
        // length depends on its species, and a warp runs to its longest list); in stencil
        // mode its cells (the stencil is the cell's)
        int nitems = kCells;
        if constexpr (MODE == 0) {
            own_chunks(s, bp, Rc, ss, [&](int t) { return sm[t].w == 0.f; });
            nitems = ss.nch;
        }
        for (int item = take_cell(ss, par, lane); item < nitems; item = take_cell(ss, par, lane)) {
            WarpCell wc;
            int i0 = 0, cnt = 32, self0 = 0;
            if constexpr (MODE == 1) {
                wc = warp_cell(s, bp, item);
                i0 = wc.valid ? Rc.start[wc.rq] : 0;
                cnt = wc.valid ? staged_count(Rc, wc.rq) : 0;
                self0 = Rc.off[wc.rq];
            }
            for (int ch = 0; ch * 32 < cnt; ++ch) {
                bool act;
                int64_t gi;
                int self;
                if constexpr (MODE == 0) {
                    chunk_lane(ss, item, lane, act, gi, self);
                    // the chunk a warp takes kBW items later: its first list rows and
                    // velocities go to L2 now, so that its prologue does not wait on DRAM
                    if (item + kBW < nitems) {
                        bool nact;
                        int64_t ngi;
                        int nself;
                        chunk_lane(ss, item + kBW, lane, nact, ngi, nself);
                        if (nact) {
                            const uint4* lq = reinterpret_cast<const uint4*>(s.list) + ngi;
                            prefetch_l2(lq);
                            prefetch_l2(lq + s.npad);
                            prefetch_l2(s.rows + ngi);
                            if (KE) {
                                prefetch_l2(s.v + ngi);
                                prefetch_l2(s.v + s.npad + ngi);
                                prefetch_l2(s.v + 2 * s.npad + ngi);
                            }
                        }
                    }
                } else {
                    const int li = ch * 32 + lane;
                    act = li < cnt;
                    gi = (int64_t)i0 + li;
                    self = self0 + li;
                }
                // issue the long-latency loads first: the first list rows, the velocity
                const uint4* lp = reinterpret_cast<const uint4*>(s.list) + gi;
                const int myrows = MODE == 0 && act ? (int)s.rows[gi] : 0;  // rows of its list
                uint4 e0 = sent, e1 = sent, e2 = sent;
                if (MODE == 0) {
                    if (myrows > 0) e0 = __ldcs(lp);
                    if (myrows > 1) e1 = __ldcs(lp + s.npad);
                    if (kListAhead > 2 && myrows > 2) e2 = __ldcs(lp + 2 * s.npad);
                }
                // (the stencil loop of MODE 1 needs every register: its velocities are read
                // after it)
                long long v0 = 0, v1 = 0, v2 = 0;
                if (KE && act && MODE == 0) {
                    v0 = s.v[gi];
                    v1 = s.v[s.npad + gi];
                    v2 = s.v[2 * s.npad + gi];
                }
                int nkb = myrows;  // the warp runs to its longest list
                if (MODE == 0)
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) nkb = max(nkb, __shfl_xor_sync(FULL, nkb, o));
                float4 me = act ? sm[self] : make_float4(-far, -far, -far, 0.f);
                const int si = me.w != 0.f ? 1 : 0;
                LaneTab T;
                if constexpr (MODE == 0) load_tab(s, si, T);
                Acc a = {0.f, 0.f, 0.f};
                if (MODE == 0) {
                    for (int kb = 0; kb < nkb; ++kb) {
                        const uint4 e = e0;
                        e0 = e1;
                        if (kListAhead > 2) {
                            e1 = e2;
                            e2 = kb + 3 < myrows ? __ldcs(lp + (int64_t)(kb + 3) * s.npad) : sent;
                        } else {
                            e1 = kb + 2 < myrows ? __ldcs(lp + (int64_t)(kb + 2) * s.npad) : sent;
                        }
                        if (kListPrefetch > 0 && kb + kListPrefetch < myrows)
                            prefetch_l2(lp + (int64_t)(kb + kListPrefetch) * s.npad);
                        float near = far;
                        pair_fast<FSHIFT>(T, me, sm[lo16(e.x)], a, near);
                        pair_fast<FSHIFT>(T, me, sm[hi16(e.x)], a, near);
                        pair_fast<FSHIFT>(T, me, sm[lo16(e.y)], a, near);
                        pair_fast<FSHIFT>(T, me, sm[hi16(e.y)], a, near);
                        pair_fast<FSHIFT>(T, me, sm[lo16(e.z)], a, near);
                        pair_fast<FSHIFT>(T, me, sm[hi16(e.z)], a, near);
                        pair_fast<FSHIFT>(T, me, sm[lo16(e.w)], a, near);
                        pair_fast<FSHIFT>(T, me, sm[hi16(e.w)], a, near);
                        const bool band = near < T.hw;
                        if (__any_sync(FULL, band) && band) {
                            const unsigned ws[4] = {e.x, e.y, e.z, e.w};
                            for (int q = 0; q < 8; ++q) {
                                int t = (q & 1) ? hi16(ws[q >> 1]) : lo16(ws[q >> 1]);
                                if constexpr (BAND_INL)
                                    pair_band<FSHIFT>(s, Rc, T, me, sm[t], t, gi, true, a);
                                else
                                    pair_band_call<FSHIFT>(s, Rc, T, me, sm[t], t, gi, true, a);
                            }
                        }
                    }
                } else {
                    // the stencil on the fly: the candidates within reach of the warp's box
                    // go into the two species streams, each stream word is filtered against
                    // the cutoff into a bitmask (as the list build does against rc + skin),
                    // band candidates are decided by the exact rule, then the forces of the
                    // set bits are added (the species of j is that of the stream)
                    StreamRings& SR = *SRp;
                    const float4 fc = warp_frame(warp_box(me, act), keep_reach(s.pt.rc2hi, 0),
                                                 keep_reach(s.pt.rc2hi, 1), SR, lane);
                    const float mx = act ? me.x - fc.x : 0.f, my = act ? me.y - fc.y : 0.f,
                                mz = act ? me.z - fc.z : 0.f;
                    const float m2x = -2.f * mx, m2y = -2.f * my, m2z = -2.f * mz;
                    const float mm = act ? fmaf(mz, mz, fmaf(my, my, mx * mx)) : far;
                    int fill[2] = {0, 0}, done[2] = {0, 0}, cself = -1;
                    // bitmask of the entries of stream S's word at cq inside the cutoff
                    auto filter_word = [&](int S, int cq) -> unsigned {
                        const StreamWord W = stream_word(SR, S, cq);
                        const float cS = mm - s.pt.rc2lo[si * 2 + S];
                        float near = far;
                        unsigned inw = word_signs(W, m2x, m2y, m2z, cS, near);
                        const int nv = fill[S] - cq;
                        unsigned valid = nv >= 32 ? 0xffffffffu : ~(0xffffffffu >> nv);
                        if (S == si && cself >= cq && cself < cq + 32)
                            valid &= ~(0x80000000u >> (cself - cq));
                        if (!act) valid = 0u;
                        inw &= valid;
                        const float bS = s.pt.rc2hi[si * 2 + S] - s.pt.rc2lo[si * 2 + S];
                        const bool chk = near < bS && valid != 0u;
                        if (__any_sync(FULL, chk) && chk) {
                            unsigned bw = valid;
                            while (bw) {
                                const int u = __clz(bw);
                                bw &= 0x7fffffffu >> u;
                                if (!(fabsf(stream_d(W, u, m2x, m2y, m2z, cS)) < bS)) continue;
                                const unsigned bit = 0x80000000u >> u;
                                inw &= ~bit;
                                if (!min_image_copy(s, fmaf(m2x, 0.5f, W.x[u]), fmaf(m2y, 0.5f, W.y[u]),
                                                    fmaf(m2z, 0.5f, W.z[u])))
                                    continue;
                                const int t = (int)SR.idx[S][(cq + u) & (kSRing - 1)];
                                const int64_t gj = staged_global(Rc, t);
                                if (r2_exact(s, gi, gj) < s.pt.rc2[si * 2 + S]) inw |= bit;
                            }
                        }
                        return inw;
                    };
                    // the forces of the set bits of stream S's word at cq
                    auto force_word = [&](int S, int cq) {
                        unsigned inw = filter_word(S, cq);
                        const StreamWord W = stream_word(SR, S, cq);
                        // the constants of the species pair (s_i, S)
                        const int k = si * 2 + S;
                        const float sig2 = s.pt.sig2[k], e48 = s.pt.eps48[k];
                        const float fcut = FSHIFT ? s.pt.fcut[k] : 0.f;
                        const float cpot = s.pt.potential == BBMD_POT_LJ ? 0.5f : 0.0f;
                        // Two entries an iteration, for the loop runs to the lane with the most
                        // entries: two-wide FP32, each half rounding like the scalar operation,
                        // the forces added one after the other.  2.05 M particles, one entry ->
                        // two: 4x4x2 1048 -> 1001 us, 4x4x4 1176 -> 1093, 4x4x8 1195 -> 1087
                        while (inw) {
                            const int u = __clz(inw);
                            inw &= 0x7fffffffu >> u;
                            const bool two = inw != 0u;
                            const int w = two ? __clz(inw) : u;
                            inw &= 0x7fffffffu >> w;
                            // p' - m' (0.5 m2 = -m' exactly)
                            const float2 h = make_float2(0.5f, 0.5f);
                            const float2 dx = __ffma2_rn(make_float2(m2x, m2x), h, make_float2(W.x[u], W.x[w]));
                            const float2 dy = __ffma2_rn(make_float2(m2y, m2y), h, make_float2(W.y[u], W.y[w]));
                            const float2 dz = __ffma2_rn(make_float2(m2z, m2z), h, make_float2(W.z[u], W.z[w]));
                            const float2 r2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __fmul2_rn(dz, dz)));
                            const float2 f = pair_f2<FSHIFT>(sig2, e48, cpot, fcut, r2);
                            a.fx = fmaf(f.x, dx.x, a.fx);
                            a.fy = fmaf(f.x, dy.x, a.fy);
                            a.fz = fmaf(f.x, dz.x, a.fz);
                            if (two) {
                                a.fx = fmaf(f.y, dx.y, a.fx);
                                a.fy = fmaf(f.y, dy.y, a.fy);
                                a.fz = fmaf(f.y, dz.y, a.fz);
                            }
                        }
                    };
                    auto flush_full = [&](int S) {
                        if (fill[S] - done[S] >= 32) {
                            force_word(S, done[S]);
                            done[S] += 32;
                            __syncwarp();
                        }
                    };
                    auto flush_last = [&](int S) {
                        if (fill[S] > done[S]) {
                            stream_pad(SR, S, fill[S], lane, s.smax);
                            __syncwarp();
                            force_word(S, done[S]);
                            done[S] += 32;
                            __syncwarp();
                        }
                    };
                    StencilScan sc = {-1, 0, 0};
                    bool more = scan_next(Rc, wc, sc);
                    while (more) {
                        compact_streams(sm, sc.g0, sc.re, SR, fill, self, cself, lane);
                        sc.g0 += 32;
                        more = scan_next(Rc, wc, sc);
                        __syncwarp();
                        flush_full(0);
                        flush_full(1);
                    }
                    flush_last(0);
                    flush_last(1);
                }
                float fx = -a.fx, fy = -a.fy, fz = -a.fz;
                if (act) {
                    if (!(isfinite(fx) && isfinite(fy) && isfinite(fz))) set_status(s, ST_NONFINITE);
                    s.F[gi] = make_float4(fx, fy, fz, 0.f);
                }
                if (KE) {
                    float k = 0.f;
                    if (act) {
                        if (MODE == 1) {
                            v0 = s.v[gi];
                            v1 = s.v[s.npad + gi];
                            v2 = s.v[2 * s.npad + gi];
                        }
                        const float h = si ? hdt1 : hdt0;
                        const float m = si ? m1 : m0;
                        const float vx = fmaf(h, fx, i64_to_f32_fast(v0) * pow2f(-kVelExp));
                        const float vy = fmaf(h, fy, i64_to_f32_fast(v1) * pow2f(-kVelExp));
                        const float vz = fmaf(h, fz, i64_to_f32_fast(v2) * pow2f(-kVelExp));
                        k = 0.5f * m * fmaf(vx, vx, fmaf(vy, vy, vz * vz));
                    }
                    const unsigned long long kc = chunk_energy(k);
                    if (lane == 0) atomicAdd(&ss.ke_fix, kc);
                }
            }
        }
    });
    if (!staged) return false;
    if (KE) {
        // every warp has passed the last block's closing barrier
        const double acc_ke = threadIdx.x == 0 ? __ull2double_rn(ss.ke_fix) * 0x1p-32 : 0.0;
        block_partials(s, lb, &acc_ke, 0, 1);
    }
    return true;
}

// ------------------------------------------------------------------ list build ----

// Each lane tests the compacted candidates of its 27-cell stencil, 32 at a time, with
// broadcast shared-memory reads: the sign of r^2 - R2lo(species of j) is shifted into a
// 32-bit word (candidate u lands in bit 31 - u) and the smallest |r^2 - R2lo| of the word
// is kept.  Only a word whose minimum falls inside the band goes through the exact rule,
// candidate by candidate.  The set bits of each word are then appended to the lane's list.
//
// The append takes 45 % of the build as a loop over each lane's own bits (two entries and one
// 4-byte store an iteration, 22 of 32 lanes active, 340 instructions a word).  With BUFFER
// every lane looks at every candidate of the word (one predicated store into its own buffer
// of 16 entries in shared memory, no divergent loop), and rows of 8 leave as they fill with
// one 16-byte store.  Microseconds a build at 2.05 M particles, loop -> buffer (before either,
// with one FP32 operation per entry and scalar reads of the streams): 4 x 4 x 2 at skin 0.4
// (1427) 1370 -> 1282; at skin 0.3 2 x 2 x 2 (1140) 1077 -> 1030, 2 x 2 x 1 (1230) 1174 -> 1108.
// 2 x 2 x 4 keeps the loop (1095 -> 1049): the buffers would leave room for two CTAs per SM
// instead of three (1140).  Looks after every 4 candidates (smaller buffers) or only when some
// buffer is full (larger ones) measured slower.

// Append the low half of e if bits & mask and the high half if bits & (mask >> 1) at the
// shared-memory address top: predicated stores, whatever the lanes' bits.
__device__ __forceinline__ void push_entries(unsigned& top, unsigned e, unsigned bits, unsigned mask) {
    asm volatile(
        "{\n .reg .pred p;\n .reg .b32 t;\n .reg .b16 lo, hi;\n"
        " mov.b32 {lo, hi}, %1;\n"
        " and.b32 t, %2, %3;\n setp.ne.u32 p, t, 0;\n"
        " @p st.shared.u16 [%0], lo;\n @p add.u32 %0, %0, 2;\n"
        " and.b32 t, %2, %4;\n setp.ne.u32 p, t, 0;\n"
        " @p st.shared.u16 [%0], hi;\n @p add.u32 %0, %0, 2;\n}"
        : "+r"(top)
        : "r"(e), "r"(bits), "r"(mask), "r"(mask >> 1)
        : "memory");
}

// The lane's entry buffer: 16 entries, 16-byte aligned.  One KB per warp, in the part of the
// description of the region being computed, buffer b's, that is free once its block is staged
// (as many warps as fit; with two staging buffers the other one describes the next block
// meanwhile), and beside it for the others.
__device__ __forceinline__ uint16_t* entry_buffer(StageShared& ss, int b, int w, int lane) {
    constexpr int kFree = (int)(sizeof(Region) - offsetof(Region, hi)) / 1024;  // warps
    constexpr int kMore = kBW > kFree ? kBW - kFree : 1;
    __shared__ __align__(16) uint16_t more[kMore][32][16];
    if (w < kFree) return reinterpret_cast<uint16_t*>(&ss.R[b].hi[0][0]) + (w * 32 + lane) * 16;
    return more[w - kFree][lane];
}

// LIMIT and false as force_body.
template <bool BUFFER, bool LIMIT = false>
__device__ __forceinline__ bool list_build_body(const DevSim& s, int lb, int lg) {
    if (!s.sc->rebuild) return true;
    extern __shared__ float4 smem[];
    StageShared& ss = stage_shared();
    Region* const R = ss.R;
    uint64_t* const mbar = ss.mbar;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int lcap = s.lcap8 * 8;
    const int lcap2 = lcap >> 1;  // pair slots per particle
    StreamRings& SR = warp_streams(w);
    if (threadIdx.x == 0) ss.next_cell[0] = ss.next_cell[1] = 0;
    int blk_it = 0;  // blocks of this CTA so far (the parity selects the cell counter)
    const float far = kFar;
    uint16_t* buf = nullptr;
    if constexpr (BUFFER) buf = entry_buffer(ss, 0, w, lane);
    return for_each_block<LIMIT>(s, lb, lg, smem, s.smax + 1, R, mbar,
                                 [&](const BlockPos& bp, const Region& Rc, const float4* sm, int b) {
        if constexpr (BUFFER && kStageBuffers > 1) buf = entry_buffer(ss, b, w, lane);
        const int par = blk_it & 1;
        if (threadIdx.x == 0) ss.next_cell[par ^ 1] = 0;  // for the next block
        ++blk_it;
        // (a cell's first 32 particles are an item, the others another: a warp that had both
        // would be the last of its block)
        for (int item = take_cell(ss, par, lane); item < 2 * kCells; item = take_cell(ss, par, lane)) {
            const int first = item < kCells ? 1 : 0;
            const WarpCell wc = warp_cell(s, bp, first ? item : item - kCells);
            const int i0 = wc.valid ? Rc.start[wc.rq] : 0;
            const int all = wc.valid ? staged_count(Rc, wc.rq) : 0;
            const int cnt = first ? min(all, 32) : all;
            const int self0 = Rc.off[wc.rq];
            for (int ch = 1 - first; ch * 32 < cnt; ++ch) {
                const int li = ch * 32 + lane;
                const bool act = li < cnt;
                const int64_t gi = (int64_t)i0 + li;
                const int self = self0 + li;
                float4 me = act ? sm[self] : make_float4(-far, -far, -far, 0.f);
                const int si = me.w != 0.f ? 1 : 0;
                // the row being filled (entries beyond the capacity are counted, not stored); with
                // BUFFER its number and the shared-memory address of the lane's next entry, else
                // the next pair slot, the entries so far and a pending odd one
                uint4* rowp = reinterpret_cast<uint4*>(s.list) + gi;
                const unsigned top0 = BUFFER ? smem_u32(buf) : 0u;
                unsigned top = top0, pend = 0u;
                int row = 0, wp = 0, len = 0;
                auto put_pair = [&](unsigned v) {
                    if (wp < lcap2) reinterpret_cast<uint32_t*>(rowp)[wp & 3] = v;
                    ++wp;
                    if ((wp & 3) == 0) rowp += s.npad;
                };
                const float4 fc = warp_frame(warp_box(me, act), keep_reach(s.pt.R2hi, 0),
                                             keep_reach(s.pt.R2hi, 1), SR, lane);
                // the lane relative to the box centre, and its constants per stream
                const float mx = act ? me.x - fc.x : 0.f, my = act ? me.y - fc.y : 0.f,
                            mz = act ? me.z - fc.z : 0.f;
                const float m2x = -2.f * mx, m2y = -2.f * my, m2z = -2.f * mz;
                const float mm = act ? fmaf(mz, mz, fmaf(my, my, mx * mx)) : far;
                int fill[2] = {0, 0}, done[2] = {0, 0}, cself = -1;
                // bitmask of the entries of stream S's word at cq (a multiple of 32) that
                // enter this particle's list (entry u in bit 31 - u)
                auto test_word = [&](int S, int cq) -> unsigned {
                    const StreamWord W = stream_word(SR, S, cq);
                    const float cS = mm - s.pt.R2lo[si * 2 + S];
                    float near = far;
                    unsigned inw = word_signs(W, m2x, m2y, m2z, cS, near);
                    const int nv = fill[S] - cq;
                    unsigned valid = nv >= 32 ? 0xffffffffu : ~(0xffffffffu >> nv);
                    if (S == si && cself >= cq && cself < cq + 32)
                        valid &= ~(0x80000000u >> (cself - cq));
                    if (!act) valid = 0u;
                    inw &= valid;
                    const float bS = s.pt.R2hi[si * 2 + S] - s.pt.R2lo[si * 2 + S];
                    const bool chk = near < bS && valid != 0u;
                    if (__any_sync(FULL, chk) && chk) {
                        // the same FP32 value decides which entries are in the band; those
                        // are decided by the exact rule
                        unsigned bw = valid;
                        while (bw) {
                            const int u = __clz(bw);
                            bw &= 0x7fffffffu >> u;
                            if (!(fabsf(stream_d(W, u, m2x, m2y, m2z, cS)) < bS)) continue;
                            const unsigned bit = 0x80000000u >> u;
                            inw &= ~bit;
                            // (p' - m' is the separation up to FP32 rounding: enough to tell
                            // the minimum-image copy from one a box length away)
                            if (!min_image_copy(s, fmaf(m2x, 0.5f, W.x[u]), fmaf(m2y, 0.5f, W.y[u]),
                                                fmaf(m2z, 0.5f, W.z[u])))
                                continue;
                            const int t = (int)SR.idx[S][(cq + u) & (kSRing - 1)];
                            const int64_t gj = staged_global(Rc, t);
                            if (r2_exact(s, gi, gj) < s.pt.R2[si * 2 + S]) inw |= bit;
                        }
                    }
                    return inw;
                };
                // the set bits of stream S's word at cq as list entries, in stream order.  BUFFER:
                // eight candidates at a time, each lane adds its own to its buffer, and lanes whose
                // buffer holds a row of eight write it with one 16-byte store.  Else: each lane
                // goes through its own bits, two at a time, one 4-byte store for both; an odd
                // last entry waits for the next word's first
                auto append_word = [&](int S, int cq, unsigned bits) {
                    if constexpr (BUFFER) {
                        const uint4* const iw = reinterpret_cast<const uint4*>(SR.idx[S] + (cq & (kSRing - 1)));
#pragma unroll
                        for (int o = 0; o < 4; ++o) {
                            const uint4 e = iw[o];
                            const unsigned es[4] = {e.x, e.y, e.z, e.w};
#pragma unroll
                            for (int u = 0; u < 4; ++u)
                                push_entries(top, es[u], bits, 0x80000000u >> (o * 8 + 2 * u));
                            const bool full = top - top0 >= 16u;
                            if (__any_sync(FULL, full) && full) {
                                uint4* const b4 = reinterpret_cast<uint4*>(buf);
                                if (row < s.lcap8) *rowp = b4[0];
                                b4[0] = b4[1];
                                top -= 16u;
                                ++row;
                                rowp += s.npad;
                            }
                        }
                    } else {
                        // (the word's entries are contiguous: it starts at a multiple of 32 in a ring
                        // of 64)
                        const uint16_t* const rw = SR.idx[S] + (cq & (kSRing - 1));
                        if ((len & 1) && bits) {
                            const int u = __clz(bits);
                            bits &= 0x7fffffffu >> u;
                            put_pair(pend | ((unsigned)rw[u] << 16));
                            ++len;
                        }
                        while (bits) {
                            const int u1 = __clz(bits);
                            bits &= 0x7fffffffu >> u1;
                            const unsigned t1 = rw[u1];
                            if (!bits) {
                                pend = t1;
                                ++len;
                                break;
                            }
                            const int u2 = __clz(bits);
                            bits &= 0x7fffffffu >> u2;
                            put_pair(t1 | ((unsigned)rw[u2] << 16));
                            len += 2;
                        }
                    }
                };
                // a stream's word is tested and appended as soon as it is full (fewer than
                // 32 entries wait in each ring before a group adds at most 32)
                auto flush_full = [&](int S) {
                    if (fill[S] - done[S] >= 32) {
                        append_word(S, done[S], test_word(S, done[S]));
                        done[S] += 32;
                        __syncwarp();
                    }
                };
                StencilScan sc = {-1, 0, 0};
                bool more = scan_next(Rc, wc, sc);
                while (more) {
                    compact_streams(sm, sc.g0, sc.re, SR, fill, self, cself, lane);
                    sc.g0 += 32;
                    more = scan_next(Rc, wc, sc);
                    __syncwarp();
                    flush_full(0);
                    flush_full(1);
                }
                // the partial last word of each stream
                auto flush_last = [&](int S) {
                    if (fill[S] > done[S]) {
                        stream_pad(SR, S, fill[S], lane, s.smax);
                        __syncwarp();
                        append_word(S, done[S], test_word(S, done[S]));
                        done[S] += 32;
                        __syncwarp();
                    }
                };
                flush_last(0);
                flush_last(1);
                const int left = (int)(top - top0) >> 1;
                if constexpr (BUFFER) len = row * 8 + left;
                if (len > lcap) {
                    // the list is cut: flagged for the host (which grows the capacity at its
                    // next synchronising call) and, until then, the forces come from the
                    // cell stencil
                    set_status(s, ST_LIST_OVERFLOW);
                    s.sc->list_short = 1;
                    atomicMax(&s.sc->max_len, len);
                }
                if (act) {
                    // the rest of the last row holds the sentinel; the particle's row count tells
                    // the force kernels where its list ends
                    if constexpr (BUFFER) {
                        if (left > 0) {
                            for (int k = left; k < 8; ++k) buf[k] = (uint16_t)s.smax;
                            if (row < s.lcap8) *rowp = *reinterpret_cast<const uint4*>(buf);
                            ++row;
                        }
                    } else {
                        if (len & 1) put_pair(pend | ((unsigned)s.smax << 16));
                        while (wp & 3) put_pair((unsigned)s.smax | ((unsigned)s.smax << 16));
                        row = wp >> 2;
                    }
                    s.rows[gi] = (uint16_t)min(row, s.lcap8);
                }
            }
        }
    });
}

// ------------------------------------------------------- one-launch step ----
// A small system's step is a chain of kernels of a few microseconds each: 16 launches, most
// of them gated off, took 54 us for 4000 particles.  One cooperative launch instead runs
// many whole steps: every phase is the body that the kernels of its own run (with their CTA
// index and count where a sum depends on it, so the states are the same bit for bit), and
// the phases are kept apart by a grid-wide barrier (about 1.3 us) only where one is needed:
// two in a step in which nothing came near the rebuild trigger, two more for the trigger,
// six or seven more for a rebuild.  Where it is used and what it measured: grid_step_grid
// (bbmd_api.cu).  At 4000 particles (2 x 2 x 1 blocks, one per SM, four warps) a step's 41 us
// were forces 14 (two rounds of chunks), barriers 6, finalize 6, integrate 2, and 0.2 rebuilds
// of 70 (its list build 45, two rounds for a cell of more than 32).
#include "sort_bodies.cuh"
#include "step_bodies.cuh"
#include "grid_bodies.cuh"

#ifndef BBMD_GRID_MIN_BLOCKS
#define BBMD_GRID_MIN_BLOCKS (BBMD_BLOCK_Z == 1 && !BBMD_WIDE ? 4 : 2)
#endif

// The rebuild after its flag is up and the cell counts are zero: sort chain and list build.
// on_last runs once at the end.
template <class OnLast>
__device__ __forceinline__ bool grid_rebuild(const DevSim& s, unsigned& gen, OnLast on_last) {
    if (!grid_sort(s, gen)) return false;
    if (s.nbr_mode == BBMD_NBR_VERLET) {
        if (!grid_barrier(s, gen)) return false;
        for (int b = (int)blockIdx.x; b < s.grid_list; b += (int)gridDim.x)
            if (!list_build_body<true, true>(s, b, s.grid_list)) return grid_abort(s);
    }
    return grid_barrier(s, gen, true, on_last);
}

// Forces with the CTA index and count of the force kernel's own launch.  False after a staging
// wait that gave up.
template <bool KE, bool FSHIFT>
__device__ __forceinline__ bool grid_force(const DevSim& s) {
    for (int b = (int)blockIdx.x; b < s.grid_cell; b += (int)gridDim.x)
        if (!force_body<0, KE, FSHIFT, false, true>(s, b, s.grid_cell) ||
            !force_body<1, KE, FSHIFT, false, true>(s, b, s.grid_cell))
            return grid_abort(s);
    return true;
}

template <bool KE, bool FSHIFT>
__global__ void __launch_bounds__(kBW * 32, BBMD_GRID_MIN_BLOCKS) k_step_grid(DevSim s, int nsteps) {
    if (given_up(s)) return;
    const int lb = (int)blockIdx.x, lg = (int)gridDim.x;
    unsigned gen = 0;
    for (int step = 0; step < nsteps; ++step) {
        integrate_body<false>(s, lb, lg);
        if (!grid_barrier(s, gen)) return;
        bool due;
        if (!grid_trigger(s, gen, due)) return;
        if (due && !grid_rebuild(s, gen, [] {})) return;
        if (!grid_force<KE, FSHIFT>(s)) return;
        if (!grid_barrier(s, gen, true, [&] { finalize_body(s, KE ? 1 : 0); })) return;
    }
}

// Steepest descent: x += h F, h = min(hmax, dmax / max |F|), nsteps times, then the forces.
template <bool FSHIFT>
__global__ void __launch_bounds__(kBW * 32, BBMD_GRID_MIN_BLOCKS)
    k_relax_grid(DevSim s, int nsteps, double hmax, double dmax) {
    if (given_up(s)) return;
    const int lb = (int)blockIdx.x, lg = (int)gridDim.x;
    unsigned gen = 0;
    for (int step = 0; step < nsteps; ++step) {
        // (squares of FP32 forces are not negative: their bits order like the values)
        uint32_t* const slot = &s.gsync[(kSyncMax0 + (step & 1)) * kSyncStride];
        if (!grid_force<false, FSHIFT>(s)) return;
        if (!grid_barrier(s, gen)) return;
        const float m = maxf_body(s, lb, lg);
        if ((threadIdx.x & 31) == 0) atomicMax(slot, __float_as_uint(m));
        zero_counts(s, lb, lg);
        if (!grid_barrier(s, gen)) return;
        const double fm = sqrt((double)__uint_as_float(*(volatile uint32_t*)slot));
        if (lb == 0 && threadIdx.x == 0) s.gsync[(kSyncMax0 + ((step + 1) & 1)) * kSyncStride] = 0u;
        sd_move_body<false>(s, lb, lg, fm, hmax, dmax);
        if (!grid_barrier(s, gen)) return;
        if (*(volatile int*)&s.sc->rebuild)
            if (!grid_rebuild(s, gen, [&] {
                    if (threadIdx.x == 0) {
                        s.sc->n_rebuilds += 1;
                        s.sc->rebuild = 0;
                    }
                }))
                return;
    }
    grid_force<false, FSHIFT>(s);
}

// ------------------------------------------------------- persistent batch step ----
// One cooperative launch advances every replica of a batch by many steps.  The step of
// each replica is a chain of phases (integrate, the two trigger passes, the six sort
// passes, the list build, forces, finalize); each phase of each replica is cut into work
// items with the same (CTA index, CTA count) as the kernels launched for one system, so a
// replica advances bit for bit as it would alone.  The items of all replicas are handed
// out from one queue, step after step and phase-major within a step: a CTA takes the next
// item, waits until the replica's previous non-empty phase is complete (for the first
// phase of a step: the finalize of the replica's previous step) by a per-replica,
// per-phase count of finished items (bounded), runs the item and counts it finished.
// Replicas never wait on each other, so the phases and steps of different replicas
// overlap; an item waits only on items handed out before it, and every CTA is resident,
// so the queue always advances.
#if BBMD_BLOCK_Z == BBMD_PERSIST_Z
// Raise the abort flag and ST_TIMEOUT on every replica (one thread).
__device__ __forceinline__ void persistent_abort(const PersistentStep& a) {
    if (atomicExch(a.abort, 1) == 0)
        for (int r = 0; r < a.nrep; ++r) atomicOr(&a.sims[r].sc->status, ST_TIMEOUT);
}

// False (on every thread) if a staging wait gave up.
template <bool KE, bool FSHIFT>
__device__ __forceinline__ bool run_phase(int phase, const DevSim& s, int lb, int lg) {
    switch (phase) {
        case kPhIntegrate: integrate_body<false>(s, lb, lg); break;
        case kPhCelltop: celltop_body(s, lb, lg); break;
        case kPhCheck: check_body(s, lb, lg); break;
        case kPhZero: zero_body(s, lb, lg); break;
        case kPhBin: bin_body(s, lb, lg); break;
        case kPhScan: scan_cta_body(s, lb, lg); break;
        case kPhScatter: scatter_body(s, lb, lg); break;
        case kPhSortGather: sortgather_body(s, lb, lg); break;
        case kPhCopyback: copyback_body(s, lb, lg); break;
        case kPhList: return list_build_body<true, true>(s, lb, lg);
        case kPhForce:
            // the list body, or for a replica whose lists are cut (and in cell mode) the
            // stencil body: each returns at once when not selected
            return force_body<0, KE, FSHIFT, false, true>(s, lb, lg) && force_body<1, KE, FSHIFT, false, true>(s, lb, lg);
        default: finalize_body(s, KE ? 1 : 0); break;
    }
    return true;
}

template <bool KE, bool FSHIFT>
__global__ void __launch_bounds__(kBW * 32, 2) k_step_persistent(PersistentStep a) {
    __shared__ DevSim sh;
    __shared__ int4 desc;  // phase, replica, lb, lg of the item (phase -1: queue empty)
    __shared__ int run;    // 0: the item's replica does not rebuild (gated phase)
    for (;;) {
        if (threadIdx.x == 0) {
            int4 d = make_int4(-1, 0, 0, 0);
            int go = 0;
            if (*(volatile int*)a.abort == 0) {
                const long long k = (long long)atomicAdd(a.head, 1u);
                if (k < (long long)a.nitems * a.nsteps) {
                    const int step = (int)(k / a.nitems);
                    d = a.items[k - (long long)step * a.nitems];
                    int dep = a.dep[d.y * kPhases + d.x], dstep = step;
                    if (dep < 0 && step > 0) {
                        dep = kPhFinalize;  // the replica's previous step
                        dstep = step - 1;
                    }
                    if (dep >= 0) {
                        const int need = a.need[d.y * kPhases + dep] * (dstep + 1);
                        const int* cnt = &a.done[d.y * kPhases + dep];
                        const unsigned long long t0 = globaltimer_ns();
                        while (*(volatile const int*)cnt < need) {
                            if (*(volatile int*)a.abort) {
                                d.x = -1;
                                break;
                            }
                            if (globaltimer_ns() - t0 > a.wait_ns) {
                                persistent_abort(a);
                                d.x = -1;
                                break;
                            }
                        }
                        __threadfence();
                    }
                    go = d.x >= 0;
                    if (go && d.x >= kPhZero && d.x <= kPhList)
                        go = *(volatile int*)&a.sims[d.y].sc->rebuild != 0;
                }
            }
            desc = d;
            run = go;
        }
        __syncthreads();
        const int4 d = desc;
        if (d.x < 0) return;
        // data of earlier phases, written by other CTAs, is read by bulk copies (the async
        // proxy) as well as by ordinary loads
        asm volatile("fence.proxy.async.global;" ::: "memory");
        if (run) {
            const int4* src4 = reinterpret_cast<const int4*>(a.sims + d.y);
            int4* dst4 = reinterpret_cast<int4*>(&sh);
            for (int k = threadIdx.x; k < (int)(sizeof(DevSim) / 16); k += blockDim.x) dst4[k] = src4[k];
            __syncthreads();
            if (!run_phase<KE, FSHIFT>(d.x, sh, d.z, d.w)) {
                if (threadIdx.x == 0) persistent_abort(a);
                return;
            }
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            __threadfence();
            atomicAdd(&a.done[d.y * kPhases + d.x], 1);
        }
    }
}
#endif  // BBMD_BLOCK_Z == BBMD_PERSIST_Z

// ------------------------------------------------------------------ FP64 form ----
// The same block region staged as exact integer positions in the block's periodic image
// (frame point + seam image + the particle's minimum-image offset from the frame, which
// stays right after the particle itself has crossed the boundary since the last build);
// distances are the exact integer differences rounded once to double (the rule the list
// decisions use), pair arithmetic and accumulation in FP64.
//
// Bound: the FP64 pipe (2 lanes a clock per SM, 16 clocks for a warp instruction whatever
// the number of active lanes).  So the kernel keeps everything but the arithmetic of
// interacting pairs off that pipe, and runs it with full warps:
//   - a candidate is classified in FP32 from the upper words of its integer position
//     (resolution 2^(32-k)): beyond the cutoff, interacting, or too close to the cutoff to
//     tell, which the exact rule then decides;
//   - each lane queues its interacting candidates (shared memory) and the warp drains the
//     queues together, so a slot of the loop computes a pair on nearly every lane, instead
//     of once per candidate that any of the 32 lanes interacts with;
//   - r^2 stays in integer units (the scale is folded into the constants), 1/r^2 and 1/r come
//     from the hardware's approximation and one third-order step, and the virial comes from the
//     energies and the sum of their attractions: 17 operations a pair for forces, 14 for the
//     sums (22 and 20 with the force shift, which needs 1/r);
//   - sums over the system (energy, virial) take each pair from one side only.
// Measured against the form that ran the FP64 arithmetic for every candidate some lane of
// the warp interacts with: energy and virial sums at 16.4 M particles (lists, skin 0.4)
// 132 -> 24 ms, at 4 M in cell mode 121 -> 8.6 ms; forces of the FP64 form at 108 000
// 0.868 -> 0.347 ms.  (At 0.63e12 lanes a second the pairs' operations take 11, 2.7 and 0.19 ms.
// Every shape measures the same at 2 M; converting the integers with two additions instead of
// a conversion instruction was 15 % slower.)

// Staged record t: hi[t] = upper words of x, y, z and (global index << 1 | species), lo[t] =
// lower words.
struct Stage64 {
    int4* hi;
    uint4* lo;
};

__device__ __forceinline__ Stage64 stage64(const DevSim& s, float4* smem) {
    Stage64 g;
    g.hi = reinterpret_cast<int4*>(smem);
    g.lo = reinterpret_cast<uint4*>(smem) + (s.smax + 1);
    return g;
}

__device__ void stage_block64(const DevSim& s, const BlockPos& b, Region& R, const Stage64& g) {
    region_info(s, b, R);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int q = w; q < kRegion; q += kBW) {
        const int o0 = R.off[q], cq = R.off[q + 1] - o0;
        const long long fx = R.fr[q][0], fy = R.fr[q][1], fz = R.fr[q][2];
        for (int t = lane; t < cq; t += 32) {
            const int64_t j = R.start[q] + t;
            const long long x = fx + min_image((long long)s.x[j] - fx, s.Lfix[0]);
            const long long y = fy + min_image((long long)s.x[s.npad + j] - fy, s.Lfix[1]);
            const long long z = fz + min_image((long long)s.x[2 * s.npad + j] - fz, s.Lfix[2]);
            g.hi[o0 + t] = make_int4((int)(x >> 32), (int)(y >> 32), (int)(z >> 32),
                                     (int)(((unsigned)j << 1) | s.sp[j]));
            g.lo[o0 + t] = make_uint4((unsigned)x, (unsigned)y, (unsigned)z, 0u);
        }
    }
    if (threadIdx.x == 0) {
        // staged positions lie in (-L_fix, 2 L_fix) with L_fix < 2^62: a sentinel at 3 * 2^61
        // on every axis is beyond every cutoff (more than L/2 from every own particle) and
        // no difference of upper words overflows
        g.hi[s.smax] = make_int4(3 << 29, 3 << 29, 3 << 29, 0);
        g.lo[s.smax] = make_uint4(0u, 0u, 0u, 0u);
    }
    __syncthreads();
}

__device__ __forceinline__ long long join64(int hi, unsigned lo) {
    return (long long)(((unsigned long long)(unsigned)hi << 32) | lo);
}

// 1/x, and 1/sqrt(x) with 1/x, in FP64: the hardware's approximation y (relative error e
// below 2^-18) and one third-order step, y (1 + e + e^2 [+ ...]) with e = 1 - x y or 1 - x y^2,
// whose own error is of order e^3 < 2^-54.  Either way 1/x has one rounding and little more: with
// the square root it comes from the rounded y^2 that e was taken of, for the square of the
// rounded 1/sqrt(x) would carry that one's error (forces of a liquid with the force shift were
// off by 1.85e-15 of their rms that way, by 1.15e-15 this way).
__device__ __forceinline__ double rcp64(double x) {
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double e = fma(-x, y, 1.0);
    return fma(y, fma(e, e, e), y);
}

__device__ __forceinline__ void rsqrt64(double x, double& r, double& r2) {
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double y2 = y * y;
    const double e = fma(-x, y2, 1.0);
    r = fma(fma(e, 0.375, 0.5), e * y, y);
    r2 = fma(fma(e, e, e), y2, y2);
}

// Queue entries per lane: full rows of 8 candidates are added while at most kQ64 - 8 wait.
constexpr int kQ64 = 32;
constexpr unsigned kBand64 = 0x8000u;  // entry left to the exact rule (staged indices < 2^15)

__device__ __forceinline__ uint16_t* warp_queue64(int w) {
    __shared__ uint16_t q_all[kBW][kQ64 * 32];
    return q_all[w];
}

// What the body computes: forces, per-particle energies (and their sums), or the sums of
// energy and virial alone.
enum : int { k64Force = 1, k64Energy = 2, k64Sums = 4 };

// One lane's pair constants and accumulators; r^2 and forces in units of 2^-k, so the constants
// of r^-6 carry 2^6k.  The energies are summed pair by pair (sums of r^-12 and r^-6 apart are
// larger than their difference, and so are their roundings: u_i of a liquid of LJ pairs was off
// by 4.0e-15 rms that way, by 1.7e-15 this way); the sum of the attractions completes the virial.
struct Lane64 {
    double a0, a1, b0, b1;                    // 48 eps sigma^12 2^6k, 24 eps sigma^6 (0: soft)
    double dc0, dc1;                          // dV/dr(rc) 2^-7k
    double e0, e1, g0, g1;                    // 4 eps sigma^12 2^6k, -4 eps sigma^6 (0: soft)
    double fx, fy, fz;                        // sum of f d
    double rc;                                // cutoff with species A 2^k
    double t0, t1;                            // sums of 4 eps ((sigma/r)^12 - (sigma/r)^6) by
                                              // species of j
    double at, q;                             // sums of -4 eps (sigma/r)^6 and (r - rc) dV/dr(rc)
    int n0, n1;                               // interacting pairs by species of j
};

template <int WHAT, bool FSHIFT>
__device__ __forceinline__ void pair_fp64(const DevSim& s, int si, long long mx, long long my,
                                          long long mz, const Stage64& g, unsigned ent, Lane64& A) {
    const int t = (int)(ent & (kBand64 - 1u));
    const int4 h = g.hi[t];
    const uint4 l = g.lo[t];
    const double dx = __ll2double_rn(join64(h.x, l.x) - mx);
    const double dy = __ll2double_rn(join64(h.y, l.y) - my);
    const double dz = __ll2double_rn(join64(h.z, l.z) - mz);
    const bool b = h.w & 1;
    if (ent & kBand64) {
        // the exact rule, in integer units (the scale is a power of two: the same roundings).
        // rc < L/2 (the box holds at least three cells of side >= rc per axis), so what it
        // accepts is the minimum-image copy (a region may hold a cell twice when nc = 3)
        const double e2 = __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
        if (!(e2 * s.sxd * s.sxd < s.pt.rc2[si * 2 + (b ? 1 : 0)])) return;
    }
    const double r2 = fma(dx, dx, fma(dy, dy, dz * dz));
    double ir2, ir = 0.0;
    if (FSHIFT) {
        rsqrt64(r2, ir, ir2);
    } else {
        ir2 = rcp64(r2);
    }
    const double ir4 = ir2 * ir2;
    const double ir6 = ir4 * ir2;
    if (WHAT & k64Force) {
        // f = (48 eps sigma^12 r^-6 - 24 eps sigma^6) r^-8 (+ dV/dr(rc) / r): the units of
        // r^-8 and d, 2^7k, are applied to the finished sum
        double f = fma(b ? A.a1 : A.a0, ir6, b ? A.b1 : A.b0) * (ir4 * ir4);
        if (FSHIFT) f = fma(b ? A.dc1 : A.dc0, ir, f);
        A.fx = fma(f, dx, A.fx);
        A.fy = fma(f, dy, A.fy);
        A.fz = fma(f, dz, A.fz);
    }
    if (WHAT & (k64Energy | k64Sums)) {
        // (selects, not branches: a divergent branch would take the FP64 pipe twice)
        const double gb = b ? A.g1 : A.g0;
        const double tn = fma(fma(b ? A.e1 : A.e0, ir6, gb), ir6, b ? A.t1 : A.t0);
        A.at = fma(gb, ir6, A.at);
        A.t0 = b ? A.t0 : tn;
        A.t1 = b ? tn : A.t1;
        if (FSHIFT) A.q = fma(b ? A.dc1 : A.dc0, fma(r2, ir, -A.rc), A.q);
        A.n0 += b ? 0 : 1;
        A.n1 += b ? 1 : 0;
    }
}

// WHAT: see above (k64Force writes F and Fd; k64Energy the per-particle energies u_i, half
// of each pair energy; k64Energy and k64Sums the energy and virial partials, from
// kEnergyPartial).
template <int MODE, int WHAT, bool KE, bool FSHIFT>
__device__ __forceinline__ void force64_body(const DevSim& s, int lb, int lg) {
    if (!force_selected<MODE>(s)) return;  // CTA-uniform, before any barrier
    if (!(WHAT & k64Force) && s.sums_role != kSumsOwn) {
        // (one thread looks: other CTAs of the pass may raise the bit meanwhile)
        const bool is_short = __syncthreads_or(threadIdx.x == 0 && (*(volatile int*)&s.sc->status & ST_SUMS_SHORT));
        if (is_short != (s.sums_role == kSumsStandIn)) return;
    }
    extern __shared__ float4 smem[];
    StageShared& ss = stage_shared();
    Region& R = ss.R[0];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const Stage64 g = stage64(s, smem);
    uint16_t* const q = warp_queue64(w) + lane;
    const bool lj = s.pt.potential == BBMD_POT_LJ;
    // FP32 thresholds in upper-word units: the truncation of the upper words moves a distance
    // by less than sqrt(3) units, FP32 rounding by less than 1e-6 of it
    const double inv_u = ldexp(1.0, s.kexp - 32);
    double acc_ke = 0.0, acc_u = 0.0, acc_w = 0.0;
    for (int64_t blk = lb; blk < s.nblocks; blk += lg) {
        const BlockPos bp = block_pos(s, blk);
        stage_block64(s, bp, R, g);
        own_chunks(s, bp, R, ss, [&](int t) { return (g.hi[t].w & 1) == 0; });
        // chunks go to the warps in a fixed order (the sums must not depend on timing)
        for (int item = w; item < ss.nch; item += kBW) {
            bool act;
            int64_t gi;
            int self;
            chunk_lane(ss, item, lane, act, gi, self);
            const int si = item >= ss.nchA ? 1 : 0;
            const int4 mh = g.hi[self];
            const uint4 ml = g.lo[self];
            const long long mx = join64(mh.x, ml.x), my = join64(mh.y, ml.y), mz = join64(mh.z, ml.z);
            float in2[2], out2[2];
#pragma unroll
            for (int b = 0; b < 2; ++b) {
                const float rc = (float)(s.pt.drc[si * 2 + b] * inv_u);
                const float lo = rc * (1.0f - 2e-6f) - 2.0f, hi = rc * (1.0f + 2e-6f) + 2.0f;
                in2[b] = lo > 0.f ? lo * lo : 0.f;
                out2[b] = hi * hi;
                // (kept in registers: computed anew for every candidate they cost FP64 operations
                // in the classification -- with the constants below so too, the sums of shifted
                // forces at 2.05 M in cell mode took 24 ms for 5)
                asm volatile("" : "+f"(in2[b]), "+f"(out2[b]));
            }
            const int kp = si * 2;
            Lane64 A;
            {
                const double c0 = s.pt.dsig2[kp] * s.pt.dsig2[kp] * s.pt.dsig2[kp];  // sigma^6
                const double c1 = s.pt.dsig2[kp + 1] * s.pt.dsig2[kp + 1] * s.pt.dsig2[kp + 1];
                A.a0 = ldexp(s.pt.deps48[kp] * c0 * c0, 6 * s.kexp);
                A.a1 = ldexp(s.pt.deps48[kp + 1] * c1 * c1, 6 * s.kexp);
                A.b0 = lj ? -0.5 * s.pt.deps48[kp] * c0 : 0.0;
                A.b1 = lj ? -0.5 * s.pt.deps48[kp + 1] * c1 : 0.0;
                A.e0 = ldexp(s.pt.deps4[kp] * c0 * c0, 6 * s.kexp);
                A.e1 = ldexp(s.pt.deps4[kp + 1] * c1 * c1, 6 * s.kexp);
                A.g0 = lj ? -s.pt.deps4[kp] * c0 : 0.0;
                A.g1 = lj ? -s.pt.deps4[kp + 1] * c1 : 0.0;
                A.dc0 = A.dc1 = A.rc = 0.0;
                if (FSHIFT) {
                    A.rc = ldexp(s.pt.drc[kp], s.kexp);
                    A.dc0 = ldexp(s.pt.dfcut[kp], -7 * s.kexp);
                    A.dc1 = ldexp(s.pt.dfcut[kp + 1], -7 * s.kexp);
                }
                // (kept in registers, or the compiler computes them anew for every pair, ldexp and
                // all: forces with the shift at 256 000 in cell mode 2.46 -> 1.80 ms)
                if (WHAT & k64Force) asm volatile("" : "+d"(A.a0), "+d"(A.a1));
                if (WHAT & (k64Energy | k64Sums)) asm volatile("" : "+d"(A.e0), "+d"(A.e1));
                if (FSHIFT) asm volatile("" : "+d"(A.dc0), "+d"(A.dc1));
                if (FSHIFT && (WHAT & (k64Energy | k64Sums))) asm volatile("" : "+d"(A.rc));
            }
            A.fx = A.fy = A.fz = A.t0 = A.t1 = A.at = A.q = 0.0;
            A.n0 = A.n1 = 0;
            int cnt = 0;
            // classify candidate t; queue it unless it is beyond the cutoff
            auto consider = [&](int t) {
                const int4 h = g.hi[t];
                const float x = (float)(int)((unsigned)h.x - (unsigned)mh.x);
                const float y = (float)(int)((unsigned)h.y - (unsigned)mh.y);
                const float z = (float)(int)((unsigned)h.z - (unsigned)mh.z);
                const float r2 = fmaf(x, x, fmaf(y, y, z * z));
                const bool b = h.w & 1;
                bool take = r2 < (b ? out2[1] : out2[0]);
                if (WHAT & k64Sums) {
                    // each pair from one side: the larger index where the two have the same
                    // parity, else the smaller (half of every particle's pairs)
                    const unsigned j = (unsigned)h.w >> 1, i = (unsigned)mh.w >> 1;
                    take = take && ((j < i) != (((j ^ i) & 1u) != 0u));
                }
                if (take) {
                    q[cnt * 32] = (uint16_t)((unsigned)t | (r2 < (b ? in2[1] : in2[0]) ? 0u : kBand64));
                    ++cnt;
                }
            };
            // pairs of the queues' tops until no lane holds more than `keep`
            auto drain = [&](int keep) {
                while (__any_sync(FULL, cnt > keep)) {
                    if (cnt > 0) {
                        --cnt;
                        pair_fp64<WHAT, FSHIFT>(s, si, mx, my, mz, g, q[cnt * 32], A);
                    }
                }
            };
            if (MODE == 0) {
                const int myrows = act ? (int)s.rows[gi] : 0;  // rows of the particle's list
                int nkb = myrows;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) nkb = max(nkb, __shfl_xor_sync(FULL, nkb, o));
                const uint4* lp = reinterpret_cast<const uint4*>(s.list) + gi;
                uint4 e = make_uint4(0u, 0u, 0u, 0u);
                if (myrows > 0) e = __ldcs(lp);
                for (int kb = 0; kb < nkb; ++kb) {
                    const unsigned ws[4] = {e.x, e.y, e.z, e.w};
                    if (kb + 1 < myrows) e = __ldcs(lp + (int64_t)(kb + 1) * s.npad);
                    if (kb < myrows) {
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            consider((int)lo16(ws[u]));
                            consider((int)hi16(ws[u]));
                        }
                    }
                    if (__any_sync(FULL, cnt > kQ64 - 8)) drain(kQ64 / 4);
                }
            } else {
                // the lane's own 27-cell stencil (the lanes of a chunk may lie in several cells)
                const int cq = act ? chunk_cell(ss, item, lane) : 0;
                for (int row = 0; row < 9; ++row) {
                    WarpCell wc;
                    wc.wr[0] = cq % kBlockXY;
                    wc.wr[1] = (cq / kBlockXY) % kBlockXY;
                    wc.wr[2] = cq / (kBlockXY * kBlockXY);
                    int rs, re;
                    stencil_run(R, wc, row, rs, re);
                    if (!act) re = rs;
                    int len = re - rs;
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) len = max(len, __shfl_xor_sync(FULL, len, o));
                    for (int o = 0; o < len; o += 8) {
#pragma unroll
                        for (int u = 0; u < 8; ++u) {
                            const int t = rs + o + u;
                            if (t < re && t != self) consider(t);
                        }
                        if (__any_sync(FULL, cnt > kQ64 - 8)) drain(kQ64 / 4);
                    }
                }
            }
            drain(0);
            double Fx = 0.0, Fy = 0.0, Fz = 0.0;
            if (WHAT & k64Force) {
                const double c = -ldexp(1.0, 7 * s.kexp);
                Fx = A.fx * c;
                Fy = A.fy * c;
                Fz = A.fz * c;
                if (act) {
                    if (!(isfinite(Fx) && isfinite(Fy) && isfinite(Fz))) set_status(s, ST_NONFINITE);
                    s.Fd[gi] = Fx;
                    s.Fd[s.npad + gi] = Fy;
                    s.Fd[2 * s.npad + gi] = Fz;
                    s.F[gi] = make_float4((float)Fx, (float)Fy, (float)Fz, 0.f);
                }
            }
            if (KE && act) {
                const double hm = 0.5 * s.sc->dt / s.pt.dmass[si];
                const double vx = __ll2double_rn(s.v[gi]) * 0x1p-52 + hm * Fx;
                const double vy = __ll2double_rn(s.v[s.npad + gi]) * 0x1p-52 + hm * Fy;
                const double vz = __ll2double_rn(s.v[2 * s.npad + gi]) * 0x1p-52 + hm * Fz;
                acc_ke += 0.5 * s.pt.dmass[si] * (vx * vx + vy * vy + vz * vz);
            }
            if ((WHAT & (k64Energy | k64Sums)) && act) {
                // V = 4 eps (s^12 - s^6) - V(rc) - (r - rc) dV/dr(rc), summed; virial
                // f r^2 = 12 (4 eps (s^12 - s^6)) + 6 (4 eps s^6) + r dV/dr(rc) (soft: no s^6).
                // (The units of the sums, 2^6k, and of q, 2^-6k: powers of two within range.)
                const double q = FSHIFT ? ldexp(A.q, 6 * s.kexp) : 0.0;
                const double v = ldexp(A.t0 + A.t1, 6 * s.kexp);
                double u = v - q, wv = fma(12.0, v, q) - 6.0 * ldexp(A.at, 6 * s.kexp);
#pragma unroll
                for (int b = 0; b < 2; ++b) {
                    const double np = (double)(b ? A.n1 : A.n0), dc = FSHIFT ? s.pt.dfcut[kp + b] : 0.0;
                    u -= np * (s.pt.dvshift[kp + b] + (s.pt.drc[kp] - s.pt.drc[kp + b]) * dc);
                    wv += np * (s.pt.drc[kp] * dc);
                }
                const double half = WHAT & k64Sums ? 1.0 : 0.5;
                if (WHAT & k64Energy) s.ud[gi] = half * u;
                acc_u += half * u;
                acc_w += half * wv;
            }
        }
        __syncthreads();
    }
    if (KE || (WHAT & (k64Energy | k64Sums))) {
        const double sums[3] = {warp_sum_d(acc_ke), warp_sum_d(acc_u), warp_sum_d(acc_w)};
        if (KE)
            block_partials(s, lb, sums, 0, 1);
        else
            block_partials(s, lb, sums + 1, kEnergyPartial, 2);
    }
}

#if !BBMD_WIDE
// ------------------------------------------------------------------ kernels ----
// Each body runs for one system (DevSim by value) or, in the _many form, for the replica of
// a batch that owns the CTA.

template <int MODE, bool KE, bool FSHIFT>
__global__ void __launch_bounds__(kBW * 32, MODE == 1 ? BBMD_CELL_MIN_BLOCKS : BBMD_FORCE_MIN_BLOCKS)
    k_force(DevSim s) {
    force_body<MODE, KE, FSHIFT>(s, (int)blockIdx.x, (int)gridDim.x);
}

template <int MODE, bool KE, bool FSHIFT>
__global__ void __launch_bounds__(kBW * 32, MODE == 1 ? BBMD_CELL_MIN_BLOCKS : BBMD_FORCE_MIN_BLOCKS)
    k_force_many(ManySims m) {
    __shared__ DevSim sh;
    int lb, lg;
    load_replica(m, sh, lb, lg);
    force_body<MODE, KE, FSHIFT>(sh, lb, lg);
}

constexpr bool kListBuffer = BBMD_BLOCK_Z != 4;  // (see the list build)

__global__ void __launch_bounds__(kBW * 32, BBMD_LIST_MIN_BLOCKS) k_list_build(DevSim s) {
    list_build_body<kListBuffer>(s, (int)blockIdx.x, (int)gridDim.x);
}

__global__ void __launch_bounds__(kBW * 32, BBMD_LIST_MIN_BLOCKS) k_list_build_many(ManySims m) {
    __shared__ DevSim sh;
    int lb, lg;
    load_replica(m, sh, lb, lg);
    list_build_body<kListBuffer>(sh, lb, lg);
}

template <int MODE, int WHAT, bool KE, bool FSHIFT>
__global__ void __launch_bounds__(kBW * 32) k_force64(DevSim s) {
    force64_body<MODE, WHAT, KE, FSHIFT>(s, (int)blockIdx.x, (int)gridDim.x);
}

template <int MODE, bool KE, bool FSHIFT>
__global__ void __launch_bounds__(kBW * 32) k_force64_many(ManySims m) {
    __shared__ DevSim sh;
    int lb, lg;
    load_replica(m, sh, lb, lg);
    force64_body<MODE, k64Force, KE, FSHIFT>(sh, lb, lg);
}

#endif  // !BBMD_WIDE

// Opt every kernel with dynamic shared memory into the largest size the device allows
// next to the kernel's static shared memory (done at create, outside any stream capture);
// each launch then requests only what it needs.
static bool g_smem_ok = true;

template <typename K>
void set_smem(K kernel) {
    int dev = 0, optin = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    cudaFuncAttributes fa;
    if (cudaFuncGetAttributes(&fa, kernel) != cudaSuccess) {
        g_smem_ok = false;
        return;
    }
    int dyn = optin - (int)fa.sharedSizeBytes;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, dyn) !=
        cudaSuccess)
        g_smem_ok = false;
}

#if !BBMD_WIDE
// Dynamic shared memory of the FP64 kernels: upper and lower words of every staged record.
static size_t smem64(int smax) { return (size_t)(smax + 1) * 32; }

// E: with per-particle energies (the FP64 form only; mixed precision has launch_energies).
template <int MODE, bool E, bool KE, bool FS>
void run_force(const DevSim& s, cudaStream_t st) {
    if (s.precision == BBMD_PREC_FP64) {
        k_force64<MODE, E ? k64Force | k64Energy : k64Force, KE, FS>
            <<<s.grid_cell, kBW * 32, smem64(s.smax), st>>>(s);
    } else {
        size_t bytes = kStageBuffers * (size_t)(s.smax + 1) * sizeof(float4);
        k_force<MODE, KE, FS><<<s.grid_cell, kBW * 32, bytes, st>>>(s);
    }
}

template <int MODE, bool KE, bool FS>
void run_force_many(const ManySims& m, int total, bool fp64, int smax_max, cudaStream_t st) {
    if (fp64) {
        k_force64_many<MODE, KE, FS><<<total, kBW * 32, smem64(smax_max), st>>>(m);
    } else {
        size_t bytes = kStageBuffers * (size_t)(smax_max + 1) * sizeof(float4);
        k_force_many<MODE, KE, FS><<<total, kBW * 32, bytes, st>>>(m);
    }
}

template <int MODE, bool FS>
void run_force_fs(const DevSim& s, cudaStream_t st, bool energy, bool ke) {
    if (energy) {
        run_force<MODE, true, false, FS>(s, st);  // (no caller asks for both)
    } else {
        if (ke) run_force<MODE, false, true, FS>(s, st); else run_force<MODE, false, false, FS>(s, st);
    }
}

template <int MODE>
void run_force_mode(const DevSim& s, cudaStream_t st, bool energy, bool ke, bool fs) {
    if (fs) run_force_fs<MODE, true>(s, st, energy, ke);
    else run_force_fs<MODE, false>(s, st, energy, ke);
}

template <int MODE, int WHAT>
void run_energies(const DevSim& s, cudaStream_t st, bool fs) {
    if (fs) k_force64<MODE, WHAT, false, true><<<s.grid_sums, kBW * 32, smem64(s.smax), st>>>(s);
    else k_force64<MODE, WHAT, false, false><<<s.grid_sums, kBW * 32, smem64(s.smax), st>>>(s);
}

template <int MODE, bool FS>
void prep_mode_fs() {
    set_smem(k_force<MODE, false, FS>);
    set_smem(k_force<MODE, true, FS>);
    set_smem(k_force_many<MODE, false, FS>);
    set_smem(k_force_many<MODE, true, FS>);
    set_smem(k_force64_many<MODE, false, FS>);
    set_smem(k_force64_many<MODE, true, FS>);
    set_smem(k_force64<MODE, k64Force, false, FS>);
    set_smem(k_force64<MODE, k64Force, true, FS>);
    set_smem(k_force64<MODE, k64Force | k64Energy, false, FS>);
    set_smem(k_force64<MODE, k64Energy, false, FS>);
    set_smem(k_force64<MODE, k64Sums, false, FS>);
}

template <int MODE>
void prep_mode() {
    prep_mode_fs<MODE, false>();
    prep_mode_fs<MODE, true>();
}

#endif  // !BBMD_WIDE

}  // namespace

// Attributes of the one-launch kernels.
static void prep_grid() {
    set_smem(k_step_grid<false, false>);
    set_smem(k_step_grid<true, false>);
    set_smem(k_step_grid<false, true>);
    set_smem(k_step_grid<true, true>);
    set_smem(k_relax_grid<false>);
    set_smem(k_relax_grid<true>);
}

#if BBMD_WIDE
bool prepare_force_kernels() {
    g_smem_ok = true;
    prep_grid();
    return g_smem_ok;
}
#else
int block_threads() { return kBW * 32; }

bool prepare_force_kernels() {
    g_smem_ok = true;
    prep_mode<0>();
    prep_mode<1>();
    set_smem(k_list_build);
    set_smem(k_list_build_many);
    prep_grid();
    return g_smem_ok;
}

int force_blocks_per_sm(const DevSim& s) {
    int nb = 0;
    size_t bytes = s.precision == BBMD_PREC_FP64 ? smem64(s.smax)
                                                 : kStageBuffers * (size_t)(s.smax + 1) * sizeof(float4);
    if (s.precision == BBMD_PREC_FP64)
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_force64<0, k64Force, true, false>, kBW * 32, bytes);
    else if (s.nbr_mode == BBMD_NBR_CELL)  // the stencil kernel is the step's force kernel
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_force<1, true, false>, kBW * 32, bytes);
    else
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_force<0, true, false>, kBW * 32, bytes);
    return nb > 0 ? nb : 1;
}

int list_blocks_per_sm(const DevSim& s) {
    int nb = 0;
    const size_t bytes = kStageBuffers * (size_t)(s.smax + 1) * sizeof(float4);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_list_build, kBW * 32, bytes);
    return nb > 0 ? nb : 1;
}

// Verlet mode launches the list kernel and, behind it, the stencil kernel: exactly one of
// the two runs, by the device flag of cut lists.
void launch_force(const DevSim& s, cudaStream_t st, bool energy, bool ke) {
    bool fs = s.pt.shift == BBMD_SHIFT_FORCE;
    if (s.nbr_mode == BBMD_NBR_VERLET) run_force_mode<0>(s, st, energy, ke, fs);
    run_force_mode<1>(s, st, energy, ke, fs);
}

// FP64 energies of the current positions from exact integer positions (FP32 coordinates would
// limit u_i to about 1e-4), either precision; the forces are left alone.  each: per-particle
// energies; else the energy and virial sums alone (partials of grid_sums CTAs, either way).
void launch_energies(const DevSim& s, cudaStream_t st, bool each) {
    const bool fs = s.pt.shift == BBMD_SHIFT_FORCE;
    if (s.nbr_mode == BBMD_NBR_VERLET) {
        if (each) run_energies<0, k64Energy>(s, st, fs);
        else run_energies<0, k64Sums>(s, st, fs);
    }
    if (each) run_energies<1, k64Energy>(s, st, fs);
    else run_energies<1, k64Sums>(s, st, fs);
}

int energies_blocks_per_sm(const DevSim& s) {
    int nb = 0;
    if (s.nbr_mode == BBMD_NBR_VERLET)
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_force64<0, k64Sums, false, false>, kBW * 32,
                                                      smem64(s.smax));
    else
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_force64<1, k64Sums, false, false>, kBW * 32,
                                                      smem64(s.smax));
    return nb > 0 ? nb : 1;
}

void launch_force_many(const ManySims& m, int total, bool fp64, bool cell, bool ke, bool fshift,
                       int smax_max, cudaStream_t st) {
    if (cell) {
        if (ke) {
            if (fshift) run_force_many<1, true, true>(m, total, fp64, smax_max, st);
            else run_force_many<1, true, false>(m, total, fp64, smax_max, st);
        } else {
            if (fshift) run_force_many<1, false, true>(m, total, fp64, smax_max, st);
            else run_force_many<1, false, false>(m, total, fp64, smax_max, st);
        }
    } else {
        // list kernel, then the stencil kernel that stands in for replicas with cut lists
        if (ke) {
            if (fshift) {
                run_force_many<0, true, true>(m, total, fp64, smax_max, st);
                run_force_many<1, true, true>(m, total, fp64, smax_max, st);
            } else {
                run_force_many<0, true, false>(m, total, fp64, smax_max, st);
                run_force_many<1, true, false>(m, total, fp64, smax_max, st);
            }
        } else {
            if (fshift) {
                run_force_many<0, false, true>(m, total, fp64, smax_max, st);
                run_force_many<1, false, true>(m, total, fp64, smax_max, st);
            } else {
                run_force_many<0, false, false>(m, total, fp64, smax_max, st);
                run_force_many<1, false, false>(m, total, fp64, smax_max, st);
            }
        }
    }
}

void launch_list_build_many(const ManySims& m, int total, int smax_max, cudaStream_t st) {
    const size_t bytes = kStageBuffers * (size_t)(smax_max + 1) * sizeof(float4);
    k_list_build_many<<<total, kBW * 32, bytes, st>>>(m);
}

void launch_list_build(const DevSim& s, cudaStream_t st) {
    if (s.nbr_mode != BBMD_NBR_VERLET) return;
    // staging buffer(s), each: staged region + sentinel record
    size_t bytes = kStageBuffers * (size_t)(s.smax + 1) * sizeof(float4);
    k_list_build<<<s.grid_list, kBW * 32, bytes, st>>>(s);
}

#endif  // BBMD_WIDE

// CTAs of the one-launch step: enough for every block and for 256 particles a CTA, at most
// what is resident at once.
int grid_step_ctas(const DevSim& s, int nsm) {
    const size_t bytes = kStageBuffers * (size_t)(s.smax + 1) * sizeof(float4);
    // (every form that may be launched with the grid: their static shared memory differs)
    const void* forms[] = {(const void*)k_step_grid<false, false>, (const void*)k_step_grid<false, true>,
                           (const void*)k_step_grid<true, false>, (const void*)k_step_grid<true, true>,
                           (const void*)k_relax_grid<false>, (const void*)k_relax_grid<true>};
    int nb = INT_MAX;
    for (const void* f : forms) {
        int one = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&one, f, kBW * 32, bytes) != cudaSuccess) {
            cudaGetLastError();
            return 0;
        }
        nb = one < nb ? one : nb;
    }
    int64_t want = (s.n + 255) / 256;
    if (want < s.nblocks) want = s.nblocks;
    return (int)(want < (int64_t)nb * nsm ? want : (int64_t)nb * nsm);
}

cudaError_t launch_grid_step(const DevSim& s, int grid, int nsteps, bool ke, cudaStream_t st) {
    DevSim a = s;
    void* params[] = {&a, &nsteps};
    const bool fs = s.pt.shift == BBMD_SHIFT_FORCE;
    const void* fn = ke ? (fs ? (const void*)k_step_grid<true, true> : (const void*)k_step_grid<true, false>)
                        : (fs ? (const void*)k_step_grid<false, true> : (const void*)k_step_grid<false, false>);
    const size_t bytes = kStageBuffers * (size_t)(s.smax + 1) * sizeof(float4);
    return cudaLaunchCooperativeKernel(fn, grid, kBW * 32, params, bytes, st);
}

cudaError_t launch_grid_relax(const DevSim& s, int grid, int nsteps, double hmax, double dmax,
                              cudaStream_t st) {
    DevSim a = s;
    void* params[] = {&a, &nsteps, &hmax, &dmax};
    const void* fn = s.pt.shift == BBMD_SHIFT_FORCE ? (const void*)k_relax_grid<true>
                                                    : (const void*)k_relax_grid<false>;
    const size_t bytes = kStageBuffers * (size_t)(s.smax + 1) * sizeof(float4);
    return cudaLaunchCooperativeKernel(fn, grid, kBW * 32, params, bytes, st);
}

#if BBMD_BLOCK_Z == BBMD_PERSIST_Z
// Dynamic shared memory of the persistent step for staged capacity smax_max.
static size_t persistent_smem(int smax_max) {
    return kStageBuffers * (size_t)(smax_max + 1) * sizeof(float4);
}

bool prepare_persistent() {
    g_smem_ok = true;
    set_smem(k_step_persistent<false, false>);
    set_smem(k_step_persistent<true, false>);
    set_smem(k_step_persistent<false, true>);
    set_smem(k_step_persistent<true, true>);
    return g_smem_ok;
}

int persistent_blocks_per_sm(int smax_max) {
    int nb = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_step_persistent<true, false>, kBW * 32,
                                                  persistent_smem(smax_max));
    return nb;
}

cudaError_t launch_persistent_step(const PersistentStep& a, int grid, int smax_max, bool ke,
                                   bool fshift, cudaStream_t st) {
    PersistentStep args = a;
    void* params[] = {&args};
    const void* fn = ke ? (fshift ? (const void*)k_step_persistent<true, true>
                                  : (const void*)k_step_persistent<true, false>)
                        : (fshift ? (const void*)k_step_persistent<false, true>
                                  : (const void*)k_step_persistent<false, false>);
    return cudaLaunchCooperativeKernel(fn, grid, kBW * 32, params, persistent_smem(smax_max), st);
}
#endif  // BBMD_BLOCK_Z == BBMD_PERSIST_Z

}  // namespace z<BBMD_BLOCK_Z>
}  // namespace bbmd
