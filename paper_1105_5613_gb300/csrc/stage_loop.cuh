// Staging of one CTA's blocks: the particles a cell contributes, and the order in which the
// blocks go through the buffers -- which buffer, which barrier phase, and what happens when a
// wait gives up.  Plain arithmetic, and control flow over an Ops object, so that it compiles for
// the host as well (tests/host_stage_loop.cpp drives it with a model of the barriers).
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define BBMD_STAGE_FN __device__ __forceinline__
#else
#define BBMD_STAGE_FN inline
#endif

namespace bbmd {

// Particles of a cell whose entries of the cell table are first and next, at most smax + 1 (the
// region overflows all the same, and a region's sum fits an int).  A launch that was given up
// half way through a sort leaves old and new entries side by side, each of them in [0, n]: the
// count is then never negative, and first + count never beyond the larger of the two.
BBMD_STAGE_FN int cell_count(int first, int next, int smax) {
    const int c = next > first ? next - first : 0;
    return c > smax ? smax + 1 : c;
}

// Particle of staged entry t <= smax of a region of `cells` cells, from its prefix off and first
// particles start.  A list from before a launch that was given up can name entries beyond
// those staged: the index is then at most n + smax, which the positions' array covers.  (An index
// cut at n costs the list-mode forces up to 1 %.)
BBMD_STAGE_FN int64_t staged_particle(const int* start, const int* off, int cells, int t) {
    int lo = 0, hi = cells - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (off[mid] <= t) lo = mid;
        else hi = mid - 1;
    }
    return (int64_t)start[lo] + (t - off[lo]);
}

// Blocks lb, lb + lg, ... of system s (below s.nblocks).  With two buffers the copies of the next block are
// in flight while a block is computed; with one, each block is staged, then computed.
//   ops.open()                initialise the buffers' barriers, synchronise the CTA
//   ops.position(s, block)    where the block lies (64-bit divisions: once a block)
//   ops.issue(s, pos, b)      start the copies of the block into buffer b
//   ops.finish(s, b, parity)  wait for them; false (on every thread) if the wait gave up
//   ops.compute(pos, b, body) compute the staged block (no CTA barrier inside)
//   ops.drain(s, b, parity)   bounded wait for copies whose block will not be computed
//   ops.sync()                CTA barrier: buffer b is read no more
//   ops.close()               invalidate the barriers: a kernel that runs several bodies opens
//                             the same ones again, and initialising a live mbarrier is undefined
// False after a wait that gave up: the barriers are then left as they are (copies could still
// be in flight), and the CTA must not stage again.  (The system is handed through, not held by
// ops: a reference inside an object would make the kernels copy their parameters to the stack.)
template <int BUFFERS, class Ops, class Sim, class Body>
BBMD_STAGE_FN bool staged_blocks(const Sim& s, Ops ops, int lb, int lg, Body& body) {
    static_assert(BUFFERS == 1 || BUFFERS == 2, "one or two staging buffers");
    ops.open();
    int64_t blk = lb;
    if (BUFFERS == 1) {
        for (int it = 0; blk < s.nblocks; ++it, blk += lg) {
            const auto pos = ops.position(s, blk);
            ops.issue(s, pos, 0);
            if (!ops.finish(s, 0, (uint32_t)(it & 1))) return false;
            ops.compute(pos, 0, body);
            ops.sync();
        }
    } else {
        auto pos = ops.position(s, blk);
        if (blk < s.nblocks) ops.issue(s, pos, 0);
        for (int it = 0; blk < s.nblocks; ++it, blk += lg) {
            const int cur = it & 1;
            const bool more = blk + lg < s.nblocks;
            const auto next = ops.position(s, blk + lg);
            if (more) ops.issue(s, next, cur ^ 1);
            if (!ops.finish(s, cur, (uint32_t)((it >> 1) & 1))) {
                if (more) ops.drain(s, cur ^ 1, (uint32_t)(((it + 1) >> 1) & 1));
                return false;
            }
            ops.compute(pos, cur, body);
            ops.sync();
            pos = next;
        }
    }
    ops.close();
    return true;
}

}  // namespace bbmd
