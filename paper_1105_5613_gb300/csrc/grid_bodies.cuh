// Grid-wide barrier of the cooperative kernels, and the rebuild trigger and sort chain run
// phase after phase inside one launch.  Included inside an anonymous namespace, after
// sort_bodies.cuh and step_bodies.cuh.
#pragma once

__device__ __forceinline__ unsigned long long globaltimer_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Barrier over the CTAs of the launch; gen counts the barriers passed.  With `last` set, the
// last CTA to arrive runs on_last before the others go on.  Every CTA is resident
// (cooperative launch), so a wait ends; should one not end within s.wait_ns, the CTA
// raises the abort flag and ST_TIMEOUT, and every CTA leaves (false) at its next barrier.
// The clock is read at every 64th look, or at every one where the limit is below a millisecond.
template <class OnLast>
__device__ __forceinline__ bool grid_barrier(const DevSim& s, unsigned& gen, bool last, OnLast on_last) {
    __shared__ int verdict;  // 0: abort, 1: go on, 2: this CTA arrived last
    volatile uint32_t* const w = s.gsync;
    ++gen;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        const unsigned target = gen * gridDim.x;
        const bool mine = atomicAdd(&s.gsync[kSyncArrive * kSyncStride], 1u) + 1u == target;
        int v = 1;
        if (last && mine) {
            v = 2;
        } else {
            const int word = (last ? kSyncRelease : kSyncArrive) * kSyncStride;
            const unsigned want = last ? gen : target;
            const unsigned skip = s.wait_ns < 1000000ull ? 0u : 63u;
            unsigned long long t0 = 0;
            for (unsigned it = 0; w[word] < want; ++it) {
                if ((it & skip) != skip) continue;
                if (t0 == 0) t0 = globaltimer_ns();
                if (w[kSyncAbort * kSyncStride] != 0u || globaltimer_ns() - t0 > s.wait_ns) {
                    w[kSyncAbort * kSyncStride] = 1u;
                    set_status(s, ST_TIMEOUT);
                    v = 0;
                    break;
                }
            }
        }
        __threadfence();
        verdict = v;
    }
    __syncthreads();
    const int v = verdict;
    if (v == 2) {
        on_last();
        __syncthreads();
        if (threadIdx.x == 0) {
            __threadfence();
            w[kSyncRelease * kSyncStride] = gen;
        }
    }
    __syncthreads();  // (verdict is written again at the next barrier)
    // data of earlier phases, written by other CTAs, is read by bulk copies (the async
    // proxy) as well as by ordinary loads
    asm volatile("fence.proxy.async.global;" ::: "memory");
    return v != 0;
}

__device__ __forceinline__ bool grid_barrier(const DevSim& s, unsigned& gen) {
    return grid_barrier(s, gen, false, [] {});
}

// Ends the launch for a CTA that cannot go on: the others leave at their next barrier.
__device__ __forceinline__ bool grid_abort(const DevSim& s) {
    if (threadIdx.x == 0) *(volatile uint32_t*)&s.gsync[kSyncAbort * kSyncStride] = 1u;
    return false;
}

// Rebuild trigger after the integrate phase (whose flags the caller has put behind a barrier):
// due, the same on every thread, tells whether a rebuild is due; the cell counts are then
// zero.  False after an abort.
__device__ __forceinline__ bool grid_trigger(const DevSim& s, unsigned& gen, bool& due) {
    const int lb = (int)blockIdx.x, lg = (int)gridDim.x;
    due = false;
    if (!*(volatile int*)&s.sc->near) return true;
    celltop_body(s, lb, lg);
    zero_counts(s, lb, lg);
    if (!grid_barrier(s, gen)) return false;
    check_body(s, lb, lg);
    if (!grid_barrier(s, gen)) return false;
    due = *(volatile int*)&s.sc->rebuild != 0;
    return true;
}

// Sort chain of a rebuild whose flag is up and whose cell counts are zero (no barrier after
// the last phase).
__device__ __forceinline__ bool grid_sort(const DevSim& s, unsigned& gen) {
    const int lb = (int)blockIdx.x, lg = (int)gridDim.x;
    clear_list_flags(s, lb);
    bin_body(s, lb, lg);
    if (!grid_barrier(s, gen)) return false;
    // cell starts: one CTA's scan where it holds all cells at once; else every CTA sums its
    // chunk, and adds the sums of the chunks before to its scan
    const int per = (int)blockDim.x * kScanItems;
    const int chunks = (s.ncell + per - 1) / per;
    if (chunks == 1 || chunks > lg || chunks > kScanParts) {
        scan_cta_body(s, lb, lg);
    } else {
        if (lb < chunks) scan_chunk_sum(s, lb);
        if (!grid_barrier(s, gen)) return false;
        if (lb < chunks) scan_chunk_down(s, lb, chunks);
    }
    if (!grid_barrier(s, gen)) return false;
    scatter_body(s, lb, lg);
    if (!grid_barrier(s, gen)) return false;
    sortgather_body(s, lb, lg);
    if (!grid_barrier(s, gen)) return false;
    copyback_body(s, lb, lg);
    return true;
}
