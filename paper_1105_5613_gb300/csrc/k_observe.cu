// Radial distribution function (Sec. 4, the g(r) of the glass study): partial ordered-pair
// histograms n_ab(q), q = floor(r / dr), r from the exact r^2 rule.
//
// Pairs are found in the cells of the last rebuild, whose particles lie contiguous (k_gr_rows);
// where the box has too few of them for rmax, on a coarse grid of cells of side >= rmax (one
// CTA per coarse cell, the 27 neighbour cells streamed through shared memory) or, when the
// box holds fewer than three of those per axis, by all pairs.  Distances are formed in FP32
// (on the last two paths from the exact integer displacement rounded once); a pair whose
// r / dr lies so near a bin edge that FP32 could be on the wrong side is binned again with
// the FP64 rule, so every count equals the FP64 definition.
#include "bbmd_internal.cuh"

namespace bbmd {

namespace {

constexpr int kT = 256;
constexpr int kChunk = 256;
constexpr float kEdgeTol = 5e-4f;

struct GrArgs {
    int nbins;
    float inv_dr, rmax2_hi;
    double dr;
    int ncg[3];
    long long Dg[3];
    int ncells;
    int32_t *gkey, *gidx, *gcount, *gstart, *gcursor;
};

__device__ __forceinline__ int bin_exact(const DevSim& s, const GrArgs& g, long long dx,
                                         long long dy, long long dz) {
    double a = __dmul_rn(__ll2double_rn(dx), s.sxd);
    double b = __dmul_rn(__ll2double_rn(dy), s.sxd);
    double c = __dmul_rn(__ll2double_rn(dz), s.sxd);
    double r2 = __dadd_rn(__dadd_rn(__dmul_rn(a, a), __dmul_rn(b, b)), __dmul_rn(c, c));
    double q = floor(__ddiv_rn(__dsqrt_rn(r2), g.dr));
    return q < (double)g.nbins ? (int)q : -1;
}

// Bin of one pair from its exact integer displacement (-1: outside the range).
__device__ __forceinline__ int pair_bin(const DevSim& s, const GrArgs& g, long long dx, long long dy,
                                       long long dz) {
    float fx = i64_to_f32(dx) * s.sx, fy = i64_to_f32(dy) * s.sx, fz = i64_to_f32(dz) * s.sx;
    float r2 = fmaf(fx, fx, fmaf(fy, fy, fz * fz));
    if (!(r2 < g.rmax2_hi)) return -1;
    float qf = sqrtf(r2) * g.inv_dr;
    float fl = floorf(qf);
    float fr = qf - fl;
    if (fr < kEdgeTol || fr > 1.0f - kEdgeTol || fl >= (float)g.nbins - 1.0f)
        return bin_exact(s, g, dx, dy, dz);
    return (int)fl;
}

__global__ void k_gr_zero(GrArgs g) {
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c <= g.ncells; c += gridDim.x * blockDim.x) {
        g.gcount[c] = 0;
        g.gcursor[c] = 0;
    }
}

__global__ void k_gr_key(DevSim s, GrArgs g) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < s.n;
         i += (int64_t)gridDim.x * blockDim.x) {
        int a[3];
        for (int d = 0; d < 3; ++d) a[d] = cell_axis((long long)s.x[d * s.npad + i], g.Dg[d], g.ncg[d]);
        int c = (a[2] * g.ncg[1] + a[1]) * g.ncg[0] + a[0];
        g.gkey[i] = c;
        atomicAdd(&g.gcount[c], 1);
    }
}

__global__ void k_gr_scan(GrArgs g) {
    // one block: exclusive scan of gcount into gstart
    __shared__ int carry;
    __shared__ int ws[32];
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    for (int base = 0; base < g.ncells; base += blockDim.x) {
        int idx = base + threadIdx.x;
        int v = idx < g.ncells ? g.gcount[idx] : 0;
        int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
        int incl = v;
        for (int o = 1; o < 32; o <<= 1) {
            int t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        if (lane == 31) ws[w] = incl;
        __syncthreads();
        if (w == 0) {
            int x = lane < (int)(blockDim.x >> 5) ? ws[lane] : 0;
            int xi = x;
            for (int o = 1; o < 32; o <<= 1) {
                int t = __shfl_up_sync(0xffffffffu, xi, o);
                if (lane >= o) xi += t;
            }
            ws[lane] = xi - x;
        }
        __syncthreads();
        int ex = ws[w] + incl - v;
        if (idx < g.ncells) g.gstart[idx] = carry + ex;
        __syncthreads();
        if (threadIdx.x == blockDim.x - 1) carry += ex + v;
        __syncthreads();
    }
    if (threadIdx.x == 0) g.gstart[g.ncells] = carry;
}

__global__ void k_gr_scatter(DevSim s, GrArgs g) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < s.n;
         i += (int64_t)gridDim.x * blockDim.x) {
        int c = g.gkey[i];
        g.gidx[g.gstart[c] + atomicAdd(&g.gcursor[c], 1)] = (int32_t)i;
    }
}

struct JEnt {
    long long x, y, z;
    int sp, gi;
};

__device__ void flush_hist(unsigned* hist, int nb4, unsigned long long* counts) {
    __syncthreads();
    for (int q = threadIdx.x; q < nb4; q += blockDim.x)
        if (hist[q]) atomicAdd(&counts[q], (unsigned long long)hist[q]);
    __syncthreads();
    for (int q = threadIdx.x; q < nb4; q += blockDim.x) hist[q] = 0;
    __syncthreads();
}

__global__ void __launch_bounds__(kT) k_gr_cells(DevSim s, GrArgs g, unsigned long long* counts) {
    extern __shared__ unsigned char gsm[];
    JEnt* stg = reinterpret_cast<JEnt*>(gsm);
    unsigned* hist = reinterpret_cast<unsigned*>(stg + kChunk);
    const int nb4 = 4 * g.nbins;
    for (int q = threadIdx.x; q < nb4; q += blockDim.x) hist[q] = 0;
    __syncthreads();
    for (int c = blockIdx.x; c < g.ncells; c += gridDim.x) {
        int a[3] = {c % g.ncg[0], (c / g.ncg[0]) % g.ncg[1], c / (g.ncg[0] * g.ncg[1])};
        int cs = g.gstart[c], ce = g.gstart[c + 1];
        for (int ib = cs; ib < ce; ib += kT) {
            int li = ib + threadIdx.x;
            bool act = li < ce;
            int64_t gi = act ? g.gidx[li] : 0;
            long long xi = act ? (long long)s.x[gi] : 0, yi = act ? (long long)s.x[s.npad + gi] : 0,
                      zi = act ? (long long)s.x[2 * s.npad + gi] : 0;
            int si = act ? s.sp[gi] : 0;
            for (int q = 0; q < 27; ++q) {
                int o[3] = {q % 3 - 1, (q / 3) % 3 - 1, q / 9 - 1};
                int b[3];
                long long wr[3];
                for (int d = 0; d < 3; ++d) {
                    int bb = a[d] + o[d];
                    wr[d] = 0;
                    if (bb < 0) {
                        bb += g.ncg[d];
                        wr[d] = -s.Lfix[d];
                    } else if (bb >= g.ncg[d]) {
                        bb -= g.ncg[d];
                        wr[d] = s.Lfix[d];
                    }
                    b[d] = bb;
                }
                int nb = (b[2] * g.ncg[1] + b[1]) * g.ncg[0] + b[0];
                int js = g.gstart[nb], je = g.gstart[nb + 1];
                for (int jb = js; jb < je; jb += kChunk) {
                    int cntc = min(kChunk, je - jb);
                    __syncthreads();
                    for (int t = threadIdx.x; t < cntc; t += blockDim.x) {
                        int gj = g.gidx[jb + t];
                        JEnt e;
                        e.x = (long long)s.x[gj] + wr[0];
                        e.y = (long long)s.x[s.npad + gj] + wr[1];
                        e.z = (long long)s.x[2 * s.npad + gj] + wr[2];
                        e.sp = s.sp[gj];
                        e.gi = gj;
                        stg[t] = e;
                    }
                    __syncthreads();
                    if (act) {
                        for (int t = 0; t < cntc; ++t) {
                            JEnt e = stg[t];
                            if (e.gi == (int)gi) continue;
                            int bin = pair_bin(s, g, e.x - xi, e.y - yi, e.z - zi);
                            if (bin >= 0) atomicAdd(&hist[(si * 2 + e.sp) * g.nbins + bin], 1u);
                        }
                    }
                }
            }
        }
    }
    flush_hist(hist, nb4, counts);
}

// All pairs (small boxes): block b takes i in [b*kT, b*kT + kT), j streamed in chunks.
__global__ void __launch_bounds__(kT) k_gr_all(DevSim s, GrArgs g, unsigned long long* counts) {
    extern __shared__ unsigned char gsm[];
    JEnt* stg = reinterpret_cast<JEnt*>(gsm);
    unsigned* hist = reinterpret_cast<unsigned*>(stg + kChunk);
    const int nb4 = 4 * g.nbins;
    for (int q = threadIdx.x; q < nb4; q += blockDim.x) hist[q] = 0;
    __syncthreads();
    for (int64_t ib = (int64_t)blockIdx.x * kT; ib < s.n; ib += (int64_t)gridDim.x * kT) {
        int64_t gi = ib + threadIdx.x;
        bool act = gi < s.n;
        long long xi = act ? (long long)s.x[gi] : 0, yi = act ? (long long)s.x[s.npad + gi] : 0,
                  zi = act ? (long long)s.x[2 * s.npad + gi] : 0;
        int si = act ? s.sp[gi] : 0;
        for (int64_t jb = 0; jb < s.n; jb += kChunk) {
            int cntc = (int)min((int64_t)kChunk, s.n - jb);
            __syncthreads();
            for (int t = threadIdx.x; t < cntc; t += blockDim.x) {
                int64_t gj = jb + t;
                JEnt e;
                e.x = (long long)s.x[gj];
                e.y = (long long)s.x[s.npad + gj];
                e.z = (long long)s.x[2 * s.npad + gj];
                e.sp = s.sp[gj];
                e.gi = (int)gj;
                stg[t] = e;
            }
            __syncthreads();
            if (act) {
                for (int t = 0; t < cntc; ++t) {
                    JEnt e = stg[t];
                    if (e.gi == (int)gi) continue;
                    long long dx = min_image(e.x - xi, s.Lfix[0]);
                    long long dy = min_image(e.y - yi, s.Lfix[1]);
                    long long dz = min_image(e.z - zi, s.Lfix[2]);
                    int bin = pair_bin(s, g, dx, dy, dz);
                    if (bin >= 0) atomicAdd(&hist[(si * 2 + e.sp) * g.nbins + bin], 1u);
                }
            }
        }
        // keep the 32-bit shared counters far from overflow
        flush_hist(hist, nb4, counts);
    }
    flush_hist(hist, nb4, counts);
}

// ------------------------------------------------------------ over the build cells ----
// A warp takes 32 particles at a time, one per lane, from segments of S cells along x (a
// chunk may cross cell boundaries, so the lanes are full).  The candidates are the particles
// of the cells within reach: the cells up to R away hold every particle within rmax, whose
// displacements since the build are bounded (rebuild trigger).  A row of cells along x is
// contiguous in memory, so the candidates come in runs, 32 loads at a time; those within
// rmax of the lanes' bounding box are compacted into a ring in shared memory, and each ring
// word is tested by all lanes (broadcast reads).  A lane queues its pairs within rmax, and
// the warp bins the queues together, a pair on nearly every lane.  Every pair is taken once
// (rows after the lane's own, and later particles of its own row) and counted for both
// orders when the CTA's histogram is added to the result.
//
// Bound: dependent instructions (57 % of the issue slots; the waits between them, shared-memory
// reads and the square roots the rest) of about 1000 ring entries and 310 binned
// pairs a particle at rmax = 5, against 5700 candidates in 64-bit arithmetic on the coarse grid:
// 108 000 particles, 500 bins, 4.2 -> 0.40 ms (0.51 when each ring word's pairs were binned on
// their own, chunks within cells).

constexpr int kRowWarps = 8;
constexpr int kRowRing = 64;
constexpr int kRowQueue = 24;  // pairs queued per lane (8 ring entries are tested between looks)

struct GrRows {
    int nbins, R[3], S, segs_x, slots;  // cells, segments of a row; chunks of a segment
    int64_t ntiles;
    float D[3];               // cell sides (exact in FP32: they have 24 significant bits)
    float gap[3];             // box side - cells x cell side: what a run past the seam adds
    float rmax, inv_dr;
};

struct RowRing {
    float4 p[kRowRing];               // position from the frame; w = (index << 1) | species
    float2 q[kRowQueue + 1][32];      // per lane: r^2 and w of the pairs to bin
};

// Add the CTA's histogram (AA, AB, BB) to the counts of ordered pairs and clear it; any
// thread may add to it meanwhile.
__device__ void flush_rows(unsigned* hist, int nbins, unsigned long long* counts, int first, int step) {
    for (int q = first; q < 3 * nbins; q += step) {
        const unsigned h = atomicExch(&hist[q], 0u);
        if (!h) continue;
        const int kind = q / nbins, b = q - kind * nbins;
        if (kind == 1) {
            atomicAdd(&counts[nbins + b], (unsigned long long)h);
            atomicAdd(&counts[2 * nbins + b], (unsigned long long)h);
        } else {
            atomicAdd(&counts[(kind == 0 ? 0 : 3) * nbins + b], 2ull * h);
        }
    }
}

__global__ void __launch_bounds__(kRowWarps * 32, 3) k_gr_rows(DevSim s, GrArgs ex, GrRows g,
                                                              unsigned long long* counts) {
    extern __shared__ __align__(16) unsigned char rsm[];
    RowRing* const rings = reinterpret_cast<RowRing*>(rsm);
    unsigned* const hist = reinterpret_cast<unsigned*>(rings + kRowWarps);  // [3][nbins]
    constexpr unsigned ALL = 0xffffffffu;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int q = threadIdx.x; q < 3 * g.nbins; q += blockDim.x) hist[q] = 0;
    __syncthreads();
    RowRing& ring = rings[w];
    const int nx = s.nc[0], ny = s.nc[1], nz = s.nc[2];
    unsigned long long added = 0;  // bound on what this warp has added since its last flush
    for (int64_t tile = (int64_t)blockIdx.x * kRowWarps + w; tile < g.ntiles;
         tile += (int64_t)gridDim.x * kRowWarps) {
        // slot-major: the first chunks of all segments, then the second ones, ...
        const int64_t nseg = g.ntiles / g.slots;
        const int slot = (int)(tile / nseg);
        const int64_t seg = tile - slot * nseg;
        const int xs = (int)(seg % g.segs_x) * g.S, xe = min(xs + g.S, nx);
        const int64_t row = seg / g.segs_x;
        const int y = (int)(row % ny), z = (int)(row / ny);
        const int home = (int)row * nx;
        const int is = s.cell_start[home + xs];
        int ie = s.cell_start[home + xe];
        if (slot + 1 < g.slots) ie = min(ie, is + (slot + 1) * 32);  // (the last takes the rest)
        for (int ib = is + slot * 32; ib < ie; ib += 32) {
            const int gi = ib + lane;
            const bool act = gi < ie;
            float mx = 0.f, my = 0.f, mz = 0.f;
            int si = 0, ax = 0;
            if (act) {
                const float4 r = s.rel[gi];
                const int wb = __float_as_int(s.relb[gi].w);
                ax = (wb >> 1) - home;
                mx = r.x;
                my = r.y;
                mz = r.z;
                si = wb & 1;
            }
            // the chunk's first and last cell; its frame is that of the first
            const int x0 = __shfl_sync(ALL, ax, 0), x1 = __shfl_sync(ALL, ax, min(31, ie - 1 - ib));
            mx = fmaf((float)(ax - x0), g.D[0], mx);
            // bounding box of the lanes
            float lo[3] = {act ? mx : 1e30f, act ? my : 1e30f, act ? mz : 1e30f};
            float hi[3] = {act ? mx : -1e30f, act ? my : -1e30f, act ? mz : -1e30f};
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    lo[d] = fminf(lo[d], __shfl_xor_sync(ALL, lo[d], o));
                    hi[d] = fmaxf(hi[d], __shfl_xor_sync(ALL, hi[d], o));
                }
            // bound on the FP32 error of a distance.  Per axis: the two frame-relative
            // coordinates and the seam's gap added to one (below D), the frame offset and the
            // coordinates' sums with it (below span for a lane, span + rmax for a candidate
            // within reach) and the difference (below rmax) are each rounded by 2^-24 of their
            // value: times sqrt(3), below 3.2e-7 (D + span + rmax).  The squares' sum, the square
            // root (2^-23) and the scaling add 3.5e-7 r.
            float span = 0.f;
#pragma unroll
            for (int d = 0; d < 3; ++d) span = fmaxf(span, fmaxf(fabsf(lo[d]), fabsf(hi[d])));
            const float err = 3.2e-7f * (span + g.rmax + fmaxf(g.D[0], fmaxf(g.D[1], g.D[2]))) + 3.5e-7f * g.rmax;
            const float tol = err * g.inv_dr;
            const float reach = g.rmax + 2.f * err, reach2 = reach * reach;
            const float keep2 = reach2 * 1.00001f, lim2 = act ? reach2 : -1.f;
            int fill = 0, done = 0, cnt = 0;
            auto drain = [&](int keep) {
                while (__any_sync(ALL, cnt > keep)) {
                    if (cnt > 0) {
                        --cnt;
                        const float2 e = ring.q[cnt][lane];
                        const unsigned jw = __float_as_uint(e.y);
                        float r;
                        asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(e.x));
                        const float qf = r * g.inv_dr;
                        const float fl = floorf(qf), fr = qf - fl;
                        int bin = (int)fl;
                        if (fr < tol || fr > 1.0f - tol) {
                            long long d3[3];
#pragma unroll
                            for (int d = 0; d < 3; ++d)
                                d3[d] = min_image((long long)s.x[d * s.npad + (jw >> 1)] -
                                                      (long long)s.x[d * s.npad + gi], s.Lfix[d]);
                            bin = bin_exact(s, ex, d3[0], d3[1], d3[2]);
                        }
                        if (bin >= 0 && bin < g.nbins)
                            atomicAdd(&hist[(si + (int)(jw & 1u)) * g.nbins + bin], 1u);
                    }
                }
            };
            // ring entry p: always stored at the queue's top, which moves on if the pair is within
            // reach (no branch)
            auto test = [&](const float4 p, bool ok) {
                const float dx = p.x - mx, dy = p.y - my, dz = p.z - mz;
                const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
                ring.q[cnt][lane] = make_float2(r2, p.w);
                cnt += r2 < lim2 && ok ? 1 : 0;
            };
            // the next 32 ring entries: pairs within reach are queued.  own: entries of the lanes'
            // own row (later particles only)
            auto word = [&](bool own) {
                const float4* const rp = ring.p + (done & (kRowRing - 1));
                const unsigned me = (unsigned)gi << 1 | 1u;
                for (int u0 = 0; u0 < 32; u0 += 8) {
                    if (own) {
#pragma unroll
                        for (int u = 0; u < 8; ++u) test(rp[u0 + u], __float_as_uint(rp[u0 + u].w) > me);
                    } else {
#pragma unroll
                        for (int u = 0; u < 8; ++u) test(rp[u0 + u], true);
                    }
                    if (__any_sync(ALL, cnt > kRowQueue - 8)) drain(kRowQueue / 4);
                }
                done += 32;
                __syncwarp();
            };
            // a last, partial word is filled up with entries beyond every reach
            auto last_word = [&](bool own) {
                if (fill == done) return;
                if (fill + lane < done + 32)
                    ring.p[(fill + lane) & (kRowRing - 1)] = make_float4(1e15f, 1e15f, 1e15f, 0.f);
                __syncwarp();
                word(own);
                fill = done;
            };
            for (int dz = 0; dz <= g.R[2]; ++dz) {
                const bool zw = z + dz >= nz;
                const int zz = zw ? z + dz - nz : z + dz;
                const float oz = fmaf((float)dz, g.D[2], zw ? g.gap[2] : 0.f);
                for (int dy = dz == 0 ? 0 : -g.R[1]; dy <= g.R[1]; ++dy) {
                    const int yw = y + dy, yy = yw < 0 ? yw + ny : (yw >= ny ? yw - ny : yw);
                    const int rb = (zz * ny + yy) * nx;
                    const float oy = fmaf((float)dy, g.D[1], yw < 0 ? -g.gap[1] : (yw >= ny ? g.gap[1] : 0.f));
                    for (int piece = -1; piece <= 1; ++piece) {  // the row's part in image `piece`
                        const int sh = piece * nx;
                        const int a = max(x0 - g.R[0], sh), b = min(x1 + g.R[0], sh + nx - 1);
                        if (a > b) continue;
                        const float ox = (float)piece * g.gap[0];
                        const int js = s.cell_start[rb + a - sh], je = s.cell_start[rb + b - sh + 1];
                        for (int jb = js; jb < je; jb += 32) {
                            const int j = jb + lane;
                            bool keep = false;
                            float4 p = make_float4(0.f, 0.f, 0.f, 0.f);
                            if (j < je) {
                                const float4 r = s.rel[j];
                                const int wb = __float_as_int(s.relb[j].w);
                                p.x = fmaf((float)((wb >> 1) - rb + sh - x0), g.D[0], r.x + ox);
                                p.y = r.y + oy;
                                p.z = r.z + oz;
                                p.w = __uint_as_float(((unsigned)j << 1) | (unsigned)(wb & 1));
                                const float bx = fmaxf(fmaxf(lo[0] - p.x, p.x - hi[0]), 0.f);
                                const float by = fmaxf(fmaxf(lo[1] - p.y, p.y - hi[1]), 0.f);
                                const float bz = fmaxf(fmaxf(lo[2] - p.z, p.z - hi[2]), 0.f);
                                keep = fmaf(bz, bz, fmaf(by, by, bx * bx)) < keep2;
                            }
                            const unsigned m = __ballot_sync(ALL, keep);
                            if (keep) ring.p[(fill + __popc(m & ((1u << lane) - 1u))) & (kRowRing - 1)] = p;
                            fill += __popc(m);
                            __syncwarp();
                            if (fill - done >= 32) word(dz == 0 && dy == 0);
                        }
                        added += (unsigned long long)(je - js) * 32u;
                    }
                    if (dz == 0 && dy == 0) last_word(true);  // the own row's rule ends here
                }
            }
            last_word(false);
            drain(0);
            if (added > (1ull << 28)) {  // keep the 32-bit counters far from overflow
                flush_rows(hist, g.nbins, counts, lane, 32);
                added = 0;
            }
        }
    }
    __syncthreads();
    flush_rows(hist, g.nbins, counts, threadIdx.x, blockDim.x);
}

// Whether the build cells serve rmax, and the arguments of k_gr_rows: R cells to each side
// hold everything within rmax given the bound on displacements since the build, and the
// cells of a row within reach are distinct.
bool gr_rows(const DevSim& s, int nbins, double rmax, GrRows& g) {
    const double moved = s.nbr_mode == BBMD_NBR_VERLET ? fmin(s.disp_thr, s.disp_far) : s.disp_far;
    g.nbins = nbins;
    g.rmax = (float)rmax;
    g.inv_dr = (float)(nbins / rmax);
    for (int d = 0; d < 3; ++d) {
        const double D = ldexp((double)s.D[d], -s.kexp);
        const double R = ceil((rmax * (1.0 + 1e-5) + 2.0 * moved * (1.0 + 1e-3) + 1e-4) / D);
        if (R > 1000.0) return false;
        g.R[d] = (int)R;
        g.D[d] = (float)D;
        g.gap[d] = (float)ldexp((double)(s.Lfix[d] - s.nc[d] * s.D[d]), -s.kexp);
        if (2 * g.R[d] + 1 > s.nc[d]) return false;
    }
    // segments of about 128 particles, as far as a row's cells stay distinct; one chunk more
    // than the mean needs, so that few segments leave the last one more than 32 particles
    const double per_cell = (double)s.n / s.ncell;
    const double cells = fmin(128.0 / fmax(per_cell, 1.0), (double)(s.nc[0] - 2 * g.R[0]));
    g.S = cells < 1.0 ? 1 : (int)cells;
    g.segs_x = (s.nc[0] + g.S - 1) / g.S;
    g.slots = (int)fmin(64.0, ceil(per_cell * g.S / 32.0)) + 1;
    g.ntiles = (int64_t)g.segs_x * s.nc[1] * s.nc[2] * g.slots;
    return true;
}

}  // namespace

namespace {

size_t gr_rows_bytes(int nbins) { return kRowWarps * sizeof(RowRing) + (size_t)3 * nbins * sizeof(unsigned); }
size_t gr_bytes(int nbins) { return kChunk * sizeof(JEnt) + (size_t)4 * nbins * sizeof(unsigned); }

}  // namespace

// Every kernel is opted into the shared memory of the most bins once and for all: set to each
// call's own need, the limit could be lowered by another thread's call between this one's set
// and its launch.
bool prepare_gr_kernels() {
    const cudaFuncAttribute most = cudaFuncAttributeMaxDynamicSharedMemorySize;
    return cudaFuncSetAttribute(k_gr_rows, most, (int)gr_rows_bytes(kGrMaxBins)) == cudaSuccess &&
           cudaFuncSetAttribute(k_gr_all, most, (int)gr_bytes(kGrMaxBins)) == cudaSuccess &&
           cudaFuncSetAttribute(k_gr_cells, most, (int)gr_bytes(kGrMaxBins)) == cudaSuccess;
}

namespace {

// Coarse cells of side >= rmax; false if the box holds fewer than three of them on an axis.
bool gr_coarse(const DevSim& s, double rmax, GrArgs& g) {
    bool cells = true;
    int64_t n = 1;
    for (int d = 0; d < 3; ++d) {
        double L = ldexp((double)s.Lfix[d], -s.kexp);
        int m = (int)floor(L / rmax);
        if (m < 3) cells = false;
        g.ncg[d] = m < 1 ? 1 : m;
        g.Dg[d] = s.Lfix[d] / g.ncg[d];
        n *= g.ncg[d];
    }
    g.ncells = (int)n;
    return cells;
}

}  // namespace

int64_t gr_scratch_ints(const DevSim& s, int nbins, double rmax) {
    GrRows rows;
    GrArgs g;
    if (gr_rows(s, nbins, rmax, rows) || !gr_coarse(s, rmax, g)) return 0;
    return 2 * s.n + 3 * ((int64_t)g.ncg[0] * g.ncg[1] * g.ncg[2] + 1);
}

// Returns 0, or -1 if scratch is too small (gr_scratch_ints).
int launch_gr(const DevSim& s, cudaStream_t st, int nbins, double rmax,
              unsigned long long* counts_dev, int32_t* scratch_i32, float4* /*scratch_f4*/,
              int64_t scratch_n) {
    GrArgs g;
    g.nbins = nbins;
    g.dr = rmax / (double)nbins;
    g.inv_dr = (float)(1.0 / g.dr);
    g.rmax2_hi = (float)(rmax * rmax * 1.001);
    const bool cells = gr_coarse(s, rmax, g);
    if (scratch_n < gr_scratch_ints(s, nbins, rmax)) return -1;
    const size_t smem = gr_bytes(nbins);
    cudaMemsetAsync(counts_dev, 0, sizeof(unsigned long long) * 4 * nbins, st);
    GrRows rows;
    if (gr_rows(s, nbins, rmax, rows)) {
        int dev = 0, nsm = 1;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
        const int64_t want = (rows.ntiles + kRowWarps - 1) / kRowWarps;
        const int grid = (int)(want < (int64_t)nsm * 3 ? want : (int64_t)nsm * 3);  // all resident
        k_gr_rows<<<grid, kRowWarps * 32, gr_rows_bytes(nbins), st>>>(s, g, rows, counts_dev);
        return 0;
    }
    if (!cells) {
        int nblk = (int)((s.n + kT - 1) / kT);
        k_gr_all<<<nblk, kT, smem, st>>>(s, g, counts_dev);
        return 0;
    }
    g.gkey = scratch_i32;
    g.gidx = scratch_i32 + s.n;
    g.gcount = scratch_i32 + 2 * s.n;
    g.gstart = g.gcount + (g.ncells + 1);
    g.gcursor = g.gstart + (g.ncells + 1);
    k_gr_zero<<<256, 256, 0, st>>>(g);
    k_gr_key<<<s.grid_part, 256, 0, st>>>(s, g);
    k_gr_scan<<<1, 1024, 0, st>>>(g);
    k_gr_scatter<<<s.grid_part, 256, 0, st>>>(s, g);
    int nblk = g.ncells < 65535 * 4 ? g.ncells : 65535 * 4;
    k_gr_cells<<<nblk, kT, smem, st>>>(s, g, counts_dev);
    return 0;
}

}  // namespace bbmd
