// The staging loop (stage_loop.cuh) on the host, over a model of the barriers and buffers that
// records every use the hardware leaves undefined.  Usage: host_stage_loop <buffers> <blocks>
// <bodies> <block whose wait gives up, or -1>; prints "ok" or the first misuse.  With the single
// argument "cells": the counts taken from a cell table of which a sort wrote only a part.
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <string>
#include <vector>

#include "../paper_1105_5613_gb300/csrc/stage_loop.cuh"

struct System {
    int64_t nblocks;
};

struct Buffer {
    bool valid = false;      // a live barrier
    int phase = 0;           // phases completed since its initialisation
    bool in_flight = false;  // copies issued and not waited for
    bool in_use = false;     // being computed from
    int64_t block = -1;      // what it holds
};

struct Model {
    std::vector<Buffer>& buf;
    int64_t fail_at;
    std::string& misuse;

    void bad(const std::string& what) {
        if (misuse.empty()) misuse = what;
    }
    void open() {
        for (Buffer& b : buf) {
            if (b.valid) bad("a live barrier is initialised");
            if (b.in_flight) bad("a barrier is initialised with copies in flight");
            b = Buffer();
            b.valid = true;
        }
    }
    int64_t position(const System&, int64_t blk) { return blk; }
    void issue(const System&, int64_t blk, int k) {
        Buffer& b = buf[(size_t)k];
        if (!b.valid) bad("copies on a dead barrier");
        if (b.in_flight || b.in_use) bad("a buffer is refilled too early");
        b.in_flight = true;
        b.block = blk;
    }
    bool wait(int k, uint32_t parity) {
        Buffer& b = buf[(size_t)k];
        if (!b.valid) bad("a wait on a dead barrier");
        if (!b.in_flight) bad("a wait for nothing");
        if ((uint32_t)(b.phase & 1) != parity) bad("a wait for the wrong phase");
        b.in_flight = false;
        ++b.phase;
        return b.block != fail_at;
    }
    bool finish(const System&, int k, uint32_t parity) {
        const bool ok = wait(k, parity);
        if (ok) buf[(size_t)k].in_use = true;
        return ok;
    }
    template <class Body>
    void compute(int64_t blk, int k, Body& body) {
        body(blk, k);
    }
    void drain(const System&, int k, uint32_t parity) { wait(k, parity); }
    void sync() {
        for (Buffer& b : buf) b.in_use = false;
    }
    void close() {
        for (Buffer& b : buf) {
            if (b.in_flight || b.in_use) bad("a barrier is invalidated in use");
            b.valid = false;
        }
    }
};

template <int BUFFERS>
static int run(int64_t blocks, int bodies, int64_t fail_at) {
    std::vector<Buffer> buf(BUFFERS);
    std::string misuse;
    Model m{buf, fail_at, misuse};
    for (int k = 0; k < bodies; ++k) {
        int64_t want = 1;  // this CTA's blocks: 1, 4, 7, ...
        auto body = [&](int64_t blk, int b) {
            if (blk != want || m.buf[(size_t)b].block != blk) m.bad("a body of the wrong block");
            if (!m.buf[(size_t)b].in_use) m.bad("a body before its copies");
            want += 3;
        };
        const bool ok = bbmd::staged_blocks<BUFFERS>(System{blocks}, m, 1, 3, body);
        const bool fails = fail_at >= 1 && fail_at < blocks && fail_at % 3 == 1;
        if (ok == fails) m.bad("a wait that gave up is not reported");
        if (ok && want < blocks) m.bad("a block is missing");
        for (const Buffer& b : m.buf)
            if (b.in_flight) m.bad("copies are left in flight");
        if (!ok) break;  // (the CTA stages no more)
    }
    std::puts(m.misuse.empty() ? "ok" : m.misuse.c_str());
    return 0;
}

// Tables of n particles in `cells` cells, every entry from one or the other of two sorts.
static int torn_cells() {
    const int cells = 144, smax = 65000;
    uint64_t x = 1;
    auto draw = [&](uint64_t m) { return (x = x * 6364136223846793005ull + 1442695040888963407ull, (x >> 33) % m); };
    for (int trial = 0; trial < 1000; ++trial) {
        const int n = trial % 2 ? 2000000000 : 20000;  // (a region overflows, or holds them all)
        std::vector<std::vector<int>> sorted(2, std::vector<int>(cells + 1));
        for (auto& s : sorted) {
            for (int& v : s) v = (int)draw((uint64_t)n + 1);
            std::sort(s.begin(), s.end());
            s[0] = 0;
            s[cells] = n;
        }
        std::vector<int> torn(cells + 1);
        for (int c = 0; c <= cells; ++c) torn[(size_t)c] = sorted[draw(2)][(size_t)c];
        int sum = 0;
        for (int c = 0; c < cells; ++c) {
            const int first = torn[(size_t)c], k = bbmd::cell_count(first, torn[(size_t)c + 1], smax);
            if (k < 0 || k > n - first || k > smax + 1 || __builtin_add_overflow(sum, k, &sum))
                return std::puts("a count out of range"), 0;
        }
        // the region's prefix, cut at smax; entries up to the sentinel's may stand in a list
        std::vector<int> off(cells + 1, 0);
        for (int c = 0, t = 0; c < cells; ++c) {
            t += bbmd::cell_count(torn[(size_t)c], torn[(size_t)c + 1], smax);
            off[(size_t)c + 1] = std::min(t, smax);
        }
        for (int t = 0; t <= smax; t += 97) {
            const int64_t i = bbmd::staged_particle(torn.data(), off.data(), cells, t);
            if (i < 0 || i > (int64_t)n + smax) return std::puts("a staged entry out of range"), 0;
        }
        const std::vector<int>& s0 = sorted[0];
        for (int c = 0; c < cells; ++c) {  // a whole table: the counts themselves
            const int k = s0[(size_t)c + 1] - s0[(size_t)c];
            if (bbmd::cell_count(s0[(size_t)c], s0[(size_t)c + 1], smax) != std::min(k, smax + 1))
                return std::puts("a count of a whole table changed"), 0;
        }
    }
    return std::puts("ok"), 0;
}

int main(int argc, char** argv) {
    if (argc == 2) return torn_cells();
    if (argc != 5) return 2;
    const int64_t blocks = std::atoll(argv[2]), fail_at = std::atoll(argv[4]);
    const int bodies = std::atoi(argv[3]);
    return std::atoi(argv[1]) == 2 ? run<2>(blocks, bodies, fail_at) : run<1>(blocks, bodies, fail_at);
}
