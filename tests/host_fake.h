// State shared by the fakes of the CUDA runtime (host_fake_runtime.cpp) and of the launches
// (host_fake_device.cu).
#pragma once
#include <cstdint>

struct FakeCounts {
    int32_t begin, grid_step, grid_relax, trigger_sort, graph_launch, sd_step, force, steps;
};

struct Fake {
    FakeCounts count;
    // what is refused: 1 launches of many steps; 2 the captured sort's launch; 4 the
    // instantiation of a graph with it; 8 replays of such a graph
    int refuse;
    int after;  // launches of many steps that still succeed
    bool capturing, captured_sort;
};
extern Fake fake;
