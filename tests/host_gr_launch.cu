// launch_gr on a box described by hand (k_observe.cu over the fakes of host_gr_runtime.cpp: no
// kernel runs).
#include <cmath>

#include "../paper_1105_5613_gb300/csrc/bbmd_internal.cuh"

extern "C" int gr_prepare() { return bbmd::prepare_gr_kernels() ? 0 : 1; }

// g(r) of a box of side L in nc cells a side, with scratch_n entries of scratch; 0, or launch_gr's
// refusal.
extern "C" int gr_call(double L, int nc, int nbins, double rmax, int64_t scratch_n) {
    bbmd::DevSim s = {};
    static int32_t scratch[1 << 20];
    static unsigned long long counts[4 * bbmd::kGrMaxBins];
    s.n = 1000;
    s.kexp = 50;
    for (int d = 0; d < 3; ++d) {
        s.Lfix[d] = std::llrint(std::ldexp(L, s.kexp));
        s.nc[d] = nc;
        s.D[d] = s.Lfix[d] / nc;
    }
    s.ncell = nc * nc * nc;
    s.disp_thr = s.disp_far = 0.3f;
    s.grid_part = 4;
    return bbmd::launch_gr(s, nullptr, nbins, rmax, counts, scratch, nullptr, scratch_n);
}
