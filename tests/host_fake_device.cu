// Fakes of the launches that bbmd_api.cu makes: nothing runs, every launch is counted.
#include "host_fake.h"

#include "../paper_1105_5613_gb300/csrc/bbmd_internal.cuh"

namespace {

cudaError_t cooperative_launch(int kind) {
    if (!(fake.refuse & kind)) return cudaSuccess;
    if (kind == 1 && fake.after > 0) {
        --fake.after;
        return cudaSuccess;
    }
    return cudaErrorCooperativeLaunchTooLarge;
}

}  // namespace

namespace bbmd {

void launch_begin(const DevSim&, cudaStream_t, int64_t, double, const bbmd_thermostat*) { ++fake.count.begin; }
void launch_check(const DevSim&, cudaStream_t) {}
void launch_check_finite(const DevSim&, cudaStream_t, const double*, int64_t) {}
void launch_check_many(const ManySims&, int, cudaStream_t) {}
void launch_clear_grid_sync(const DevSim&, cudaStream_t) {}
void launch_clear_rebuild(const DevSim&, cudaStream_t) {}
void launch_finalize(const DevSim&, cudaStream_t, bool) {}
void launch_finalize_many(const ManySims&, int, bool, cudaStream_t) {}
void launch_finish(const DevSim&, cudaStream_t) {}
void launch_forces_of_ids(const DevSim&, cudaStream_t, const int32_t*, const int64_t*, int64_t, double*, double*) {}
bool prepare_gr_kernels() { return true; }
int64_t gr_scratch_ints(const DevSim&, int, double) { return 0; }
int launch_gr(const DevSim&, cudaStream_t, int, double, unsigned long long*, int32_t*, float4*, int64_t) { return 0; }
void launch_init_fcc(const DevSim&, cudaStream_t, int, double, uint64_t) {}
void launch_init_mb(const DevSim&, cudaStream_t, double, uint64_t, double*, double*) {}
void launch_integrate(const DevSim&, cudaStream_t) {}
void launch_integrate_many(const ManySims&, int, bool, cudaStream_t) {}
void launch_list_counts(const DevSim&, cudaStream_t, const int32_t*, int64_t, int64_t*) {}
void launch_list_ids(const DevSim&, cudaStream_t, const int32_t*, int64_t, const int64_t*, int64_t*) {}
void launch_msd_fs(const DevSim&, cudaStream_t, const double*, double, double*) {}
void launch_observe_sums(const DevSim&, cudaStream_t, bool, double*) {}
void launch_pack_state(const DevSim&, cudaStream_t, const double*, const double*, const int32_t*, bool) {}
void launch_rebuild_chain(const DevSim&, cudaStream_t) {}
void launch_rebuild_chain_many(const ManySims&, const ManySims&, const ManySims&, int, int, int, cudaStream_t) {}
void launch_sd_step(const DevSim&, cudaStream_t, double, double) { ++fake.count.sd_step; }
void launch_set_K(const DevSim&, cudaStream_t) {}
void launch_set_ref(const DevSim&, cudaStream_t, double*) {}
void launch_slot_of(const DevSim&, cudaStream_t, int32_t*) {}
void launch_state_sums(const DevSim&, cudaStream_t) {}
void launch_unpack_cells(const DevSim&, cudaStream_t, int64_t*) {}
void launch_unpack_forces(const DevSim&, cudaStream_t, double*, double*) {}
void launch_unpack_state(const DevSim&, cudaStream_t, double*, double*, int32_t*) {}
int scan_grid(const DevSim&) { return 1; }
int trigger_sort_ctas(const DevSim&, int) { return 152; }
cudaError_t launch_trigger_sort(const DevSim&, int, cudaStream_t) {
    const cudaError_t e = cooperative_launch(2);
    if (e == cudaSuccess && fake.capturing) fake.captured_sort = true;
    ++fake.count.trigger_sort;
    return e;
}

#define FAKE_GRID(ns)                                                                                  \
    namespace ns {                                                                                     \
    bool prepare_force_kernels() { return true; }                                                      \
    int grid_step_ctas(const DevSim&, int nsm) { return 4 * nsm; }                                     \
    cudaError_t launch_grid_step(const DevSim&, int, int nsteps, bool, cudaStream_t) {                 \
        const cudaError_t e = cooperative_launch(1);                                                   \
        ++fake.count.grid_step;                                                                             \
        if (e == cudaSuccess) fake.count.steps += nsteps;                                                   \
        return e;                                                                                      \
    }                                                                                                  \
    cudaError_t launch_grid_relax(const DevSim&, int, int nsteps, double, double, cudaStream_t) {      \
        const cudaError_t e = cooperative_launch(1);                                                   \
        ++fake.count.grid_relax;                                                                            \
        if (e == cudaSuccess) fake.count.steps += nsteps;                                                   \
        return e;                                                                                      \
    }                                                                                                  \
    }
#define FAKE_SHAPE(ns)                                                                                 \
    FAKE_GRID(ns)                                                                                      \
    namespace ns {                                                                                     \
    int force_blocks_per_sm(const DevSim&) { return 2; }                                               \
    int list_blocks_per_sm(const DevSim&) { return 2; }                                                \
    int energies_blocks_per_sm(const DevSim&) { return 2; }                                            \
    void launch_force(const DevSim&, cudaStream_t, bool, bool) { ++fake.count.force; }                      \
    void launch_energies(const DevSim&, cudaStream_t, bool) {}                                         \
    void launch_list_build(const DevSim&, cudaStream_t) {}                                             \
    void launch_list_build_many(const ManySims&, int, int, cudaStream_t) {}                            \
    void launch_force_many(const ManySims&, int, bool, bool, bool, bool, int, cudaStream_t) {}         \
    }
FAKE_SHAPE(z1)
FAKE_SHAPE(z2)
FAKE_SHAPE(z4)
FAKE_SHAPE(z8)
FAKE_GRID(z1w)

namespace BBMD_PERSIST_NS {
bool prepare_persistent() { return true; }
int persistent_blocks_per_sm(int) { return 2; }
cudaError_t launch_persistent_step(const PersistentStep&, int, int, bool, bool, cudaStream_t) { return cudaSuccess; }
}  // namespace BBMD_PERSIST_NS

}  // namespace bbmd
