// The library's launch wrappers for a device that runs nothing (fake_runtime.cpp):
// they only write down that they were called.
#include <cstdint>
#include <cstdio>
#include "sph_internal.cuh"
#include "fake_device.h"

namespace {
void note(const char* what, int* status = nullptr) { fake_note(what, status); }
int device_of(const void* p) { return fake_device_of(p); }
}  // namespace

namespace sphg {

size_t radix_work_words(int64_t) { return 16; }
size_t radix_work_capacity(int64_t) { return 16; }
int64_t scan_tmp_words(int64_t) { return 16; }

int launch_reset_red(const Launch&, int, PatchRed*, const SortClear&) { return 1; }
int launch_reduce_bbox(const Launch&, const State&, const WorkItem* items, int nitems, PatchRed*)
{
    char s[64];
    snprintf(s, sizeof(s), "items=%lld", nitems ? (long long)items[nitems - 1].end : 0ll);
    note(s);
    return 1;
}
int launch_h_hist(const Launch&, const State&, const WorkItem*, int, PatchRed*) { return 1; }
int launch_grid_params(const Launch&, int, const PatchRed*, PatchDev*, double, int*, unsigned long long*) { return 1; }
int launch_keys(const Launch&, int64_t n, const State&, const uint16_t*, PatchDev*, const RadixSort&, int)
{
    char s[64];
    snprintf(s, sizeof(s), "keys=%lld", (long long)n);
    note(s);
    return 1;
}
int launch_radix_sort(const Launch&, int64_t, int, const RadixSort&, int* status) { note("sort", status); return 1; }
int launch_gather(const Launch&, int64_t, const uint32_t*, const uint32_t*, const State&, const State&, const uint32_t*,
                  uint32_t*, const PatchDev*, const Grid&, const Recs&, const Fp64&, int, int, const RowHint&, const int*,
                  const double*, double*) { return 1; }
int launch_refresh_records(const Launch&, int64_t, const State&, const uint16_t*, const PatchDev*, const uint32_t*,
                           const Recs&, const Fp64&, int, int) { return 1; }
int launch_cell_tables(const Launch&, int, PatchDev*, const Grid&, const float4*, int, float*, unsigned long long*) { return 1; }
int launch_nb_lists(const Launch&, const NbArgs& a, int exact)
{
    note(exact ? "lists" : "superset", a.status);
    a.pool_used[1] = 8;
    return 1;
}
int launch_nb_filter(const Launch&, const NbArgs& a, const uint32_t*, const uint32_t*) { note("filter", a.status); return 1; }
int launch_pair_bins(const Launch&, int64_t, const uint32_t*, const RadixSort&, uint32_t*, int* status) { note("bins", status); return 1; }
int launch_density(const Launch&, const PairArgs& a, int, int) { note("density", a.status); return 1; }
int launch_momentum(const Launch&, const PairArgs& a, int, int) { note("momentum", a.status); return 1; }
int launch_density_binned(const Launch&, PairArgs a, int, int) { note("density_binned", a.status); return 1; }
int launch_momentum_binned(const Launch&, PairArgs a, int, int) { note("momentum_binned", a.status); return 1; }
int launch_fused_density(const Launch&, const NbArgs&, const PairArgs&, int) { return 1; }
int launch_fused_momentum(const Launch&, const NbArgs&, const PairArgs&, int) { return 1; }
int launch_dt(const Launch&, const StepArgs&) { return 1; }
int launch_update(const Launch&, const StepArgs&) { return 1; }
int launch_step_finalize(const Launch&, const StepArgs&) { return 1; }
int launch_conserved_items(const Launch&, const StepArgs&) { return 1; }
int launch_conserved_finalize(const Launch&, const StepArgs&) { return 1; }
int launch_skin_radius(const Launch&, int64_t, const State&, const uint32_t*, const double*, double, double, double*) { return 1; }
int launch_skin_snapshot(const Launch&, int64_t, const State&, const SkinRef&) { return 1; }
// no particle has moved: the superset holds
int launch_skin_check(const Launch&, int64_t, const State&, const uint16_t*, const PatchDev*, const SkinRef&,
                      unsigned long long*, int* flag) { *flag = 1; return 3; }
int launch_unpermute_f64(const Launch&, int64_t, const double*, const uint32_t*, double*) { return 1; }
int launch_unpermute_f32(const Launch&, int64_t, const float*, int, const uint32_t*, double*) { return 1; }
int launch_unpermute_u32(const Launch&, int64_t, const uint32_t*, const uint32_t*, double*) { return 1; }
// (what a kernel would read and write directly is noted by where it lives)
int launch_load(const Launch&, int64_t, const double* const src[9], const State& s, uint32_t*, int*)
{
    bool own = true, here = true;
    double* const f[9] = {s.x, s.y, s.z, s.vx, s.vy, s.vz, s.m, s.h, s.u};
    for (int k = 0; k < 9; k++) {
        own = own && src[k] == f[k];
        here = here && device_of(src[k]) == 0;
    }
    note(own ? "load_own" : here ? "load_direct" : "load_elsewhere");
    return 1;
}
int launch_scan_u32_to_u64(const Launch&, int64_t, const uint32_t*, uint64_t* out, uint64_t*)
{
    if (device_of(out) != 0) note("scan_elsewhere");
    return 3;
}
int launch_canonical_rows(const Launch&, int64_t, const unsigned long long*, const uint32_t*, const uint64_t*, const uint32_t*,
                          uint32_t* out)
{
    note(device_of(out) == 0 ? "rows" : "rows_elsewhere");
    return 1;
}

}  // namespace sphg
