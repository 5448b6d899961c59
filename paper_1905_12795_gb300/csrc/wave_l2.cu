// L2-resident variant of the persistent modelling launch, for grids whose two
// time levels do not fit the shared memory of a cluster (e.g. the 921 x 301 grid
// at 10 m with a 60-cell damping layer).  Same scheme and fused
// source/receiver/misfit work as the other variants (section "Testing
// approach": 2nd order in time, 4th/8th order in space, damping layer, Ricker
// source, l2 misfit), on groups of co-resident CTAs (wave_group.cuh) with the
// damped update written as g (u^n - u^{n-1}) + u^{n-1} + (a g / 2) lap.
//
// Measured on the grid above, order 8, 16 shots, 2826 steps: 81.7 ms on
// thread-block clusters of 10 CTAs of 512 threads with a cluster barrier per
// step (two rounds of 13 clusters, 243 G updates/s), 44.7 ms on groups (443 G
// updates/s); 64 shots, 471 steps: 34.8 and 29.8 ms.
#include "wave_group.cuh"

namespace empso {

namespace {

template <int RF, bool HIST, bool WIDE = false>
__global__ void __launch_bounds__(WAVE_THREADS, GroupCtas<RF>::v)
wave_l2_kernel(const GridDev *__restrict__ grids, const Inst *__restrict__ insts, int n_inst, int group, int *ws,
               float *slots, long long slot_floats, int *err, double *partial)
{
    group_cta<RF, true, HIST, WIDE>(grids, insts, n_inst, group, ws, slots, slot_floats, err, partial);
}

WaveFn l2_fn(int R, bool hist, bool wide)
{
    if (wide) return hist ? wave_l2_kernel<0, true, true> : wave_l2_kernel<0, false, true>;
    if (hist) {
        if (R == 4) return wave_l2_kernel<4, true>;
        if (R == 2) return wave_l2_kernel<2, true>;
        return R == 1 ? wave_l2_kernel<1, true> : nullptr;
    }
    if (R == 4) return wave_l2_kernel<4, false>;
    if (R == 2) return wave_l2_kernel<2, false>;
    return R == 1 ? wave_l2_kernel<1, false> : nullptr;
}

}  // namespace

// What the variant takes: at least 8 padded rows for each of the C SMs of an instance
// (C = 1 when the library chooses the split), and at most as many receivers a shot as
// tables of 28 bytes each fill `limit` bytes (about 8300).  A group needs neither;
// they are what EMPSO_KERNEL_CLUSTER_L2 refuses and the streaming kernels take.
bool l2_fits(const GridDev &g, int C, int nrec, size_t limit)
{
    const int rows_c = (g.NZ + C - 1) / C;
    const size_t table = sizeof(float) * (4 + (2 * (size_t)nrec + 3) / 4 * 4) + 20 * (size_t)nrec;
    return C >= 1 && C <= 16 && rows_c >= 8 && (C - 1) * rows_c < g.NZ && table <= limit;
}

// C > 0: the CTAs of C SMs for each instance
WaveSplit l2_split(const GridDev *const *grids, int n_grids, int R, long long n_inst, long long by_l2, int C, int sms,
                   bool hist)
{
    const int ctas = group_max_ctas(l2_fn(R, hist, group_wide(grids, n_grids)));
    return group_split(grids, n_grids, ctas, n_inst, by_l2, C > 0 ? C * std::max(1, ctas / sms) : 0);
}

cudaError_t launch_wave_l2(int R, const GridDev *grids_dev, const Inst *insts, int n_inst, const WaveSplit &s,
                           void *ws, float *slots, long long slot_floats, int *err, double *partial, cudaStream_t st,
                           bool hist)
{
    return launch_groups(l2_fn(R, hist, s.wide), grids_dev, insts, n_inst, s, ws, slots, slot_floats, err, partial, st);
}

}  // namespace empso
