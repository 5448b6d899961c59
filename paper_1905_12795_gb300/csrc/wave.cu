// Acoustic forward modelling of every (model, shot) instance of a generation
// in one persistent launch, with the L2 misfit fused into the time loop
// (section "Testing approach": 2nd order in time, 8th (or 4th) order in space,
// damping layer, Ricker source, receivers along a line, l2 misfit).
//
// Scheme (centred in time, damped, constant density):
//   u^{n+1} = [2 u^n - (1 - t) u^{n-1} + a (lap_h u^n + s^n)] / (1 + t)
// with a = v^2 dt^2, t = (eta_x + eta_z) dt / 2, lap_h the order-2R centred
// Laplacian with zero values outside the padded grid, and s^n the bilinear
// point source r(n dt) b / (hx hz).  Trace sample n is the bilinear sample of
// u^{n+1}; phi = 1/2 sum (d - d_obs)^2.
//
// The instance runs on a group of co-resident CTAs (wave_group.cuh), with the
// update as written above.  One CTA of 512 threads per instance, as before,
// left an order-16 batch of 16 shots on 16 SMs: 1628 ms for 2014 steps of 16
// shots on the 921 x 301 grid + 60 cells, 43.0 ms on 16 groups of 19 CTAs (328 G
// updates/s).  Bound by the issue slots (41 % active with 8 warps per SM: the
// window's 17 rows leave registers for no more) and the barrier.
#include "wave_group.cuh"

namespace empso {

namespace {

template <int RF, bool HIST, bool WIDE = false>
__global__ void __launch_bounds__(WAVE_THREADS, GroupCtas<RF>::v)
wave_kernel(const GridDev *__restrict__ grids, const Inst *__restrict__ insts, int n_inst, int group, int *ws,
            float *slots, long long slot_floats, int *err, double *partial)
{
    group_cta<RF, false, HIST, WIDE>(grids, insts, n_inst, group, ws, slots, slot_floats, err, partial);
}

// (the history only at radius 8: the gradients of the other orders run their
// forward pass on the cluster kernels or per step)
WaveFn wave_fn(int R, bool hist, bool wide)
{
    if (wide) return hist ? (R == 8 ? wave_kernel<8, true, true> : nullptr) : wave_kernel<0, false, true>;
    if (hist) return R == 8 ? wave_kernel<8, true> : nullptr;
    if (R == 8) return wave_kernel<8, false>;
    if (R == 4) return wave_kernel<4, false>;
    if (R == 2) return wave_kernel<2, false>;
    return R == 1 ? wave_kernel<1, false> : wave_kernel<0, false>;
}

}  // namespace

WaveSplit wave_split(const GridDev *const *grids, int n_grids, int R, long long n_inst, long long by_l2, bool hist)
{
    return group_split(grids, n_grids, group_max_ctas(wave_fn(R, hist, group_wide(grids, n_grids))), n_inst, by_l2);
}

cudaError_t launch_wave(int R, const GridDev *grids_dev, const Inst *insts, int n_inst, const WaveSplit &s,
                        void *ws, float *slots, long long slot_floats, int *err, double *partial, cudaStream_t st,
                        bool hist)
{
    return launch_groups(wave_fn(R, hist, s.wide), grids_dev, insts, n_inst, s, ws, slots, slot_floats, err, partial, st);
}

// misfit[p] = sum_s weight_s partial[p][s] in fixed shot order; non-finite
// sums become +inf and are counted in nf[0] (running) and nf[1] (per call).
__global__ void finalize_kernel(const double *partial, const float *weights, int P, int S,
                                double *misfit, unsigned long long *nf)
{
    int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= P) return;
    double s = 0.0;
    for (int k = 0; k < S; ++k) s += (double)weights[k] * partial[(size_t)p * S + k];
    if (!isfinite(s)) {
        s = __longlong_as_double(0x7ff0000000000000LL);
        if (nf) {
            atomicAdd(nf, 1ull);
            atomicAdd(nf + 1, 1ull);
        }
    }
    misfit[p] = s;
}

cudaError_t launch_finalize(const double *partial, const float *weights, int P, int S,
                            double *misfit, unsigned long long *nf, cudaStream_t st)
{
    if (P <= 0) return cudaSuccess;
    finalize_kernel<<<(P + 127) / 128, 128, 0, st>>>(partial, weights, P, S, misfit, nf);
    return cudaGetLastError();
}

}  // namespace empso
